// zmc_runtime.h — host-side helpers shared by the runtime translation units.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

#include "zmc_internal.h"

namespace zmc {

struct TilePlan {
  int lanes = 32;   // threads summing one unit-split (power of two)
  int splits = 1;   // sample ranges per (point, trial) unit
  int block = 256;  // threads per block
  // How the launch is shaped; neither changes a result.
  int trials = 1;          // trials of a point that the same lanes sample (1, 2, 4)
  int launch_block = 256;  // threads per block of the launch, at most `block`
  bool tuned = false;      // lanes, splits and block are the autotuner's
};

// Byte offsets of each region inside one scan's device scratch.  The slice
// is cut into `chunks` chunks of `chunk_points` grid points; the partial sums
// hold one chunk, the host-memory output regions `nbuf` chunks each.
struct ScanLayout {
  size_t partial, partial_bytes;
  size_t vals, mean, err, errw, s1, s2;  // SIZE_MAX when not used
  size_t total;
  int64_t chunk_points = 0, chunks = 0;
  int nbuf = 1;
};

int fail(int status, const char* fmt, ...);
int cuda_fail(cudaError_t e, const char* what);
void clear_error();
const char* last_error();

int validate(const zmc_scan_desc* d, int64_t* P_out, int64_t* count_out);
TilePlan plan_tiles(int N, int64_t S, int T, int64_t count, int sm_count, int threads_per_sm,
                    int lanes_req, int splits_req, int block_req, int precision);
// The tile plan of a scan on a device with `sm` SMs of `tps` threads each:
// an autotuner entry for the scan's class when the caller leaves the tiles
// open and one is recorded (memory reads only), else plan_tiles.
TilePlan plan_with(const zmc_scan_desc* d, int64_t count, int sm, int tps);
// The launch shape (trials, launch_block) of a launch over `count` points with the
// sums of `tp`.
void plan_launch(const zmc_scan_desc* d, int64_t count, int sm, TilePlan* tp);
// plan_with for the current device (its properties from the device state),
// after loading the autotuner's cache file once.
int plan_for(const zmc_scan_desc* d, int64_t count, TilePlan* tp);
// User integrands compiled at run time (zmc_user.cu).
bool is_user_integrand(int id);
int user_validate(const zmc_scan_desc* d);
int user_info(int id, zmc_integrand_info* info);
int user_launch(const zmc_scan_desc* d, const ScanArgs& a, int block, int64_t grid, size_t smem,
                cudaStream_t stream);
// Tuned-table access (zmc_tune.cu).  tune_find reads memory only.
void tune_ensure_loaded();
bool tune_find(int prec, int gid, int N, int64_t S, int* lanes, int* block, int* gpl);
ScanLayout layout_for(const zmc_scan_desc* d, int64_t count, const TilePlan& tp);
int64_t chunk_points_for(const zmc_scan_desc* d, int64_t count, const TilePlan& tp);
// The most trials of a point that one lane of this scan's kernel samples.
int max_lane_trials(const zmc_scan_desc* d);
// Philox calls of a scan of `count` points.
int64_t scan_calls(const zmc_scan_desc* d, int64_t count);
// The plan of a batched or served scan with at most `trials` trials per lane and
// about `lane_calls` Philox calls per lane, but no lane shorter than
// `least_groups` sample groups; and the number of tiles of `count` points.
TilePlan plan_batch_scan(const zmc_scan_desc* d, int trials, int64_t lane_calls,
                         int64_t least_groups);
int64_t batch_tiles(const zmc_scan_desc* d, int64_t count, const TilePlan& tp);
// The plans of the n scans of a batch on a device of `sm` SMs.
void plan_batch(const zmc_scan_desc* d, const int64_t* counts, int n, int sm, TilePlan* plans);
// A persistent launch gets this many lanes per resident thread, if they keep
// kBatchLeastGroups sample groups each.  Measured on GB300 on small batches: 27
// scans (4.2e7 evaluations) 640 us with lanes of up to 1024 groups whatever the
// batch's size, 150 / 143 / 144 us with 1 / 2 / 4; 37 scans (1.3e8) 1314 us and
// 502 / 460 / 456 us.  Lanes of at least 32 groups against 64: 87 and 125 us for
// 29 scans of 1.3e7 evaluations; 16 gives no more.
constexpr int64_t kBatchWaves = 4;
constexpr int64_t kBatchLeastGroups = 32;
// Tiles per SM from which on lanes take b trials in the persistent kernel: a
// launch with fewer is short of independent work, and its largest bodies spill
// registers with four.  Measured: 4.2e7 evaluations with four trials per lane
// 1019 us, one 640 us; 5.4e9 in 6500 tiles 12.31 and 12.33 ms with 2 and 4 (12.98
// with one, before the round keys took uniform registers); 7.4e10 in 10^5 tiles
// 224.2 and 223.8 ms.
constexpr int64_t batch_rounds(int b) { return b >= 4 ? 200 : b >= 2 ? 12 : 0; }
// Lane groups of a launch over `count` points (and how many of them take four
// and two trials, may be null).
int64_t lane_groups_of(const zmc_scan_desc* d, int64_t count, const TilePlan& tp, int64_t* lu4,
                       int64_t* lu2);
double box_volume(const zmc_scan_desc* d);
void fill_scan_args(const zmc_scan_desc* d, int64_t count, const TilePlan& tp,
                    const double* vals_dev, double* partial_dev, ScanArgs* a);
int launch_scan_args(const zmc_scan_desc* d, const ScanArgs& a, const TilePlan& tp,
                     cudaStream_t stream);
int scan_ex(const zmc_scan_desc* d, zmc_scan_out* o);
// The current device's check words in ZMC_DEBUG builds (once its state is set
// up by an allocating entry point), else null.
unsigned long long* debug_words();
// ZMC_DEBUG builds: wait for the device, read and clear its check words;
// returns the failed checks since the last read (first failure in *code and
// *index), or -1 in release builds.
int64_t debug_take(unsigned* code, long long* index);

}  // namespace zmc
