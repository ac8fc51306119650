// zmc_batch_inst.cu — the persistent batched sampling kernel (K3) for one
// precision (compiled once per ZMC_INST_PREC).
//
// Many scans of different integrands, dimensions, grid sizes and sample counts
// run in one launch.  The host cuts every scan into tiles — the lane groups one
// block sums at once, all of one scan — and orders them longest first.  Each
// resident block takes the next tile from a device counter (one atomicAdd by
// thread 0, no waiting on other blocks), stages that scan's lists or constant
// tables into shared memory when the scan changes, takes its Philox round
// keys into uniform registers, and runs the same per-lane sampling and reduction code
// as the single-scan kernel, writing each unit-split's FP64 partial sums into
// that scan's slice of the batch's partial buffer.
// The batched bodies keep as many Philox calls in flight per lane as the
// single-scan kernel; the order of the compensated additions does not depend
// on the blocking in any case, so results stay bit-identical to solo runs.
#include "zmc_scan_kernel.cuh"
#if ZMC_INST_PREC == 0
#include "zmc_integrands_fixed.cuh"
#endif

#ifndef ZMC_INST_PREC
#error "ZMC_INST_PREC must be defined"
#endif

namespace zmc {

#if ZMC_INST_PREC == 0
#define ZMC_BF(name) name##64
#else
#define ZMC_BF(name) name##32
#endif

// Resident blocks per SM the register allocation is held to: 2 x 256 threads
// (128 registers), so that the FP32 bodies do not spill; the largest bodies
// set the residency of the whole launch (measured: faster than 85 or 64).
#ifndef ZMC_BATCH_MIN_BLOCKS
#define ZMC_BATCH_MIN_BLOCKS 2
#endif

// One tile.  Not inlined: each (integrand, N) body gets its own register
// allocation instead of the union of all 48 bodies (one call per tile).
template <int N, class F, int PREC>
__device__ __noinline__ void batch_tile(const ScanArgs& a, const BatchTile& t, bool restage,
                                           double* smem, float* dimc, const int64_t* fxc,
                                           const int64_t* fxe, double* red) {
  // Lists / tables of this scan (kept when the previous tile was the same scan).
  const void* table = nullptr;
  if (restage) {
    table = stage_lists<N, F>(a, smem, dimc);
  } else {
    table = a.stage_smem ? static_cast<const void*>(smem) : nullptr;
  }
  // The round keys are the same for the whole warp: a reduction's result lives in
  // uniform registers, which leaves 20 of the 128 to the body (spilled stores of the
  // largest bodies 340-550 bytes without it, at most 200 with it; 64 uneven scans
  // 12.50 -> 12.31 ms).
  uint32_t rk0[10], rk1[10];
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    rk0[r] = __reduce_or_sync(0xffffffffu, a.rk0[r]);
    rk1[r] = __reduce_or_sync(0xffffffffu, a.rk1[r]);
  }
  FieldConst fc;
  fc.mask = __reduce_or_sync(0xffffffffu, a.field.mask);
  fc.one = __reduce_or_sync(0xffffffffu, a.field.one);
  fc.shl4 = __reduce_or_sync(0xffffffffu, a.field.shl4);
  block_work<N, F, PREC>(a, fc, rk0, rk1, table, dimc,
                         FxOf<F, PREC>::kTable == kFxExpTable ? fxe : fxc, t.first_w, t.units,
                         red);
}

#define ZMC_CASE_N(gid, F, n)                                                        \
  case (gid)*8 + (n)-1:                                                              \
    batch_tile<n, F<n>, ZMC_INST_PREC>(a, t, restage, smem, dimc, fxc, fxe, red);              \
    break;
#define ZMC_CASES(gid, F)                                                            \
  ZMC_CASE_N(gid, F, 1) ZMC_CASE_N(gid, F, 2) ZMC_CASE_N(gid, F, 3)                  \
  ZMC_CASE_N(gid, F, 4) ZMC_CASE_N(gid, F, 5) ZMC_CASE_N(gid, F, 6)                  \
  ZMC_CASE_N(gid, F, 7) ZMC_CASE_N(gid, F, 8)

template <int PREC>
__global__ void __launch_bounds__(256, ZMC_BATCH_MIN_BLOCKS)
batch_kernel(const __grid_constant__ BatchArgs b) {
  extern __shared__ double smem[];
  __shared__ double red[kReduceDoubles];
  __shared__ float dimc[3 * ZMC_MAX_N];
  __shared__ long long s_tile;
  const int64_t *fxc = nullptr, *fxe = nullptr;
#if ZMC_INST_PREC == 0
  __shared__ int64_t fx_tables[kFxCosEntries + kFxExpEntries];
  fx_fill_tables(fx_tables);  // the first barrier of the loop is behind it
  fxc = fx_tables;
  fxe = fx_tables + kFxCosEntries;
#endif
  int staged = -1;  // scan whose lists/tables are in shared memory
  for (;;) {
    if (threadIdx.x == 0) s_tile = static_cast<long long>(atomicAdd(b.counter, 1ull));
    __syncthreads();
    const long long tile = s_tile;
    if (tile >= b.ntiles) break;
    const BatchTile t = b.tiles[tile];
    if (ZMC_CHECK(b.dbg, t.scan >= 0 && t.scan < b.nscans && t.units >= 0, kDbgTile, tile)) {
      const ScanArgs& a = b.scans[t.scan];
      const bool restage = t.scan != staged;
      staged = t.scan;
      switch (a.gid * 8 + a.N - 1) {
        ZMC_CASES(ZMC_G_CONST, ZMC_BF(Const))
        ZMC_CASES(ZMC_G_COSPROD, ZMC_BF(CosProd))
        ZMC_CASES(ZMC_G_GAUSS03, ZMC_BF(Gauss))
        ZMC_CASES(ZMC_G_POLY, ZMC_BF(Poly))
        ZMC_CASES(ZMC_G_OSC01, ZMC_BF(Osc))
        ZMC_CASES(ZMC_G_SINSUM, ZMC_BF(SinSum))
        default:
          break;
      }
    }
    __syncthreads();  // the tile is done before shared memory or s_tile is reused
  }
}

#define ZMC_BATCH_FN2(p) batch_launch_p##p
#define ZMC_BATCH_FN(p) ZMC_BATCH_FN2(p)
#define ZMC_BATCH_OCC2(p) batch_occupancy_p##p
#define ZMC_BATCH_OCC(p) ZMC_BATCH_OCC2(p)

// The FP64 kernel holds both fixed-point tables beside the scans' lists.
#if ZMC_INST_PREC == 0
constexpr size_t kBatchTables = (kFxCosEntries + kFxExpEntries) * sizeof(int64_t);
#else
constexpr size_t kBatchTables = 0;
#endif

int ZMC_BATCH_FN(ZMC_INST_PREC)(const BatchArgs& b, int grid, int block, size_t smem,
                                void* stream) {
  const cudaError_t e = allow_smem(batch_kernel<ZMC_INST_PREC>, kBatchTables, smem);
  if (e != cudaSuccess) return static_cast<int>(e);
  batch_kernel<ZMC_INST_PREC><<<grid, block, smem, static_cast<cudaStream_t>(stream)>>>(b);
  return static_cast<int>(cudaGetLastError());
}

int ZMC_BATCH_OCC(ZMC_INST_PREC)(int block, size_t smem, int* out) {
  const cudaError_t e = allow_smem(batch_kernel<ZMC_INST_PREC>, kBatchTables, smem);
  if (e != cudaSuccess) return static_cast<int>(e);
  return static_cast<int>(
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, batch_kernel<ZMC_INST_PREC>, block,
                                                    smem));
}

}  // namespace zmc
