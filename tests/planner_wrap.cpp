// C wrappers around the planner of csrc/zmc_runtime.h, linked with libzmc.so by
// test_planner_cpu.py.
#include "zmc_runtime.h"

extern "C" int launch_shape(const zmc_scan_desc* d, int64_t count, int sm, int lanes, int splits,
                            int block, int* out) {
  zmc::TilePlan tp;
  tp.lanes = lanes;
  tp.splits = splits;
  tp.block = block;
  zmc::plan_launch(d, count, sm, &tp);
  out[0] = tp.trials;
  out[1] = tp.launch_block;
  return 0;
}

extern "C" void batch_trials(const zmc_scan_desc* d, const int64_t* counts, int n, int sm,
                             int* out) {
  zmc::TilePlan plans[64];
  zmc::plan_batch(d, counts, n, sm, plans);
  for (int i = 0; i < n; ++i) {
    out[3 * i] = plans[i].trials;
    out[3 * i + 1] = plans[i].lanes;
    out[3 * i + 2] = plans[i].splits;
  }
}
