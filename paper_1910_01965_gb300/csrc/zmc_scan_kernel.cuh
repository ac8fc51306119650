// zmc_scan_kernel.cuh — the sampling kernel (K1) and its building blocks.
//
// Direct Monte Carlo over a parameter grid (Eq. 1, Sec. 2): every unit
// (grid point p, trial t) sums g over its S samples.  The paper gives each
// grid point to one GPU thread that loops over all samples (Sec. 2, Fig. 1);
// here a unit's samples are cut into `splits` ranges and each range is summed
// by `lanes` threads, so that a grid of any shape fills all SMs.  Up to four
// trials of a point are summed by the same threads, which share a part of their
// Philox calls.  Lane sums
// are reduced with warp shuffles and, for ranges wider than a warp, through
// shared memory, in a fixed order; each range writes one FP64 (sum g,
// sum g^2) pair.  The finalize kernel (K2) adds the ranges in order and forms
// the statistics.
//
// Sample groups: G = group_samples(N) consecutive samples use exactly
// C = group_calls(N) Philox calls (G*N = 5C fields), so a lane always works
// on whole groups and never shares a call with another lane.
#pragma once

#include <cstdint>

#include "zmc_integrands.cuh"
#include "zmc_internal.h"
#include "zmc_philox.cuh"

namespace zmc {

enum { kPrecFP64 = ZMC_FP64, kPrecFP32 = ZMC_FP32, kPrecFP32K = ZMC_FP32_KAHAN };

// Compile-time tuning knobs (defaults are the shipped configuration).
#ifndef ZMC_LB_THREADS
#define ZMC_LB_THREADS 512   // __launch_bounds__ maximum block size
#endif
#ifndef ZMC_LB_MIN_BLOCKS
#define ZMC_LB_MIN_BLOCKS 1  // __launch_bounds__ minimum resident blocks
#endif
// ZMC_CALLS_IN_FLIGHT, when defined, overrides every functor's kCallsInFlight
// (independent Philox calls per lane per loop block in the FP32 paths).

// How a functor evaluates: in floating point, or in fixed point with one of the
// tables in shared memory or with none.
enum { kFxNone = 0, kFxCosTable = 1, kFxExpTable = 2, kFxNoTable = 3 };

// The fixed-point functors specialise this: their table, their lane sums and
// the FP64 functor that takes the parameters outside their range.
template <class F, int PREC>
struct FxOf;

template <int PREC>
struct LaneAcc;

template <>
struct LaneAcc<kPrecFP64> {
  double s1 = 0.0, s2 = 0.0;
  __device__ __forceinline__ void add(double g) {
    s1 += g;
    s2 = fma(g, g, s2);
  }
  __device__ __forceinline__ void add2(double a, double b) {
    add(a);
    add(b);
  }
  template <int K>
  __device__ __forceinline__ void add_group(const double* v) {
#pragma unroll
    for (int i = 0; i < K; ++i) add(v[i]);
  }
  __device__ __forceinline__ double sum1() const { return s1; }
  __device__ __forceinline__ double sum2() const { return s2; }
};

template <>
struct LaneAcc<kPrecFP32> {
  float s1 = 0.0f, s2 = 0.0f;
  __device__ __forceinline__ void add(float g) {
    s1 += g;
    s2 = fmaf(g, g, s2);
  }
  __device__ __forceinline__ void add2(float a, float b) {
    add(a);
    add(b);
  }
  template <int K>
  __device__ __forceinline__ void add_group(const float* v) {
#pragma unroll
    for (int i = 0; i < K; ++i) add(v[i]);
  }
  __device__ __forceinline__ double sum1() const { return s1; }
  __device__ __forceinline__ double sum2() const { return s2; }
};

// Kahan-compensated FP32 sums: c carries the negated low part, so the lane's
// sum is s - c, taken in FP64.
template <>
struct LaneAcc<kPrecFP32K> {
  float s1 = 0.0f, c1 = 0.0f, s2 = 0.0f, c2 = 0.0f;
  __device__ __forceinline__ void add(float g) {
    const float y1 = g - c1;
    const float t1 = s1 + y1;
    c1 = (t1 - s1) - y1;
    s1 = t1;
    const float y2 = fmaf(g, g, -c2);
    const float t2 = s2 + y2;
    c2 = (t2 - s2) - y2;
    s2 = t2;
  }
  // Two samples: their plain FP32 pair sums enter the compensated sums (the
  // pair's own rounding is at the scale of one sample, not of the running
  // sum, which is what the compensation protects).
  __device__ __forceinline__ void add2(float a, float b) {
    const float u = a + b;
    const float v = fmaf(a, a, b * b);
    const float y1 = u - c1;
    const float t1 = s1 + y1;
    c1 = (t1 - s1) - y1;
    s1 = t1;
    const float y2 = v - c2;
    const float t2 = s2 + y2;
    c2 = (t2 - s2) - y2;
    s2 = t2;
  }
  // K samples at once (a sample group): their plain FP32 sums, formed in a
  // fixed order, enter the compensated sums in one step.
  template <int K>
  __device__ __forceinline__ void add_group(const float* v) {
    float u = v[0], w = v[0] * v[0];
#pragma unroll
    for (int i = 1; i < K; ++i) {
      u += v[i];
      w = fmaf(v[i], v[i], w);
    }
    const float y1 = u - c1;
    const float t1 = s1 + y1;
    c1 = (t1 - s1) - y1;
    s1 = t1;
    const float y2 = w - c2;
    const float t2 = s2 + y2;
    c2 = (t2 - s2) - y2;
    s2 = t2;
  }
  __device__ __forceinline__ double sum1() const {
    return static_cast<double>(s1) - static_cast<double>(c1);
  }
  __device__ __forceinline__ double sum2() const {
    return static_cast<double>(s2) - static_cast<double>(c2);
  }
};

template <class F, int PREC>
struct FxOf {
  static constexpr int kTable = kFxNone;
  static constexpr size_t kStaticBytes = 0;
  using Acc = LaneAcc<PREC>;
};

// List that staged value `idx` belongs to.
__device__ __forceinline__ int list_of(const ScanArgs& a, int idx) {
  int k = 0;
  for (int i = 1; i < a.M; ++i)
    if (idx >= a.off[i]) k = i;
  return k;
}

// One mixed-radix digit: d = p mod L, p = p div L, in 32 bits when the whole
// slice's indices fit (the common case), else in 64.
__device__ __forceinline__ int64_t next_digit(const ScanArgs& a, int64_t& p, int64_t L) {
  if (a.idx32) {
    const uint32_t p32 = static_cast<uint32_t>(p), L32 = static_cast<uint32_t>(L);
    const uint32_t q = p32 / L32;
    p = q;
    return p32 - q * L32;
  }
  const int64_t q = p / L;
  const int64_t d = p - q * L;
  p = q;
  return d;
}

// Decode the flat grid index p (C order, last list fastest; Sec. 2: the grid
// is the Cartesian product of the lists) and hand the parameters to f.
// `table` is the block's staged per-value table (null when not staged) and
// `dimc` its per-dimension constants.
template <int N, class F>
__device__ __forceinline__ void load_params(const ScanArgs& a, const void* table,
                                            const float* dimc, int64_t p, F& f) {
  if constexpr (F::kTable) {
#pragma unroll
    for (int i = N - 1; i >= 0; --i) {
      const int64_t d = next_digit(a, p, a.len[i]);
      int idx = a.off[i] + static_cast<int>(d);
      if (!ZMC_CHECK(a.dbg, d >= 0 && d < a.len[i] && idx < a.nvals, kDbgListOffset, idx))
        idx = 0;
      const float2 v = table ? static_cast<const float2*>(table)[idx]
                             : F::value(i, a.vals[idx], a.lo[i], a.hi[i]);
      f.load(i, v, &dimc[3 * i]);
    }
  } else if constexpr (F::kFixedM > 0) {
    // one compiled M: the parameters land in registers
    const double* vals = table ? static_cast<const double*>(table) : a.vals;
#pragma unroll
    for (int i = F::kFixedM - 1; i >= 0; --i) {
      const int64_t d = next_digit(a, p, a.len[i]);
      int64_t idx = a.off[i] + d;
      if (!ZMC_CHECK(a.dbg, d >= 0 && d < a.len[i] && idx < a.nvals, kDbgListOffset, idx))
        idx = 0;
      f.set_param(i, vals[idx]);
    }
    f.finish(a.lo, a.hi);
  } else if constexpr (F::kPerDim) {
    // M == N: parameter i pairs with dimension i.
    const double* vals = table ? static_cast<const double*>(table) : a.vals;
#pragma unroll
    for (int i = N - 1; i >= 0; --i) {
      const int64_t d = next_digit(a, p, a.len[i]);
      int64_t idx = a.off[i] + d;
      if (!ZMC_CHECK(a.dbg, d >= 0 && d < a.len[i] && idx < a.nvals, kDbgListOffset, idx))
        idx = 0;
      f.set(i, vals[idx], a.lo[i], a.hi[i]);
    }
  } else {
    const double* vals = table ? static_cast<const double*>(table) : a.vals;
    for (int i = a.M - 1; i >= 0; --i) {
      const int64_t d = next_digit(a, p, a.len[i]);
      int64_t idx = a.off[i] + d;
      if (!ZMC_CHECK(a.dbg, d >= 0 && d < a.len[i] && idx < a.nvals, kDbgListOffset, idx))
        idx = 0;
      f.add(vals[idx]);
    }
    f.finish(a.lo, a.hi);
  }
}

// Stage the lists into shared memory: per-value FP32 constants for kTable
// functors, the FP64 values otherwise.  Every thread of the block calls it.
template <int N, class F>
__device__ __forceinline__ const void* stage_lists(const ScanArgs& a, double* smem,
                                                   float* dimc) {
  if constexpr (F::kTable) {
    if (threadIdx.x < N)
      F::dim(threadIdx.x, a.lo[threadIdx.x], a.hi[threadIdx.x], &dimc[3 * threadIdx.x]);
    if (a.stage_smem) {
      float2* tab = reinterpret_cast<float2*>(smem);
      // With one dimension every grid point is a value of the one list, so the list is as
      // long as the grid: there the values go four at a time where each is a chain of FP64
      // operations (cos-product, T = 1, S = 65536, 4000 values: 272 -> 228 us, 1000 values
      // 61.6 -> 57.5 us).  With more dimensions, or where a value is only converted, one at
      // a time is the faster by up to 3 %.
      if constexpr (N == 1 && F::kValueChain) {
        const double lo = a.lo[0], hi = a.hi[0];
        for (int i0 = threadIdx.x; i0 < a.nvals; i0 += 4 * blockDim.x) {
          double x[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * blockDim.x;
            x[u] = i < a.nvals ? a.vals[i] : 0.0;
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * blockDim.x;
            if (i < a.nvals &&
                ZMC_CHECK(a.dbg, (i + 1) * sizeof(float2) <= dynamic_smem_bytes(),
                          kDbgStagedTable, i))
              tab[i] = F::value(0, x[u], lo, hi);
          }
        }
      } else {
        for (int i = threadIdx.x; i < a.nvals; i += blockDim.x) {
          if (!ZMC_CHECK(a.dbg, (i + 1) * sizeof(float2) <= dynamic_smem_bytes(),
                         kDbgStagedTable, i))
            break;
          const int k = list_of(a, i);
          tab[i] = F::value(k, a.vals[i], a.lo[k], a.hi[k]);
        }
      }
    }
    __syncthreads();
    return a.stage_smem ? smem : nullptr;
  } else {
    if (a.stage_smem) {
      for (int i = threadIdx.x; i < a.nvals; i += blockDim.x) {
        if (!ZMC_CHECK(a.dbg, (i + 1) * sizeof(double) <= dynamic_smem_bytes(),
                       kDbgStagedTable, i))
          break;
        smem[i] = a.vals[i];
      }
      __syncthreads();
      return smem;
    }
    return nullptr;
  }
}

// Sample g of a group whose C calls' words are r[0 .. 4C): its N unit values
// come from the group's fields g*N .. g*N + N - 1 (field e is field e mod 5
// of the group's call e / 5).
template <int N, class F>
__device__ __forceinline__ auto eval_sample(const F& f, const FieldConst& fc,
                                            const uint32_t* r, int g) {
  typename F::unit_t u[N];
#pragma unroll
  for (int k = 0; k < N; ++k) {
    const int e = g * N + k;
    u[k] = field_value<typename F::unit_t>(fc, r + 4 * (e / kFieldsPerCall),
                                           e % kFieldsPerCall);
  }
  return f.eval(u);
}

// A lane samples this many trials of one grid point together at most (they
// share a part of every Philox call); the FP64 kernels, bound elsewhere, the
// constant integrand, which draws nothing, and the user integrands (kFixedM) take
// one.  A user's function has any number of operations and registers: four copies of
// one with a sine, two exponentials and a root per dimension run at 0.50 (N = 6, 8) to
// 0.89 (N = 1) of the rate of one and take 2.5 to 8 times as long to compile, while a
// short one (cosine products) gains 1.07.
template <int N, class F, int PREC>
constexpr int max_trials() {
  return PREC == kPrecFP64 || !F::kUsesSamples || F::kFixedM > 0 ? 1 : max_lane_trials(N);
}

// Sums over the sample groups [q, q_end) with stride `step` (one lane) of B
// trials, trial u of them with the Philox constants b1[u], b2[u].
//
// What bounds the FP32 kernels: the ALU together with the FMA-heavy pipe.  On GB300
// a LOP3 or shift holds the ALU for 2 clocks, and a 32x32->64 multiply the FMA-heavy
// pipe for 4 and the ALU for 2 (probes: a multiply and n LOP3 take 2 + 2 n clocks,
// a 32-bit multiply and a LOP3 together 2).  A call of B trials has 15 + 2/B such
// multiplies, 17 + 2/B XORs and 8 field operations.  Gaussian N = 4, evaluations/s:
// 4.49e11 at first, 4.69e11 with one ALU operation fewer per field, 4.84e11 with
// B = 4 as well.
//
// Order of the compensated additions of a trial (the same for every blocking
// choice below, so that the results do not depend on how many trials a lane
// takes, and the single-scan and batched kernels agree bit for bit): with
// G = 5, each group's five samples enter in one step (LaneAcc::add_group), in
// group order; with G = 1, consecutive groups are paired and a last unpaired
// group enters alone.
template <int N, class F, int PREC, int B, class Acc>
__device__ __forceinline__ void lane_groups(const uint32_t* __restrict__ rk0,
                                            const uint32_t* __restrict__ rk1, uint32_t a2,
                                            uint32_t b0, const uint32_t (&b1)[B],
                                            const uint32_t (&b2)[B], const F& f,
                                            const FieldConst& fc, uint32_t q, uint32_t q_end,
                                            uint32_t step, Acc (&acc)[B]) {
  constexpr int G = group_samples(N);
  constexpr int C = group_calls(N);
  // Groups per loop block: about kCallsInFlight independent Philox chains
  // per lane (a group of C calls of B trials already has C B).  The FP64 path
  // draws one group at a time.
#ifdef ZMC_CALLS_IN_FLIGHT
  constexpr int kCalls = PREC == kPrecFP64 ? 1 : ZMC_CALLS_IN_FLIGHT;
#else
  constexpr int kCalls = PREC == kPrecFP64 ? 1 : F::kCallsInFlight;
#endif
  constexpr int kBlock = kCalls / (C * B) > 1 ? kCalls / (C * B) : 1;
  using T = decltype(eval_sample<N>(f, fc, static_cast<const uint32_t*>(nullptr), 0));
  // M0 * j for the lane's calls, carried along by 64-bit adds: call c of
  // group q has j = q C + c; the product for q C advances with the lane's
  // stride and call c adds the constant M0 c to it.
  StridedProduct sp;
  sp.init(q * C, step * C);
  // Words of call c of the current group, every trial: out[u][4 * at ..].
  auto call = [&](int c, auto& out, int at) {
    uint32_t H, L;
    sp.at(c, H, L);
    const PhiloxShared sh = philox_shared(a2, b0, H, L);
#pragma unroll
    for (int u = 0; u < B; ++u) philox_finish(sh, b1[u], b2[u], rk0, rk1, &out[u][4 * at]);
  };
  // Draw the words of V consecutive groups of this lane.
  auto draw = [&](auto& r) {
    constexpr int V = sizeof(r) / sizeof(r[0]);
#pragma unroll
    for (int i = 0; i < V; ++i) {
#pragma unroll
      for (int c = 0; c < C; ++c) call(c, r[i], c);
      sp.advance();
    }
  };
  if constexpr (G > 1) {
    constexpr int U = kBlock;
    auto consume = [&](const auto& r) {
      constexpr int V = sizeof(r) / sizeof(r[0]);
#pragma unroll
      for (int i = 0; i < V; ++i) {
#pragma unroll
        for (int u = 0; u < B; ++u) {
          T v[G];
#pragma unroll
          for (int g = 0; g < G; ++g) v[g] = eval_sample<N>(f, fc, r[i][u], g);
          acc[u].template add_group<G>(v);
        }
      }
    };
    if constexpr (U == 1 && C > 2) {
      // One long group at a time: each call is drawn just before the first
      // sample that reads it, so a call's words die once its last sample is
      // evaluated (fewer live registers than drawing all C calls first).
      for (; q < q_end; q += step) {
        uint32_t r[B][4 * C];
        T v[B][G];
#pragma unroll
        for (int g = 0; g < G; ++g) {
          const int c0 = g == 0 ? 0 : (g * N - 1) / kFieldsPerCall + 1;
          const int c1 = (g * N + N - 1) / kFieldsPerCall;
#pragma unroll
          for (int c = c0; c <= c1; ++c) call(c, r, c);
#pragma unroll
          for (int u = 0; u < B; ++u) v[u][g] = eval_sample<N>(f, fc, r[u], g);
        }
#pragma unroll
        for (int u = 0; u < B; ++u) acc[u].template add_group<G>(v[u]);
        sp.advance();
      }
    } else {
      for (; q + (U - 1) * step < q_end; q += U * step) {
        uint32_t r[U][B][4 * C];
        draw(r);
        consume(r);
      }
      if constexpr (U > 1) {
        for (; q < q_end; q += step) {
          uint32_t r[1][B][4 * C];
          draw(r);
          consume(r);
        }
      }
    }
  } else {
    // G == 1: consecutive groups are paired; U groups (U/2 pairs) per block.
    constexpr int U = kBlock >= 2 ? kBlock & ~1 : 2;
    auto consume = [&](const auto& r) {
      constexpr int V = sizeof(r) / sizeof(r[0]);
#pragma unroll
      for (int i = 0; i < V; i += 2)
#pragma unroll
        for (int u = 0; u < B; ++u)
          acc[u].add2(eval_sample<N>(f, fc, r[i][u], 0), eval_sample<N>(f, fc, r[i + 1][u], 0));
    };
    for (; q + (U - 1) * step < q_end; q += U * step) {
      uint32_t r[U][B][4 * C];
      draw(r);
      consume(r);
    }
    // Fewer than U groups left: pairs, then a single group.
    if constexpr (U > 2) {
      for (; q + step < q_end; q += 2 * step) {
        uint32_t r[2][B][4 * C];
        draw(r);
        consume(r);
      }
    }
    if (q < q_end) {
      uint32_t r[1][B][4 * C];
      draw(r);
#pragma unroll
      for (int u = 0; u < B; ++u) acc[u].add(eval_sample<N>(f, fc, r[0][u], 0));
    }
  }
}

// The ragged last group of a unit when G does not divide S: its valid samples
// enter one at a time.
template <int N, class F, class Acc>
__device__ __forceinline__ void lane_tail_group(const uint32_t* __restrict__ rk0,
                                                const uint32_t* __restrict__ rk1,
                                                const PhiloxUnit& pu, const F& f,
                                                const FieldConst& fc, uint32_t q, int valid, Acc& acc) {
  constexpr int G = group_samples(N);
  constexpr int C = group_calls(N);
  uint32_t r[4 * C];
#pragma unroll
  for (int c = 0; c < C; ++c) philox_call(pu, rk0, rk1, q * C + c, &r[4 * c]);
#pragma unroll
  for (int g = 0; g < G; ++g)
    if (g < valid) acc.add(eval_sample<N>(f, fc, r, g));
}

// Sums of one lane over its part of split `split` of trials t .. t + B - 1 of
// point p.
template <int N, class F, int PREC, int B>
__device__ __forceinline__ void sample_trials(const ScanArgs& a, const FieldConst& fc,
                                              const uint32_t* rk0, const uint32_t* rk1,
                                              const F& f, int64_t p, uint32_t t, int64_t split,
                                              int lane, double* s1, double* s2) {
  constexpr int G = group_samples(N);
  typename FxOf<F, PREC>::Acc acc[B];
  const int64_t q0 = split * a.gps;
  const int64_t q1 = min(q0 + a.gps, a.ngroups);
  if constexpr (!F::kUsesSamples) {
    // g does not depend on y: the stream is not drawn at all.
    for (int64_t q = q0 + lane; q < q1; q += a.lanes) {
      const int64_t left = a.S - q * G;
      const int cnt = left < G ? static_cast<int>(left) : G;
      for (int g = 0; g < cnt; ++g) acc[0].add(f.eval(nullptr));
    }
  } else {
    PhiloxUnit pu[B];
    uint32_t b1[B], b2[B];
#pragma unroll
    for (int u = 0; u < B; ++u) {
      pu[u] = philox_unit(rk0, rk1, static_cast<uint64_t>(p), t + u);
      b1[u] = pu[u].b1;
      b2[u] = pu[u].b2;
    }
    const int64_t nfull = a.S / G;
    const int64_t qf = min(q1, nfull);
    if (q0 + lane < qf)
      lane_groups<N, F, PREC, B>(rk0, rk1, pu[0].a2, pu[0].b0, b1, b2, f, fc,
                                 static_cast<uint32_t>(q0 + lane), static_cast<uint32_t>(qf),
                                 static_cast<uint32_t>(a.lanes), acc);
    if (G > 1) {
      const int valid = static_cast<int>(a.S - nfull * G);
      if (valid > 0 && nfull >= q0 && nfull < q1 && ((nfull - q0) & (a.lanes - 1)) == lane)
#pragma unroll
        for (int u = 0; u < B; ++u)
          lane_tail_group<N, F>(rk0, rk1, pu[u], f, fc, static_cast<uint32_t>(nfull), valid,
                                acc[u]);
    }
  }
#pragma unroll
  for (int u = 0; u < B; ++u) {
    s1[u] = acc[u].sum1();
    s2[u] = acc[u].sum2();
  }
}

// The same for one trial with an FP64 functor, for parameters outside a
// fixed-point functor's range.  Not inlined, so that it takes no registers from
// the usual path.
template <int N, class F, int PREC>
__device__ __noinline__ void sample_unit_wide(const ScanArgs& a, const void* table, int64_t p,
                                              uint32_t t, int64_t split, int lane, double* s1,
                                              double* s2) {
  F f{};
  load_params<N>(a, table, static_cast<const float*>(nullptr), p, f);
  sample_trials<N, F, PREC, 1>(a, a.field, a.rk0, a.rk1, f, p, t, split, lane, s1, s2);
}

// The work of the `lanes` threads of lane group w: `trials` trials from t on of
// grid point first + lp, sample split `split`.  The groups with four trials come
// first, then those with two, then single trials (lu4, lu2: how many).
struct LaneWork {
  int64_t lp, split;
  uint32_t t;
  int trials;
};

__device__ __forceinline__ int lane_trials(const ScanArgs& a, int64_t w) {
  return w < a.lu4 ? 4 : w < a.lu4 + a.lu2 ? 2 : 1;
}

template <int MAXB>
__device__ __forceinline__ LaneWork lane_work(const ScanArgs& a, int64_t w) {
  int per = a.T;  // lane groups of this size per point and split
  LaneWork k;
  k.trials = 1;
  k.t = 0;
  if constexpr (MAXB > 1) {
    k.trials = lane_trials(a, w);
    if (k.trials == 4) {
      per = a.T >> 2;
    } else if (k.trials == 2) {
      w -= a.lu4;
      k.t = a.lu4 ? a.T & ~3 : 0;
      per = (a.T - static_cast<int>(k.t)) >> 1;
    } else {
      w -= a.lu4 + a.lu2;
      k.t = a.lu2 ? a.T & ~1 : a.lu4 ? a.T & ~3 : 0;
      per = a.T - static_cast<int>(k.t);
    }
  }
  const int64_t unit = w / a.splits;
  k.split = w - unit * a.splits;
  k.lp = unit / per;
  k.t += static_cast<uint32_t>(k.trials) * static_cast<uint32_t>(unit - k.lp * per);
  return k;
}

// Work of one lane of lane group w: decode, prepare, sample, sum; the sums of
// its trials in s1, s2 (zero beyond them).  rk0/rk1 are the ten Philox round
// keys (parameter space in the single-scan kernel, uniform registers in the
// batched one); fx the fixed-point functors' table.
template <int N, class F, int PREC>
__device__ __forceinline__ void lane_sums(const ScanArgs& a, const FieldConst& fc,
                                          const uint32_t* rk0, const uint32_t* rk1,
                                          const void* table, const float* dimc,
                                          const int64_t* fx, const LaneWork& k, int lane,
                                          double* s1, double* s2) {
  const int64_t p = a.first + k.lp;
  if (!ZMC_CHECK(a.dbg, k.lp >= 0 && k.lp < a.count && k.split < a.splits &&
                            k.t + k.trials <= static_cast<uint32_t>(a.T),
                 kDbgGridIndex, k.lp))
    return;

  F f{};
  load_params<N>(a, table, dimc, p, f);
  if constexpr (FxOf<F, PREC>::kTable != kFxNone) {
    if (!f.in_range()) {
      sample_unit_wide<N, typename FxOf<F, PREC>::Wide, PREC>(a, table, p, k.t, k.split, lane,
                                                              s1, s2);
      return;
    }
    if constexpr (FxOf<F, PREC>::kTable != kFxNoTable) f.fx = fx;
  }
  if constexpr (max_trials<N, F, PREC>() > 2) {
    if (k.trials == 4) {
      sample_trials<N, F, PREC, 4>(a, fc, rk0, rk1, f, p, k.t, k.split, lane, s1, s2);
      return;
    }
  }
  if constexpr (max_trials<N, F, PREC>() > 1) {
    if (k.trials == 2) {
      sample_trials<N, F, PREC, 2>(a, fc, rk0, rk1, f, p, k.t, k.split, lane, s1, s2);
      return;
    }
  }
  sample_trials<N, F, PREC, 1>(a, fc, rk0, rk1, f, p, k.t, k.split, lane, s1, s2);
}

// Cross-warp sums of a block: 16 warps of up to 2 kMaxLaneTrials values.
constexpr int kReduceDoubles = 16 * 2 * kMaxLaneTrials;

// Reduce V values per thread (a power of two) over the `lanes` threads of each
// lane group, in a fixed order.  Within a warp: a butterfly in which, at each of
// the first steps, the two partners each keep half of the values they still hold
// and send the other half, so that V values cost V - 1 FP64 adds and one more
// per further step instead of V per step (an FP64 add holds the SM's one FP64
// unit for 16 clocks a warp; for four trials in 32 lanes 9 adds instead of 40).
// Every value's sum is the same tree of the same numbers either way.  Wider lane
// groups then add the warps' sums from shared memory, in order.  Every thread of
// the block calls it; afterwards the threads of a lane group's first warp hold
// its sums, this one values owner[0] .. owner[0] + owner[1] - 1 in x[0 ..).
template <int V>
__device__ __forceinline__ void reduce_lanes(const ScanArgs& a, double (&x)[V], double* red,
                                             int* owner) {
  const int width = a.lanes < 32 ? a.lanes : 32;
  const int lane = threadIdx.x & 31;
  int held = V;   // values this thread still holds, in x[0 .. held)
  int first = 0;  // the first of them
  int m = width >> 1;
#pragma unroll
  for (int h = V >> 1; h >= 1; h >>= 1) {
    if (m < 1) break;
    const bool up = (lane & m) != 0;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const double mine = up ? x[i + h] : x[i];
      const double other = up ? x[i] : x[i + h];
      x[i] = mine + __shfl_xor_sync(0xffffffffu, other, m);
    }
    if (up) first += h;
    held = h;
    m >>= 1;
  }
  for (; m >= 1; m >>= 1)  // one value left (held == 1)
    x[0] += __shfl_xor_sync(0xffffffffu, x[0], m);
  owner[0] = first;
  owner[1] = held;
  if (a.lanes > 32) {
    // x[0] is value `first` of this warp (held == 1: 32 lanes >= V)
    const int warp = threadIdx.x >> 5;
    if ((lane & (32 / V - 1)) == 0) red[warp * V + first] = x[0];
    __syncthreads();
    const int wpu = a.lanes >> 5;
    if ((warp & (wpu - 1)) == 0) {
      double t = red[warp * V + first];
      for (int w = 1; w < wpu; ++w) t += red[(warp + w) * V + first];
      x[0] = t;
    }
  }
}

// Reduce a block's lane sums (sum g of V / 2 trials, then sum g^2) and write the
// lane groups' partial sums, each from one thread.
template <int V>
__device__ __forceinline__ void write_sums(const ScanArgs& a, const LaneWork& k, bool active,
                                           int lane, double (&x)[V], double* red) {
  int owner[2];
  reduce_lanes<V>(a, x, red, owner);
  const int width = a.lanes < 32 ? a.lanes : 32;
  const int copies = width * owner[1] / V;  // threads that hold the same values
  if (active && lane < width && (copies <= 1 || (lane & (copies - 1)) == 0)) {
#pragma unroll
    for (int i = 0; i < V; ++i) {
      if (i >= owner[1]) break;
      const int v = owner[0] + i, u = v & (V / 2 - 1);
      if (u >= k.trials) continue;
      const int64_t us = (k.lp * a.T + k.t + u) * a.splits + k.split;
      if (ZMC_CHECK(a.dbg, us >= 0 && us < a.n_us, kDbgPartialSlot, us))
        a.partial[2 * us + (v >= V / 2 ? 1 : 0)] = x[i];
    }
  }
}

// A block's lane groups first_w .. first_w + units - 1 (units <= blockDim.x /
// lanes): sample, reduce and write each trial's partial sums.  Every thread of
// the block calls it.
template <int N, class F, int PREC>
__device__ __forceinline__ void block_work(const ScanArgs& a, const FieldConst& fc,
                                           const uint32_t* rk0, const uint32_t* rk1,
                                           const void* table, const float* dimc,
                                           const int64_t* fx, int64_t first_w, int units,
                                           double* red) {
  constexpr int kB = max_trials<N, F, PREC>();
  const int lane = threadIdx.x & (a.lanes - 1);
  const int local = threadIdx.x >> a.lanes_log2;
  const bool active = local < units;
  LaneWork k{0, 0, 0, 0};
  double x[2 * kB];  // sum g of the trials, then sum g^2
#pragma unroll
  for (int u = 0; u < 2 * kB; ++u) x[u] = 0.0;
  if (active) {
    k = lane_work<kB>(a, first_w + local);
    lane_sums<N, F, PREC>(a, fc, rk0, rk1, table, dimc, fx, k, lane, x, x + kB);
  }
  if constexpr (kB > 1) {
    // lane groups of one size lie together, the larger ones first
    if (lane_trials(a, first_w) > 1) {
      write_sums<2 * kB>(a, k, active, lane, x, red);
      return;
    }
  }
  double y[2] = {x[0], x[kB]};
  write_sums<2>(a, k, active, lane, y, red);
}

template <int N, class F, int PREC>
__global__ void __launch_bounds__(ZMC_LB_THREADS, ZMC_LB_MIN_BLOCKS)
scan_kernel(const __grid_constant__ ScanArgs a) {
  extern __shared__ double smem[];
  __shared__ double red[kReduceDoubles];
  __shared__ float dimc[3 * ZMC_MAX_N];
  const int64_t* fx = nullptr;
  if constexpr (FxOf<F, PREC>::kTable == kFxCosTable || FxOf<F, PREC>::kTable == kFxExpTable) {
    __shared__ int64_t fx_table[FxOf<F, PREC>::kEntries];
    FxOf<F, PREC>::fill(fx_table);
    if (!a.stage_smem) __syncthreads();  // else stage_lists ends with one
    fx = fx_table;
  }
  const void* table = stage_lists<N, F>(a, smem, dimc);
  const int per_block = blockDim.x >> a.lanes_log2;
  const int64_t first_w = static_cast<int64_t>(blockIdx.x) * per_block;
  const int64_t left = a.n_lw - first_w;
  block_work<N, F, PREC>(a, a.field, a.rk0, a.rk1, table, dimc, fx, first_w,
                         left < per_block ? static_cast<int>(left) : per_block, red);
}

#ifndef __CUDACC_RTC__
// Ask for more than the 48 KB of shared memory that a kernel gets unasked, where
// `smem` bytes of lists beside `table_bytes` of tables may need it.  The limit belongs
// to the kernel and not to the launch, so every call asks for the same, the longest
// lists: no thread takes back what another is about to launch with.
constexpr size_t kOtherSmem = 4096;  // bound of the sums', constants' and counters' arrays
static_assert(kReduceDoubles * sizeof(double) + 3 * ZMC_MAX_N * sizeof(float) + 256 <= kOtherSmem,
              "static shared memory beside the tables");
template <class Kernel>
cudaError_t allow_smem(Kernel kernel, size_t table_bytes, size_t smem) {
  if (smem + table_bytes + kOtherSmem <= 48 * 1024) return cudaSuccess;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(kMaxSmemVals * sizeof(double)));
}

template <int N, class F, int PREC>
int launch_scan(const ScanArgs& a, int block, int64_t grid, size_t smem, void* stream) {
  const cudaError_t e =
      allow_smem(scan_kernel<N, F, PREC>, FxOf<F, PREC>::kStaticBytes, smem);
  if (e != cudaSuccess) return static_cast<int>(e);
  scan_kernel<N, F, PREC><<<static_cast<unsigned>(grid), block, smem,
                            static_cast<cudaStream_t>(stream)>>>(a);
  return static_cast<int>(cudaGetLastError());
}
#endif  // __CUDACC_RTC__

}  // namespace zmc
