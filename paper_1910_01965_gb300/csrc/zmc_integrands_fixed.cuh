// zmc_integrands_fixed.cuh — the FP64 integrands in 64-bit fixed point.
//
// Each functor evaluates its integrand from the sample's 23-bit fields with the
// arithmetic of zmc_fixed64.cuh.  `set`/`finish` turn the box and the
// parameters into fixed-point constants; `in_range` says whether they are large
// and small enough for that.  Out of range, and for NaN or infinite parameters, the
// unit is sampled by the FP64 functor named in FxOf (zmc_integrands.cuh, suffix
// Wide).
//
// The cosines and sines have an absolute resolution (2^-56 in a cosine, 2^-60 in a
// product and in g^2), so they are in range only where g is not small over the
// whole box: R, the root mean square of g, follows from the phases' ranges.  The lines
// lie where the error is no larger than the FP64 functor's, sample by sample, even in
// boxes whose sides and parameters it represents without rounding.  Root mean square
// over R and R^2 against 80-bit arithmetic, largest of some 800 boxes each, fixed point
// over FP64: products g 0.91 (N = 1), 0.55 (2), 0.29 (8), g^2 0.91, 0.78, 0.77;
// sine-sum g 1.00, g^2 0.96.  At R = 2^-6 instead g^2 is 5.6 times off for N = 2.
//
// What bounds them (ncu, registry grids): the FMA-heavy pipe, 82-87 % busy, and
// beside it the ALU, which a multiply holds for 2 clocks too; the FP64 unit, 92 %
// busy before, is left to the sums.  An N = 2 cosine product has 22 multiplies and
// about 45 other operations per dimension.  GB300, evaluations/s before and after
// (10^5-point grids): cos-product N = 1 2.6e10 -> 2.1e11, N = 8 3.4e9 -> 2.9e10;
// Gaussian N = 4 2.3e10 -> 1.2e11; oscillatory N = 6 1.4e10 -> 7.9e10; polynomial
// N = 1 1.1e11 -> 2.3e11, N = 8 1.7e10 -> 4.8e10.  Tables of 2048 steps, 20 and
// 16 KB a block: the two 8-byte loads of a cosine take 12 shared-memory wavefronts
// (31 % of the load unit); fewer steps need a further Taylor term, more shared
// memory buys none less.  Products of 64-bit numbers with IMAD.WIDE and 64-bit
// addends instead of high-half multiplies are 10 % slower.
//
// With u = (2 v + 1) 2^-24 and w = b - a (rounded to FP64, as there):
// y = a + w 2^-24 + (w 2^-23) v.
#pragma once

#include "zmc_fixed64.cuh"
#include "zmc_scan_kernel.cuh"

namespace zmc {

// Lane sums of values g with |g| <= 1, held as 2^62 g + 2^31: exact sums of g
// and of g^2 rounded to 2^-SCALE each, converted to FP64 once per lane.  Integer sums
// cost 5 adds against 64 SMSP clocks for one FP64 add.
template <int SCALE>
struct FxLaneAcc {
  FxSum a1, a2;
  uint64_t n = 0;
  __device__ __forceinline__ void sum(int64_t g) {
    a1.add(g);
    a2.add(fx_square<SCALE>(g));
  }
  __device__ __forceinline__ void add(int64_t g) {
    sum(g);
    n += 1;
  }
  __device__ __forceinline__ void add2(int64_t a, int64_t b) {
    sum(a);
    sum(b);
    n += 2;
  }
  template <int K>
  __device__ __forceinline__ void add_group(const int64_t* v) {
#pragma unroll
    for (int i = 0; i < K; ++i) sum(v[i]);
    n += K;
  }
  __device__ __forceinline__ double sum1() const { return a1.value(n, 62); }
  __device__ __forceinline__ double sum2() const { return a2.value(0, SCALE); }
};

// prod_k cos(x_k y_k): a 96-bit phase per dimension.  In range: phases below
// 2^20 radians; the mean of each factor's square over the box at least 2^-6, and of g^2
// at least 2^-8 (N <= 5) or 2^-11 (the least over boxes that reach from 0 is 2^-10.8).
template <int N>
struct CosProd64 {
  static constexpr bool kPerDim = true;
  static constexpr bool kTable = false;
  static constexpr bool kUsesSamples = true;
  static constexpr int kCallsInFlight = 1;
  static constexpr int kFixedM = 0;
  using unit_t = uint32_t;
  const int64_t* fx;
  bool ok = true;
  float mean2 = 1.0f;  // of g^2
  uint32_t b0[N], b1[N], b2[N];
  uint64_t c[N];
  __device__ void set(int i, double xi, double ai, double bi) {
    const double w = bi - ai;
    ok = ok && fx_below(xi * w, 20) && fx_below(xi * ai, 20);
    const FxTurns b = fx_turns_mul(xi, w, -23);
    b0[i] = b.w0;
    b1[i] = b.w1;
    b2[i] = b.w2;
    const FxTurns xa = fx_turns_mul(xi, ai, 0);
    c[i] = fx_phase0(fx_turns_add(xa, fx_turns_sar(b, 1)));
    const uint32_t xw = fx_lead23(b);
    const float m = fx_mean_cos2(2 * xa.w2 + xw, fx_sinc(static_cast<float>(xi * w), xw));
    ok = ok && m >= 0x1p-6f;
    mean2 *= m;
  }
  __device__ bool in_range() const { return ok && mean2 >= (N <= 5 ? 0x1p-8f : 0x1p-11f); }
  __device__ int64_t eval(const uint32_t* v) const {
    int64_t g = fx_cos(fx_phase_step(c[0], v[0], b0[0], b1[0], b2[0]), fx);
#pragma unroll
    for (int k = 1; k < N; ++k)
      g = fx_mul62(g, fx_cos(fx_phase_step(c[k], v[k], b0[k], b1[k], b2[k]), fx));
    return g;
  }
};

// sin(sum_k y_k + sum_l x_l) as the cosine a quarter turn behind.  In range:
// the parameters' sum and the box's sides and corner below 2^20; the mean of g^2 over
// the box at least 2^-6.
template <int N>
struct SinSum64 {
  static constexpr bool kPerDim = false;
  static constexpr bool kTable = false;
  static constexpr bool kUsesSamples = true;
  static constexpr int kCallsInFlight = 1;
  static constexpr int kFixedM = 0;
  using unit_t = uint32_t;
  const int64_t* fx;
  bool ok = true;
  double xsum;
  uint32_t b0[N], b1[N], b2[N];
  uint64_t c;
  __device__ void add(double xi) { xsum += xi; }
  __device__ void finish(const double* lo, const double* hi) {
    ok = fx_below(xsum, 20);
    FxTurns t = fx_turns_add(fx_turns(xsum, 0), {0, 0, 0xC0000000u});
    uint32_t widths = 0;
    float sincs = 1.0f;
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const double w = hi[k] - lo[k];
      ok = ok && fx_below(lo[k], 20) && fx_below(w, 20);
      const FxTurns b = fx_turns(w, -23);
      b0[k] = b.w0;
      b1[k] = b.w1;
      b2[k] = b.w2;
      t = fx_turns_add(t, fx_turns_add(fx_turns(lo[k], 0), fx_turns_sar(b, 1)));
      widths += fx_lead23(b);
      sincs *= fx_sinc(static_cast<float>(w), fx_lead23(b));
    }
    c = fx_phase0(t);
    // t lies half a field of each dimension (2^-24 of its width) above the corner
    ok = ok && fx_mean_cos2(2 * t.w2 + widths, sincs) >= 0x1p-6f;
  }
  __device__ bool in_range() const { return ok; }
  __device__ int64_t eval(const uint32_t* v) const {
    uint64_t th = c;
#pragma unroll
    for (int k = 0; k < N; ++k) th = fx_phase_step(th, v[k], b0[k], b1[k], b2[k]);
    return fx_cos(th, fx);
  }
};

// frac(0.1 a b 2^k / (2 pi)) from the exact products.
__device__ __forceinline__ FxTurns fx_turns_quad(double a, double b, int k) {
  const double p = a * b;
  return fx_turns_add(fx_turns_mul(kOscQuad, p, k), fx_turns_mul(kOscQuad, fma(a, b, -p), k));
}

// cos(sum_k x_k y_k + 0.1 y_k^2).  In turns, dimension k adds
//   (q v + l) v + const,  q = 0.1 w^2 2^-46,  l = (x w + 0.2 a w) 2^-23 + q,
// by Horner's rule with q 2^23 and l held to 96 bits.  In range: box within
// 2^10 of the origin, x w and x a below 2^20; phases that reach over a radian,
// or over which |cos| stays above 1/4.
template <int N>
struct Osc64 {
  static constexpr bool kPerDim = true;
  static constexpr bool kTable = false;
  static constexpr bool kUsesSamples = true;
  static constexpr int kCallsInFlight = 1;
  static constexpr int kFixedM = 0;
  using unit_t = uint32_t;
  const int64_t* fx;
  bool ok = true;
  uint32_t q0[N], q1[N], q2[N];  // q 2^23, below 1/2
  uint32_t l0[N], l1[N], l2[N];
  uint64_t c = uint64_t(1) << 52;  // half a table step
  float width = 0.0f, drop = 0.0f;  // of the phases' range
  __device__ void set(int i, double xi, double ai, double bi) {
    const double w = bi - ai;
    ok = ok && fx_below(xi * w, 20) && fx_below(xi * ai, 20) && fx_below(ai, 10) &&
         fx_below(w, 10);
    const FxTurns xw = fx_turns_mul(xi, w, -23);
    const FxTurns q = fx_turns_quad(w, w, -23);
    const FxTurns aw = fx_turns_quad(ai, w, -22);
    const FxTurns lin = fx_turns_add(xw, aw);
    const FxTurns l = fx_turns_add(lin, fx_turns_sar(q, 23));
    q0[i] = q.w0;
    q1[i] = q.w1;
    q2[i] = q.w2;
    l0[i] = l.w0;
    l1[i] = l.w1;
    l2[i] = l.w2;
    // x a + 0.1 a^2 + half a field of the linear part + 0.1 w^2 2^-48
    const FxTurns k0 = fx_turns_add(fx_turns_mul(xi, ai, 0), fx_turns_quad(ai, ai, 0));
    const FxTurns k1 = fx_turns_add(fx_turns_sar(lin, 1), fx_turns_sar(q, 25));
    const FxTurns k = fx_turns_add(k0, k1);
    c += (static_cast<uint64_t>(k.w2) << 32) | k.w1;
    const FxReach r = fx_quad_reach(static_cast<float>(xi), static_cast<float>(kOscQuad),
                                    static_cast<float>(ai), static_cast<float>(w));
    width += r.width;
    drop += r.drop;
  }
  __device__ bool in_range() const {
    const uint32_t at = static_cast<uint32_t>((c - (uint64_t(1) << 52)) >> 32);
    return ok && (width >= 1.0f ||
                  fx_cos_range(at - static_cast<uint32_t>(drop * 683565275.6f), width));
  }
  __device__ int64_t eval(const uint32_t* v) const {
    uint64_t th = c;
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const uint32_t f = v[k] << 9;  // v 2^-23 as a 32-bit fraction
      const uint64_t p1 = fx_uwide(f, q1[k]) + fx_umulhi(f, q0[k]);
      const uint64_t p2 = fx_uwide(f, q2[k]) + (p1 >> 32);
      const FxTurns s = fx_turns_add({static_cast<uint32_t>(p1), static_cast<uint32_t>(p2),
                                      static_cast<uint32_t>(p2 >> 32)},
                                     {l0[k], l1[k], l2[k]});
      th = fx_phase_step(th, v[k], s.w0, s.w1, s.w2);
    }
    return fx_cos(th, fx);
  }
};

// 2^-q, q = sum_k d_k^2, d = scale (y - x) as a signed 5.59-bit number.  In
// range: |d| < 15.9 over the box in every dimension and q < 990, so that 2^-q
// is a normal double.  The sums stay FP64 (the FP64 unit is otherwise idle).
template <int N>
struct Gauss64 {
  static constexpr bool kPerDim = true;
  static constexpr bool kTable = false;
  static constexpr bool kUsesSamples = true;
  static constexpr int kCallsInFlight = 1;
  static constexpr int kFixedM = 0;
  using unit_t = uint32_t;
  // 2^61 sqrt(log2(e) / 0.18)
  static constexpr uint64_t kScale61 = 0x5a9825b501cd145cull;
  const int64_t* fx;
  bool ok = true;
  float qmax = 0.0f;
  uint32_t w0[N], w1[N];
  int64_t c[N];
  __device__ void set(int i, double xi, double ai, double bi) {
    const double w = bi - ai;
    // a - x as an exact sum of two doubles
    const double s = ai - xi, bb = s - ai;
    const double e = (ai - (s - bb)) + (-xi - bb);
    const float m = 2.8310728f * fmaxf(fabsf(static_cast<float>(s)),
                                       fabsf(static_cast<float>(bi - xi)));
    qmax = fmaf(m, m, qmax);
    ok = ok && m < 15.9f && qmax < 990.0f && xi == xi;  // fmaxf drops a NaN
    const uint64_t cw = static_cast<uint64_t>(fx_scale59(w, kScale61));
    w0[i] = static_cast<uint32_t>(cw);
    w1[i] = static_cast<uint32_t>(cw >> 32);
    c[i] = fx_scale59(s, kScale61) + fx_scale59(e, kScale61) +
           static_cast<int64_t>(((cw >> 23) + 1) >> 1) + kFxBias;
  }
  __device__ bool in_range() const { return ok; }
  __device__ double eval(const uint32_t* v) const {
    uint64_t q = uint64_t(1) << 42;  // half a table step
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const uint32_t f = v[k] << 9;  // v 2^-23 as a 32-bit fraction
      const int64_t d = c[k] + static_cast<int64_t>(fx_uwide(f, w1[k]) + fx_umulhi(f, w0[k]));
      const int32_t h = fx_top(d);
      const int32_t t = fx_mulhi(h, fx_low(d));
      q += static_cast<uint64_t>(fx_wide(h, h) + (2 * t + 1));
    }
    return fx_exp2neg(q, fx);
  }
};

// prod_k (1 + x_k y_k^2), each factor over a power of two above its largest
// value in the box, so that every product is at most 1; the powers return in g's
// exponent.  In range: factors below 2^60.  The sums stay FP64.
template <int N>
struct Poly64 {
  static constexpr bool kPerDim = true;
  static constexpr bool kTable = false;
  static constexpr bool kUsesSamples = true;
  static constexpr int kCallsInFlight = 1;
  static constexpr int kFixedM = 0;
  using unit_t = uint32_t;
  bool ok = true;
  int scale = 0;
  int64_t c0[N], c1[N], c2[N];
  __device__ void set(int i, double xi, double ai, double bi) {
    const FxPoly p = fx_poly(xi, ai, bi - ai);
    ok = ok && p.ok;
    scale += p.s;
    c0[i] = p.c0;
    c1[i] = p.c1;
    c2[i] = p.c2;
  }
  __device__ bool in_range() const { return ok; }
  __device__ double eval(const uint32_t* v) const {
    int64_t g = fx_poly_eval(c0[0], c1[0], c2[0], v[0]);
    int e = scale;
#pragma unroll
    for (int k = 1; k < N; ++k) {
      if (k > 1 && k % 2 == 0) g = fx_normalise(g, &e);  // every second factor
      g = fx_mul62(g, fx_poly_eval(c0[k], c1[k], c2[k], v[k]));
    }
    return fx_to_double(g - kFxBias, e);
  }
};

__device__ __forceinline__ void fx_fill(int64_t* dst, const int64_t* src, int n) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
}

// Both tables, the cosines first (the batched kernel).
__device__ __forceinline__ void fx_fill_tables(int64_t* dst) {
  fx_fill(dst, kFxTables.c, kFxCosEntries);
  fx_fill(dst + kFxCosEntries, kFxTables.e, kFxExpEntries);
}

template <int N>
struct FxOf<Poly64<N>, kPrecFP64> {
  static constexpr int kTable = kFxNoTable;
  static constexpr size_t kStaticBytes = 0;
  using Wide = Poly64Wide<N>;
  using Acc = LaneAcc<kPrecFP64>;
};

template <class W, int SCALE = 60>
struct FxCosOf {
  static constexpr int kTable = kFxCosTable;
  static constexpr int kEntries = kFxCosEntries;
  static constexpr size_t kStaticBytes = kEntries * sizeof(int64_t);
  using Wide = W;
  using Acc = FxLaneAcc<SCALE>;
  static __device__ __forceinline__ void fill(int64_t* dst) {
    fx_fill(dst, kFxTables.c, kEntries);
  }
};
// (products of four and more cosines are small enough to need the finer squares)
template <int N>
struct FxOf<CosProd64<N>, kPrecFP64> : FxCosOf<CosProd64Wide<N>, N <= 3 ? 60 : 62> {};
template <int N>
struct FxOf<SinSum64<N>, kPrecFP64> : FxCosOf<SinSum64Wide<N>> {};
template <int N>
struct FxOf<Osc64<N>, kPrecFP64> : FxCosOf<Osc64Wide<N>> {};
template <int N>
struct FxOf<Gauss64<N>, kPrecFP64> {
  static constexpr int kTable = kFxExpTable;
  static constexpr int kEntries = kFxExpEntries;
  static constexpr size_t kStaticBytes = kEntries * sizeof(int64_t);
  using Wide = Gauss64Wide<N>;
  using Acc = LaneAcc<kPrecFP64>;
  static __device__ __forceinline__ void fill(int64_t* dst) {
    fx_fill(dst, kFxTables.e, kEntries);
  }
};

}  // namespace zmc
