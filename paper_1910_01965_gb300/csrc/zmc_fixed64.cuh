// zmc_fixed64.cuh — 64-bit fixed-point arithmetic for the FP64 integrands.
//
// GB300 has one FP64 unit per SM (2 lanes per clock: an FP64 instruction holds
// it for 16 clocks a warp), against 32 lanes per clock for 32x32->64 integer
// multiplies.  The FP64 integrands are therefore evaluated in 64-bit fixed
// point on the integer pipes.  The cosine is held to an absolute 2^-56 (it is
// at most 1; one FP64 rounding there is 2^-54), a product of cosines to 2^-60 and
// g^2 to 2^-60 or 2^-62, so this holds what FP64 does only where g is not small all over the
// box: the range tests (fx_mean_cos2, fx_cos_range) send the others to the FP64
// functors.  The exponential and the polynomial keep their bits at any size.  Two
// building blocks:
//
//  * phases in turns: theta = phase / (2 pi) mod 1 as a 64-bit fraction, so the
//    reduction of the argument is integer wrap-around and costs nothing; cos of
//    it from a 2048-step table and a Taylor step of degree 4 in the remainder;
//  * 2^-q for q in [0, 1000) as a 10.54-bit number, from a 2048-step table of
//    2^-i/2048 and a Taylor step of degree 4.
//
// 64x64-bit products are formed from 32-bit halves with the low half signed
// (the value is rounded, not cut, to its high half): a value is kept with a
// bias of 2^31, whose high word then is the rounded high half and whose low
// word with the top bit flipped the signed low half.  The product of the two
// low halves, below 2^-62 of the result, is left out.
//
// The functions are plain C++ as well: the CPU tests compile this file with
// the host compiler and compare them with quad precision.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define ZMC_FX __device__ __forceinline__
#define ZMC_FX_TABLE static __device__ const
#else
#define ZMC_FX inline
#define ZMC_FX_TABLE static const
#endif

namespace zmc {

// ------------------------------------------------------------- primitives --
#if defined(__CUDA_ARCH__)
ZMC_FX int32_t fx_mulhi(int32_t a, int32_t b) { return __mulhi(a, b); }
ZMC_FX uint32_t fx_umulhi(uint32_t a, uint32_t b) { return __umulhi(a, b); }
ZMC_FX uint64_t fx_umulhi64(uint64_t a, uint64_t b) { return __umul64hi(a, b); }
ZMC_FX uint64_t fx_double_bits(double v) {
  return static_cast<uint64_t>(__double_as_longlong(v));
}
ZMC_FX double fx_bits_double(uint64_t v) {
  return __longlong_as_double(static_cast<long long>(v));
}
ZMC_FX int fx_clz(uint32_t v) { return __clz(static_cast<int>(v)); }
ZMC_FX float fx_cosf(float v) { return __cosf(v); }
#else
inline int32_t fx_mulhi(int32_t a, int32_t b) {
  return static_cast<int32_t>((static_cast<int64_t>(a) * b) >> 32);
}
inline uint32_t fx_umulhi(uint32_t a, uint32_t b) {
  return static_cast<uint32_t>((static_cast<uint64_t>(a) * b) >> 32);
}
inline uint64_t fx_umulhi64(uint64_t a, uint64_t b) {
  return static_cast<uint64_t>((static_cast<unsigned __int128>(a) * b) >> 64);
}
inline uint64_t fx_double_bits(double v) {
  uint64_t u;
  __builtin_memcpy(&u, &v, 8);
  return u;
}
inline double fx_bits_double(uint64_t u) {
  double v;
  __builtin_memcpy(&v, &u, 8);
  return v;
}
inline int fx_clz(uint32_t v) { return v ? __builtin_clz(v) : 32; }
inline float fx_cosf(float v) { return __builtin_cosf(v); }
#endif

ZMC_FX int64_t fx_wide(int32_t a, int32_t b) { return static_cast<int64_t>(a) * b; }
ZMC_FX uint64_t fx_uwide(uint32_t a, uint32_t b) { return static_cast<uint64_t>(a) * b; }
ZMC_FX int32_t fx_top(int64_t v) { return static_cast<int32_t>(v >> 32); }
// The signed low half of a value kept with a bias of 2^31.
ZMC_FX int32_t fx_low(int64_t biased) {
  return static_cast<int32_t>(static_cast<uint32_t>(biased) ^ 0x80000000u);
}
constexpr int64_t kFxBias = int64_t(1) << 31;

// (a * b) >> 64 for a = (ah, al), b = (bh, bl) with signed low halves, |al bh|
// and |ah bl| below 2^62, without al bl; `round` is added (1 makes up for the
// two cuts, and half of what the caller shifts out makes its shift round).
ZMC_FX int64_t fx_mul(int32_t ah, int32_t al, int32_t bh, int32_t bl, int32_t round) {
  const int32_t t = fx_mulhi(al, bh) + (fx_mulhi(ah, bl) + round);
  return fx_wide(ah, bh) + t;
}

// ------------------------------------------------------------------ turns --
// A phase in turns, mod 1, with 96 fraction bits (w2 the most significant).
struct FxTurns {
  uint32_t w0, w1, w2;
};

ZMC_FX FxTurns fx_turns_add(FxTurns a, FxTurns b) {
  const uint64_t s0 = static_cast<uint64_t>(a.w0) + b.w0;
  const uint64_t s1 = static_cast<uint64_t>(a.w1) + b.w1 + (s0 >> 32);
  return {static_cast<uint32_t>(s0), static_cast<uint32_t>(s1),
          static_cast<uint32_t>(a.w2 + b.w2 + static_cast<uint32_t>(s1 >> 32))};
}

// Arithmetic shift right by s (1..31) of a turn in [-1/2, 1/2).
ZMC_FX FxTurns fx_turns_sar(FxTurns a, int s) {
  return {(a.w0 >> s) | (a.w1 << (32 - s)), (a.w1 >> s) | (a.w2 << (32 - s)),
          static_cast<uint32_t>(static_cast<int32_t>(a.w2) >> s)};
}

// frac(c 2^k / (2 pi)) to 96 bits, for |c 2^k| < 2^30 (k of either sign): the
// 53-bit mantissa times floor(2^(e + 160) / (2 pi)), cut out of the constant
// 2^192 / (2 pi), of which bits 64..159 are the result.  The cut constant is
// short by less than 1, the result by less than 2^-107 + 2^-96.
ZMC_FX FxTurns fx_turns(double c, int k) {
  const uint64_t u = fx_double_bits(c);
  const int ex = static_cast<int>((u >> 52) & 0x7ff);
  const uint64_t m = ex ? (u & 0xfffffffffffffull) | (uint64_t(1) << 52) : 0;
  const int sh = 192 - 160 - (ex - 1075 + k);  // right shift of the constant: >= 52
  if (m == 0 || sh >= 192) return {0, 0, 0};
  const uint64_t c0 = 0x36d8a5664f10e410ull, c1 = 0x7f09d5f47d4d3770ull,
                 c2 = 0x28be60db9391054aull;  // floor(2^192 / (2 pi))
  const int q = sh >> 6, b = sh & 63;
  const uint64_t d0 = q == 0 ? c0 : q == 1 ? c1 : c2;
  const uint64_t d1 = q == 0 ? c1 : q == 1 ? c2 : 0;
  const uint64_t d2 = q == 0 ? c2 : 0;
  const uint64_t i0 = b ? (d0 >> b) | (d1 << (64 - b)) : d0;
  const uint64_t i1 = b ? (d1 >> b) | (d2 << (64 - b)) : d1;
  const uint64_t i2 = d2 >> b;
  // bits 64.. of m * (i2:i1:i0)
  uint64_t lo = fx_umulhi64(m, i0);
  const uint64_t p1 = m * i1;
  lo += p1;
  const uint64_t hi = fx_umulhi64(m, i1) + m * i2 + (lo < p1 ? 1 : 0);
  FxTurns r{static_cast<uint32_t>(lo), static_cast<uint32_t>(lo >> 32),
            static_cast<uint32_t>(hi)};
  if (u >> 63) {
    r = {~r.w0, ~r.w1, ~r.w2};
    r = fx_turns_add(r, {1, 0, 0});
  }
  return r;
}

// frac(a b 2^k / (2 pi)) from the exact product of two doubles (|a b 2^k| < 2^29).
ZMC_FX FxTurns fx_turns_mul(double a, double b, int k) {
  const double p = a * b;
  return fx_turns_add(fx_turns(p, k), fx_turns(fma(a, b, -p), k));
}

// |v| below 2^e (false for NaN and infinities); e within [-1000, 1000].
ZMC_FX bool fx_below(double v, int e) {
  return static_cast<int>((fx_double_bits(v) >> 52) & 0x7ff) < 1023 + e;
}

// cos and sin of the turn with the leading 32 bits w, to about 2^-20.
ZMC_FX float fx_cos_lead(uint32_t w) {
  return fx_cosf(static_cast<float>(static_cast<int32_t>(w)) * 1.4629180792671596e-9f);
}
ZMC_FX float fx_sin_lead(uint32_t w) { return fx_cos_lead(w - 0x40000000u); }
// The leading bits of 2^23 times a turn.
ZMC_FX uint32_t fx_lead23(FxTurns t) { return (t.w2 << 23) | (t.w1 >> 9); }
// sin(w) / w for w = `lead` in turns mod 1.
ZMC_FX float fx_sinc(float w, uint32_t lead) {
  return fabsf(w) < 0x1p-6f ? 1.0f - w * w * (1.0f / 6.0f) : fx_sin_lead(lead) / w;
}
// The mean of cos^2 over phases that are a sum of uniform ones: `centre2` is twice
// the middle of their range in turns (leading bits), `sincs` the product of
// sin(w) / w over the widths w.
ZMC_FX float fx_mean_cos2(uint32_t centre2, float sincs) {
  return 0.5f + 0.5f * fx_cos_lead(centre2) * sincs;
}

// Whether |cos| stays above 1/4 over the phases from `lead` (turns, leading bits)
// to `width` radians further, or the phases reach over a radian.
ZMC_FX bool fx_cos_range(uint32_t lead, float width) {
  if (width >= 1.0f) return true;
  const float a = fx_cos_lead(lead);
  const float b = fx_cos_lead(lead + static_cast<uint32_t>(width * 683565275.6f));
  return a * b > 0.0f && fabsf(a) >= 0.25f && fabsf(b) >= 0.25f;
}

// x y + q y^2 for y from a to a + w, q > 0: how far its values reach (`width`) and
// by how much the lowest lies below the one at a (`drop`).
struct FxReach {
  float width, drop;
};
ZMC_FX FxReach fx_quad_reach(float x, float q, float a, float w) {
  const float u = x + 2.0f * q * a;  // the slope at a
  const float v = u + 2.0f * q * w;  // and at a + w
  if (u < 0.0f && v > 0.0f) {        // lowest inside, at a - u / (2 q)
    const float m = u * u / (4.0f * q), n = v * v / (4.0f * q);
    return {m > n ? m : n, m};
  }
  const float d = w * (u + q * w);
  return {fabsf(d), d < 0.0f ? -d : 0.0f};
}

// The 64-bit fraction of a turn plus half a table step: what fx_cos takes.
ZMC_FX uint64_t fx_phase0(FxTurns t) {
  return ((static_cast<uint64_t>(t.w2) << 32) | t.w1) + (uint64_t(1) << 52);
}

// theta + b v mod 1 for a 96-bit turn b and a 23-bit v: exact but for the cut
// of b's product at 2^-64.
ZMC_FX uint64_t fx_phase_step(uint64_t theta, uint32_t v, uint32_t b0, uint32_t b1,
                              uint32_t b2) {
  const uint64_t p = fx_uwide(v, b1) + fx_umulhi(v, b0);
  return theta + p + (static_cast<uint64_t>(v * b2) << 32);
}

// ------------------------------------------------------------------ tables --
constexpr int kFxCosEntries = 2560;  // 2048 steps of a turn, and 512 more for -sin
constexpr int kFxExpEntries = 2048;

struct FxTables {
  int64_t c[kFxCosEntries];  // 2^62 cos(2 pi i / 2048) + 2^31
  int64_t e[kFxExpEntries];  // 2^62 2^(-i / 2048) + 2^31
};

// 2^-126 a b, rounded down, for |a|, |b| <= 2^126.
constexpr __int128 fx_mul126(__int128 a, __int128 b) {
  const bool neg = (a < 0) != (b < 0);
  const unsigned __int128 x = static_cast<unsigned __int128>(a < 0 ? -a : a);
  const unsigned __int128 y = static_cast<unsigned __int128>(b < 0 ? -b : b);
  const uint64_t x0 = static_cast<uint64_t>(x), x1 = static_cast<uint64_t>(x >> 64);
  const uint64_t y0 = static_cast<uint64_t>(y), y1 = static_cast<uint64_t>(y >> 64);
  using U = unsigned __int128;
  const U mid = ((U(x0) * y0) >> 64) + static_cast<uint64_t>(U(x0) * y1) +
                static_cast<uint64_t>(U(x1) * y0);
  const U hi = U(x1) * y1 + ((U(x0) * y1) >> 64) + ((U(x1) * y0) >> 64) + (mid >> 64);
  const U r = (hi << 2) | (static_cast<uint64_t>(mid) >> 62);
  return neg ? -static_cast<__int128>(r) : static_cast<__int128>(r);
}

constexpr __int128 fx_i128(uint64_t hi, uint64_t lo) {
  return static_cast<__int128>((static_cast<unsigned __int128>(hi) << 64) | lo);
}

// Both tables by repeated rotation / multiplication in 126-bit fixed point
// (errors below 2^-112), rounded to 62 bits.
constexpr FxTables fx_make_tables() {
  FxTables t{};
  // cos and sin of 2 pi / 2048 and 2^(-1/2048), times 2^126
  const __int128 ch = fx_i128(0x3fffec42c43a03a5ull, 0x4c0c50df5fb32e78ull);
  const __int128 sh = fx_i128(0x003243f17d994974ull, 0x95d203de55ad91c2ull);
  const __int128 eh = fx_i128(0x3ffa74acbdf6c9d5ull, 0x777c74a28de290e3ull);
  __int128 c = __int128(1) << 126, s = 0, e = __int128(1) << 126;
  const __int128 half = __int128(1) << 63;
  for (int i = 0; i < kFxCosEntries; ++i) {
    if (i % 512 == 0) {  // the axes, exactly
      const int q = (i / 512) % 4;
      c = q == 0 ? __int128(1) << 126 : q == 2 ? -(__int128(1) << 126) : 0;
      s = q == 1 ? __int128(1) << 126 : q == 3 ? -(__int128(1) << 126) : 0;
    }
    t.c[i] = static_cast<int64_t>((c + half) >> 64) + kFxBias;
    const __int128 c2 = fx_mul126(c, ch) - fx_mul126(s, sh);
    s = fx_mul126(s, ch) + fx_mul126(c, sh);
    c = c2;
    if (i < kFxExpEntries) {
      t.e[i] = static_cast<int64_t>((e + half) >> 64) + kFxBias;
      e = fx_mul126(e, eh);
    }
  }
  return t;
}

ZMC_FX_TABLE FxTables kFxTables = fx_make_tables();

// -------------------------------------------------------------------- cos --
// 2^62 cos(2 pi (theta - 2^-12)) + 2^31, theta with half a table step added
// (fx_phase0).  With i the step nearest to the angle and d the rest in radians
// (|d| <= pi / 2048), c and n = -s from the table:
//   cos = c + d (n - d/2 (c - 2 d h)),  h = s c3 + c d / 24 as a 32-bit number,
// c3 = 1/6 less 0.87 max(d)^2 / 120, which leaves 2^-56.6 of the degree-5 term.
ZMC_FX int64_t fx_cos(uint64_t theta, const int64_t* table) {
  const int i = static_cast<int>(theta >> 53);
  const int64_t c = table[i], n = table[i + 512];
  // the remainder as a 64-bit signed fraction of half a step
  const uint64_t r = (theta << 11) ^ (uint64_t(1) << 63);
  // d 2^71 = r pi/4, both halves: t is below 2^32 with the bias that makes the
  // low half signed
  const int32_t kh = 0x6487ed51, kl = 0x10b4611a;
  const int32_t rh = static_cast<int32_t>(r >> 32);
  const uint32_t t = fx_umulhi(static_cast<uint32_t>(r), static_cast<uint32_t>(kh)) +
                     (static_cast<uint32_t>(fx_mulhi(rh, kl)) + 0x80000000u);
  const int64_t d = fx_wide(rh, kh) + static_cast<int64_t>(static_cast<uint64_t>(t));
  const int32_t dh = fx_top(d), dl = fx_low(d);  // d = dh 2^-39 + dl 2^-71
  const int32_t chi = fx_top(c), nhi = fx_top(n);
  // -h 2^31 (s = -n), then x = c - 2 d h, still biased
  const int32_t u = nhi - (fx_mulhi(dh, chi) >> 9);
  const int32_t h = fx_mulhi(u, 0x555554c3);
  const int64_t x = c + (fx_wide(dh, h) >> 7);
  // y = n - d x / 2, biased
  const int64_t y = n - (fx_mul(dh, dl, fx_top(x), fx_low(x), 1 + 128) >> 8);
  return c + (fx_mul(dh, dl, fx_top(y), fx_low(y), 1 + 64) >> 7);
}

// 2^62 a b for biased a, b (times 2^62, at most 2^62 in size), biased.
ZMC_FX int64_t fx_mul62(int64_t a, int64_t b) {
  const int64_t p = fx_mul(fx_top(a), fx_low(a), fx_top(b), fx_low(b), 1);
  return static_cast<int64_t>(static_cast<uint64_t>(p) << 2) + kFxBias;
}

// 2^SCALE g^2 for g = 2^62 g + 2^31, to about a unit (the cuts average out): 2^-60
// with two multiplies of high halves, 2^-62 with the low half's whole product.
template <int SCALE>
ZMC_FX int64_t fx_square(int64_t g) {
  static_assert(SCALE == 60 || SCALE == 62, "scale of the squares");
  const int32_t h = fx_top(g), l = fx_low(g);
  if constexpr (SCALE == 60) {
    return fx_wide(h, h) + (2 * fx_mulhi(h, l) + 1);
  } else {
    return 4 * fx_wide(h, h) + ((fx_wide(h, l) + (1 << 28)) >> 29);
  }
}

// -------------------------------------------------------------------- exp --
// The double 2^-q for q 2^54 = q - 2^42 (half a table step added by the
// caller), 0 <= q < 1000.  With i the nearest step of q's fraction and r ln 2
// the rest (|p| <= ln 2 / 4096): T (1 - p (1 - p (1/2 - p/6 + p^2/24))).
ZMC_FX double fx_exp2neg(uint64_t q, const int64_t* table) {
  const int n = static_cast<int>(q >> 54);
  const int i = static_cast<int>(q >> 43) & 2047;
  const int64_t tb = table[i];
  const uint64_t r = (q << 21) ^ (uint64_t(1) << 63);
  const int32_t kh = 0x58b90bfc, kl = static_cast<int32_t>(0xe8e7bcd6u);  // ln 2, 2^63
  const int32_t rh = static_cast<int32_t>(r >> 32);
  const uint32_t t = fx_umulhi(static_cast<uint32_t>(r), static_cast<uint32_t>(kh)) +
                     (static_cast<uint32_t>(fx_mulhi(rh, kl)) + 0x80000000u);
  const int64_t p = fx_wide(rh, kh) + static_cast<int64_t>(static_cast<uint64_t>(t));
  const int32_t ph = fx_top(p);  // p = ph 2^-42 + (low half) 2^-74
  const int32_t u = 349525 - fx_mulhi(ph, 85);            // 2^21 (1/6 - p/24)
  const int32_t h2 = (1 << 30) - fx_mulhi(ph, u);         // 2^31 (1/2 - p/6 + p^2/24)
  const int32_t k = static_cast<int32_t>(fx_wide(ph, h2) >> 29);  // 2^44 p h2
  const int64_t e = p - (fx_wide(ph, k) >> 12);           // 2^74 p (1 - p h2), biased
  const int64_t f =
      tb - kFxBias - (fx_mul(fx_top(tb), fx_low(tb), fx_top(e), fx_low(e), 1 + 512) >> 10);
  // f in (0.49, 1.01) 2^62 to a double: the leading bit to bit 63, rounded
  const uint64_t fu = static_cast<uint64_t>(f);
  const int z = fx_clz(static_cast<uint32_t>(fu >> 32));
  const uint64_t m = ((fu << z) >> 10) + 1;  // bit 53 leads
  return fx_bits_double((static_cast<uint64_t>(1023 - n - z) << 52) + (m >> 1));
}

// A biased product shifted up to the top of its range (62 bits), with its exponent,
// so that a long product of small factors keeps its precision.
ZMC_FX int64_t fx_normalise(int64_t g, int* exponent) {
  const int64_t m = g - kFxBias;
  const int32_t h = fx_top(m);
  const int c = fx_clz(static_cast<uint32_t>(h ^ (h >> 31)));
  const int z = c > 2 ? c - 2 : 0;
  *exponent -= z;
  return static_cast<int64_t>(static_cast<uint64_t>(m) << z) + kFxBias;
}

// The double nearest to g 2^(S - 62), |S| <= 900 (g of any sign, 0 included).
ZMC_FX double fx_to_double(int64_t g, int S) {
  const uint64_t sign = static_cast<uint64_t>(g) & (uint64_t(1) << 63);
  uint64_t m = static_cast<uint64_t>(g < 0 ? -g : g);
  const uint32_t h = static_cast<uint32_t>(m >> 32);
  const int z = h ? fx_clz(h) : 32 + fx_clz(static_cast<uint32_t>(m));
  if (z >= 64) return 0.0;
  m = ((m << z) >> 10) + 1;  // bit 53 leads
  return fx_bits_double(sign | ((static_cast<uint64_t>(1023 + S - z) << 52) + (m >> 1)));
}

// round(v 2^k) for |v 2^k| < 2^63.
ZMC_FX int64_t fx_fix(double v, int k) {
  const uint64_t u = fx_double_bits(v);
  const int ex = static_cast<int>((u >> 52) & 0x7ff);
  const uint64_t m = ex ? (u & 0xfffffffffffffull) | (uint64_t(1) << 52) : 0;
  const int s = 1075 - ex - k;  // right shift of m
  const uint64_t w = s <= 0 ? m << -s : s > 54 ? 0 : ((m >> (s - 1)) + 1) >> 1;
  return u >> 63 ? -static_cast<int64_t>(w) : static_cast<int64_t>(w);
}

// (c u) >> 32 for a 64-bit c with signed low half (ch, cl) and a signed 32-bit u.
ZMC_FX int64_t fx_mul32(int32_t ch, int32_t cl, int32_t u) {
  return fx_wide(ch, u) + fx_mulhi(cl, u);
}

// Twofold numbers hi + lo for the polynomial's constants.
struct FxTwo {
  double hi, lo;
};
ZMC_FX FxTwo fx_two_sum(double a, double b) {
  const double s = a + b, t = s - a;
  return {s, (a - (s - t)) + (b - t)};
}
ZMC_FX FxTwo fx_two_mul(FxTwo a, double b) {
  const double p = a.hi * b;
  return {p, fma(a.hi, b, -p) + a.lo * b};
}

// 1 + x y^2, y = a + w (2 v + 1) 2^-24, as c0 + u (c1 + u c2) in the centred field
// u = (v - 2^22) 2^-23, all over 2^s: 2^62 times, c0 and c1 with the bias.
struct FxPoly {
  int64_t c0, c1, c2;
  int s;
  bool ok;
};
ZMC_FX FxPoly fx_poly(double x, double a, double w) {
  const double k = 0.5 + 0x1p-24;
  const double wk = w * k;
  FxTwo m = fx_two_sum(a, wk);
  m.lo += fma(w, k, -wk);
  const FxTwo mw = fx_two_mul(m, w);
  FxTwo mm = fx_two_mul(m, m.hi);
  mm.lo += m.hi * m.lo;
  const FxTwo xmm = fx_two_mul(mm, x);
  FxTwo c0 = fx_two_sum(1.0, xmm.hi);
  c0.lo += xmm.lo;
  const FxTwo c1 = fx_two_mul(mw, 2.0 * x);
  const double ww = w * w;
  const FxTwo c2 = fx_two_mul({ww, fma(w, w, -ww)}, x);
  const double q0 = fabs(c0.hi), q1 = fabs(c1.hi), q2 = fabs(c2.hi);
  double b = q0 + 0.5 * q1 + 0.25 * q2;
  b = q1 + 0.5 * q2 > b ? q1 + 0.5 * q2 : b;
  b = q2 > b ? q2 : b;
  FxPoly r{0, 0, 0, 0, fx_below(b, 60) && fx_below(x, 200) && fx_below(a, 200) &&
                           fx_below(w, 200)};
  if (!r.ok) return r;
  // b < 2^s with room for the roundings
  r.s = static_cast<int>((fx_double_bits(b * (1.0 + 0x1p-20)) >> 52) & 0x7ff) - 1022;
  r.c0 = fx_fix(c0.hi, 62 - r.s) + fx_fix(c0.lo, 62 - r.s) + kFxBias;
  r.c1 = fx_fix(c1.hi, 62 - r.s) + fx_fix(c1.lo, 62 - r.s) + kFxBias;
  r.c2 = fx_fix(c2.hi, 62 - r.s) + fx_fix(c2.lo, 62 - r.s) + kFxBias;
  return r;
}

// Its value at field v, times 2^(62 - s), biased.
ZMC_FX int64_t fx_poly_eval(int64_t c0, int64_t c1, int64_t c2, uint32_t v) {
  const int32_t u = static_cast<int32_t>((v << 9) ^ 0x80000000u);  // u 2^32
  const int64_t t = c1 + fx_mul32(fx_top(c2), fx_low(c2), u);
  return c0 + fx_mul32(fx_top(t), fx_low(t), u);
}

// round(v K 2^(59 - 61)) for a constant K below 2^63 and |v K 2^-61| < 31.9
// (from 16 on only a v > 0, whose result is read as unsigned).
ZMC_FX int64_t fx_scale59(double v, uint64_t K) {
  const uint64_t u = fx_double_bits(v);
  const int ex = static_cast<int>((u >> 52) & 0x7ff);
  const uint64_t m = ex ? (u & 0xfffffffffffffull) | (uint64_t(1) << 52) : 0;
  // v K 2^-2 = (hi:lo) 2^(ex - 1077)
  const uint64_t hi = fx_umulhi64(m, K), lo = m * K;
  const int s = 1077 - ex;  // right shift of hi:lo, at least 45 here
  uint64_t w;
  if (s >= 118) {
    w = 0;
  } else if (s > 64) {
    w = ((hi >> (s - 65)) + 1) >> 1;
  } else if (s == 64) {
    w = hi + (lo >> 63);
  } else {
    w = ((hi << (64 - s)) | (lo >> s)) + ((lo >> (s - 1)) & 1);
  }
  return u >> 63 ? -static_cast<int64_t>(w) : static_cast<int64_t>(w);
}

// ------------------------------------------------------------------- sums --
// 128-bit sums of 64-bit terms (no term count reaches 2^64).
struct FxSum {
  uint32_t w0 = 0, w1 = 0, w2 = 0, w3 = 0;
  ZMC_FX void add(int64_t v) {
#if defined(__CUDA_ARCH__)
    const uint32_t lo = static_cast<uint32_t>(v), hi = static_cast<uint32_t>(v >> 32);
    const uint32_t sg = static_cast<uint32_t>(static_cast<int32_t>(hi) >> 31);
    asm("add.cc.u32 %0, %0, %4;\n\taddc.cc.u32 %1, %1, %5;\n\t"
        "addc.cc.u32 %2, %2, %6;\n\taddc.u32 %3, %3, %6;"
        : "+r"(w0), "+r"(w1), "+r"(w2), "+r"(w3) : "r"(lo), "r"(hi), "r"(sg));
#else
    unsigned __int128 s = (static_cast<unsigned __int128>(hi64()) << 64) | lo64();
    s += static_cast<unsigned __int128>(static_cast<__int128>(v));
    set(static_cast<uint64_t>(s >> 64), static_cast<uint64_t>(s));
#endif
  }
  ZMC_FX uint64_t lo64() const { return (static_cast<uint64_t>(w1) << 32) | w0; }
  ZMC_FX uint64_t hi64() const { return (static_cast<uint64_t>(w3) << 32) | w2; }
  ZMC_FX void set(uint64_t hi, uint64_t lo) {
    w0 = static_cast<uint32_t>(lo);
    w1 = static_cast<uint32_t>(lo >> 32);
    w2 = static_cast<uint32_t>(hi);
    w3 = static_cast<uint32_t>(hi >> 32);
  }
  // Less n * 2^31 (the bias of n terms), as a double times 2^-scale.
  ZMC_FX double value(uint64_t n, int scale) const {
    uint64_t lo = lo64(), hi = hi64();
    const uint64_t blo = n << 31, bhi = n >> 33;
    hi -= bhi + (lo < blo ? 1 : 0);
    lo -= blo;
    const bool neg = (hi >> 63) != 0;
    if (neg) {
      lo = ~lo + 1;
      hi = ~hi + (lo == 0 ? 1 : 0);
    }
    // nearest double of hi:lo, by its 64 leading bits with a sticky bit
    double v;
    if (hi == 0) {
      v = static_cast<double>(lo);
    } else {
      const uint32_t h32 = static_cast<uint32_t>(hi >> 32);
      const int z = h32 ? fx_clz(h32) : 32 + fx_clz(static_cast<uint32_t>(hi));
      const uint64_t top = z ? (hi << z) | (lo >> (64 - z)) : hi;
      const uint64_t rest = z ? lo << z : lo;
      v = static_cast<double>(top | (rest ? 1 : 0));
      scale -= 64 - z;
    }
    v *= fx_bits_double(static_cast<uint64_t>(1023 - scale) << 52);
    return neg ? -v : v;
  }
};

}  // namespace zmc
