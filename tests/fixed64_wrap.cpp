// C wrappers around csrc/zmc_fixed64.cuh, built with the host compiler by
// test_fixed64_cpu.py.
#include <cmath>
#include <vector>
using std::fabs;
using std::fma;
#include "zmc_fixed64.cuh"

using namespace zmc;

extern "C" {
const int64_t* fx_cos_table() { return kFxTables.c; }
const int64_t* fx_exp_table() { return kFxTables.e; }
void fx_cos_n(const uint64_t* th, int64_t* out, int n) {
  for (int i = 0; i < n; ++i) out[i] = fx_cos(th[i], kFxTables.c) - kFxBias;
}
void fx_exp_n(const uint64_t* q, double* out, int n) {
  for (int i = 0; i < n; ++i) out[i] = fx_exp2neg(q[i], kFxTables.e);
}
void fx_mul62_n(const int64_t* a, const int64_t* b, int64_t* out, int n) {
  for (int i = 0; i < n; ++i) out[i] = fx_mul62(a[i] + kFxBias, b[i] + kFxBias) - kFxBias;
}
void fx_turns_n(const double* c, const int* k, uint32_t* out, int n) {
  for (int i = 0; i < n; ++i) {
    const FxTurns t = fx_turns(c[i], k[i]);
    out[3 * i] = t.w0;
    out[3 * i + 1] = t.w1;
    out[3 * i + 2] = t.w2;
  }
}
uint64_t fx_phase(uint64_t th, uint32_t v, const uint32_t* b) {
  return fx_phase_step(th, v, b[0], b[1], b[2]);
}
int64_t fx_scale(double v, uint64_t K) { return fx_scale59(v, K); }
// prod_k (1 + x_k y_k^2) at n rows of d fields; returns whether it is in range
int fx_poly_n(const double* x, double a, double w, const uint32_t* v, double* out, int d, int n) {
  FxPoly p[8];
  int scale = 0;
  for (int k = 0; k < d; ++k) {
    p[k] = fx_poly(x[k], a, w);
    if (!p[k].ok) return 0;
    scale += p[k].s;
  }
  for (int i = 0; i < n; ++i) {
    int e = scale;
    int64_t g = 0;
    for (int k = 0; k < d; ++k) {
      if (k > 1 && k % 2 == 0) g = fx_normalise(g, &e);
      const int64_t f = fx_poly_eval(p[k].c0, p[k].c1, p[k].c2, v[i * d + k]);
      g = k ? fx_mul62(g, f) : f;
    }
    out[i] = fx_to_double(g - kFxBias, e);
  }
  return 1;
}
double fx_sum(const int64_t* g, int n, int scale) {
  FxSum s;
  for (int i = 0; i < n; ++i) s.add(g[i] + kFxBias);
  return s.value(static_cast<uint64_t>(n), scale);
}
void fx_square_60(const int64_t* g, int64_t* out, int n) {
  for (int i = 0; i < n; ++i) out[i] = fx_square<60>(g[i] + kFxBias);
}
void fx_square_62(const int64_t* g, int64_t* out, int n) {
  for (int i = 0; i < n; ++i) out[i] = fx_square<62>(g[i] + kFxBias);
}
// The mean of cos^2 of prod_k cos(x_k y_k)'s factors, multiplied, and the least of them;
// at n rows of d fields 2^62 g and its square as the FP64 kernel adds them.
void fx_cosprod_n(const double* x, double a, double w, const uint32_t* v, int d, int n,
                  float* mean2, float* least, int64_t* g, int64_t* sq) {
  std::vector<FxTurns> b(d);
  std::vector<uint64_t> c(d);
  *mean2 = *least = 1.0f;
  for (int k = 0; k < d; ++k) {
    b[k] = fx_turns_mul(x[k], w, -23);
    const FxTurns xa = fx_turns_mul(x[k], a, 0);
    c[k] = fx_phase0(fx_turns_add(xa, fx_turns_sar(b[k], 1)));
    const uint32_t xw = fx_lead23(b[k]);
    const float m = fx_mean_cos2(2 * xa.w2 + xw, fx_sinc(static_cast<float>(x[k] * w), xw));
    *mean2 *= m;
    *least = m < *least ? m : *least;
  }
  for (int i = 0; i < n; ++i) {
    int64_t p = 0;
    for (int k = 0; k < d; ++k) {
      const int64_t f =
          fx_cos(fx_phase_step(c[k], v[i * d + k], b[k].w0, b[k].w1, b[k].w2), kFxTables.c);
      p = k ? fx_mul62(p, f) : f;
    }
    g[i] = p - kFxBias;
    sq[i] = d <= 3 ? fx_square<60>(p) : fx_square<62>(p);
  }
}
// The same of sin(sum_k y_k + xsum), y_k from a_k on, w_k wide.
void fx_sinsum_n(double xsum, const double* a, const double* w, const uint32_t* v, int d, int n,
                 float* mean2, int64_t* g, int64_t* sq) {
  std::vector<FxTurns> b(d);
  FxTurns t = fx_turns_add(fx_turns(xsum, 0), {0, 0, 0xC0000000u});
  uint32_t widths = 0;
  float sincs = 1.0f;
  for (int k = 0; k < d; ++k) {
    b[k] = fx_turns(w[k], -23);
    t = fx_turns_add(t, fx_turns_add(fx_turns(a[k], 0), fx_turns_sar(b[k], 1)));
    widths += fx_lead23(b[k]);
    sincs *= fx_sinc(static_cast<float>(w[k]), fx_lead23(b[k]));
  }
  *mean2 = fx_mean_cos2(2 * t.w2 + widths, sincs);
  for (int i = 0; i < n; ++i) {
    uint64_t th = fx_phase0(t);
    for (int k = 0; k < d; ++k)
      th = fx_phase_step(th, v[i * d + k], b[k].w0, b[k].w1, b[k].w2);
    const int64_t p = fx_cos(th, kFxTables.c);
    g[i] = p - kFxBias;
    sq[i] = fx_square<60>(p);
  }
}
void fx_quad(float x, float q, float a, float w, float* out) {
  const FxReach r = fx_quad_reach(x, q, a, w);
  out[0] = r.width;
  out[1] = r.drop;
}
int fx_range(uint32_t lead, float width) { return fx_cos_range(lead, width); }
}
