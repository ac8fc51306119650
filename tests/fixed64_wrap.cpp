// C wrappers around csrc/zmc_fixed64.cuh, built with the host compiler by
// test_fixed64_cpu.py.
#include <cmath>
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
}
