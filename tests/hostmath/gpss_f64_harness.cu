// Host build of further parts of the CUDA path's device arithmetic, for CPU
// tests.  Compiled by tests/test_host_f64.py with nvcc into a shared library.
#include "gpss_kernels.cuh"
#include "gpss_prod.cuh"

using namespace gpss;

extern "C" {

// out2: an event's share of the sums (prod_tally)
void hf_prod_tally(double S, double dS, double e, double de, double *out2) {
  out2[0] = out2[1] = 0.0;
  prod_tally(S, dS, e, de, 1.0f / (float)S, out2[0], out2[1]);
}

// The plain FP64 filter's step scalars (f, f', F1, I_ff, I_pp, I_FF).
void hf_plain64_scalars(double t, double a, double beta, double *out6) {
  TermC<double> c;
  c.a = a;
  c.beta = beta;
  c.w2 = beta + a * a;
  c.qc = c.var = 1.0;
  finish_termc(c);
  double cs[TAB64_N + 2], tab[TAB64_LEN];
  const double T = taylor64_unit(c.r2);
  tab[6 * TAB64_N] = 1.0 / T;
  taylor64_c(c.a * T, c.w2 * T * T, cs);
  for (int e = 0; e < 6 * TAB64_N; ++e) tab[e] = taylor64_entry(cs, e / TAB64_N, e % TAB64_N);
  const Disc<double> d = discretize_tab64(t, c, tab);
  const double v[6] = {d.f, d.fp, d.F1, d.Iff, d.Ipp, d.IFF};
  for (int i = 0; i < 6; ++i) out6[i] = v[i];
}

// A product oscillator's step scalars (f, f', I_ff, I_pp) and their tangent
// with respect to omega0 (which = 0) or Q (1), from the records that the
// kernels keep per step.
void hf_prod_dual(float dt, float w0, float Q, int which, double *out8) {
  using T = Dual2<float>;
  T a, beta;
  osc_rates<T, float>(mk(w0, which == 0 ? 1.f : 0.f, 0.f), mk(Q, which == 1 ? 1.f : 0.f, 0.f), a,
                      beta);
  const Disc<float> d = discretize<float, float, true>(dt, a.v, beta.v);
  float4 ta, tb;
  prod_tangents(dt, a.v, beta.v, prod_unit(w0), ta, tb);
  const Disc<T> e = prod_dual(make_float4(d.f, d.fp, d.Iff, d.Ipp), ta, tb,
                              prod_rates_tangent(a, beta, w0));
  const T v[4] = {e.f, e.fp, e.Iff, e.Ipp};
  for (int i = 0; i < 4; ++i) {
    out8[i] = v[i].v;
    out8[4 + i] = v[i].da;
  }
}

}  // extern "C"
