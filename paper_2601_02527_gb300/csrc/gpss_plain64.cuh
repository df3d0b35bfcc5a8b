// The plain FP64 filter (log-likelihood only): the sequential recursion of
// Eqs. integrated_kalman_pred / integrated_kalman_update / kalman_update, one
// block of two warps per output row.
//
// What bounds it: this GPU's FP64 pipe takes one lane per clock and SM
// sub-partition, so an FP64 instruction occupies it for 32 clocks however many
// of its lanes do useful work.  One thread per series therefore left 31 of 32
// slots idle where series are few, and ran the step's discretisation (about
// 1600 of its FP64 instructions for two terms) inside the serial chain.  Here
//  * warp 1 discretises 32 events at a time, one event per lane, into a record
//    in shared memory (two buffers: the next 32 while warp 0 filters), and
//    sums log S and v^2/S of the events filtered before, one event per lane;
//  * warp 0 runs the recursion with one covariance entry per lane.  Predict is
//    two products with the sparse Phi~ (T = [P; m] Phi~^T, then Phi~ T + Q~),
//    at most 2 NT + 1 terms per entry each;
//  * the Taylor branch of the step scalars is a Horner evaluation of per-row
//    coefficients (same truncation as disc_taylor<double>), 114 FMAs instead
//    of the double sums' 1000.
// 150 series of 300 to 2500 exposures, SHO + Matern-3/2: 253.4 ms with one
// thread per series, 4.45 ms here (0.89 us per event of the longest series).
// The recursion stays sequential in time: its error against extended
// arithmetic is that of the textbook filter for any parameters.
#pragma once

#include "gpss_device.cuh"

namespace gpss {

// Taylor coefficients per scalar: those with n + m <= TaylorOrder<double>::N + 1
constexpr int TAB64_N = TaylorOrder<double>::N;

// Table entry k of scalar j (definitions at the step-scalar tables) from f's
// Taylor coefficients c[0..TAB64_N+1].
GPSS_HD double taylor64_entry(const double *c, int j, int k) {
  if (j == 0) return c[k + 1];
  if (j == 1) return c[k + 1] * (double)(k + 1);
  if (j == 2) return c[k + 1] / (double)(k + 2);
  double s = 0.0;
  for (int n = 1; n <= k + 1; ++n) {
    const int m = k + 2 - n;
    if (n > TAB64_N || m > TAB64_N) continue;
    const double pp = c[n] * c[m];
    s += j == 3 ? pp : j == 4 ? pp * (double)(n * m) : pp / (double)((n + 1) * (m + 1));
  }
  return s / (double)(j == 3 ? k + 3 : j == 4 ? k + 1 : k + 5);
}

// The unit of time T of a row's coefficients: a power of two within a factor of
// two of 1/r.  In the caller's unit the last of them is of the size r^20 / 21!,
// which leaves FP64's range for rates beyond about 1e17 or 1e-17; in this one
// every entry is of order one at most.  Scaling by it is exact.
GPSS_HD double taylor64_unit(double r2) {
  return r2 > 0.0 && isfinite(r2) ? ldexp(1.0, -(ilogb(r2) >> 1)) : 1.0;
}

// f's Taylor coefficients by its recurrence, from a T and w2 T^2.
GPSS_HD void taylor64_c(double a, double w2, double *c) {
  c[0] = 0.0;
  c[1] = 1.0;
  c[2] = -a;
  for (int n = 1; n + 2 <= TAB64_N + 1; ++n)
    c[n + 2] = -(2.0 * a * (n + 1) * c[n + 1] + w2 * c[n]) / (double)((n + 2) * (n + 1));
}

// A row's table: the entries of the six scalars, then 1/T.
constexpr int TAB64_LEN = 6 * TAB64_N + 1;

GPSS_HD Disc<double> disc_tab64(double t, const double *tab) {
  double g[6];
  const double u = t * tab[6 * TAB64_N];
#pragma unroll
  for (int j = 0; j < 6; ++j) g[j] = tab[j * TAB64_N + TAB64_N - 1];
  for (int k = TAB64_N - 2; k >= 0; --k)
#pragma unroll
    for (int j = 0; j < 6; ++j) g[j] = fma(g[j], u, tab[j * TAB64_N + k]);
  const double t2 = t * t, t3 = t2 * t;
  return Disc<double>{g[0] * t, g[1], g[2] * t2, g[3] * t3, g[4] * t, g[5] * (t3 * t2)};
}

// The step's scalars, branches as discretize<double, double, true>.
GPSS_HD Disc<double> discretize_tab64(double t, const TermC<double> &c, const double *tab) {
  if (t == 0.0) return Disc<double>{0.0, 1.0, 0.0, 0.0, 0.0, 0.0};
  constexpr double xt2 = TaylorOrder<double>::XT2;
  if (c.r2 * t * t <= xt2) return disc_tab64(t, tab);
  double f, fp;
  if (c.beta < 0.0) {
    const double l1 = c.w2 / sqrt(c.r2);
    if (l1 * t * l1 * t < xt2) {
      double h;
      const int k = halvings<double>(t, c.r2, xt2, h);
      Disc<double> d = disc_tab64(h, tab);
      for (int i = 0; i < k; ++i) {
        disc_double_integrals<double, double>(d, c.a, c.w2);
        h *= 2.0;
        od_f_fp<double, double>(h, c.a, c.beta, c.b, c.w2, d.f, d.fp);
      }
      return d;
    }
    od_f_fp<double, double>(t, c.a, c.beta, c.b, c.w2, f, fp);
  } else {
    const double E = exp(-c.a * t), tau = c.b * t;
    double s, co;
    sincos(tau, &s, &co);
    const double S = tau < 1e-6 ? t * (1.0 - tau * tau * (1.0 / 6.0)) : s * c.rb;
    f = E * S;
    fp = E * (co - c.a * S);
  }
  return disc_closed_ffp<double, double>(t, c.a, c.w2, c.rw2, c.r4a, f, fp);
}

// An event's record in shared memory: per term the twelve Blocks values, then
// 0, 1, y, yerr^2, 1/delta.  The length is odd: lanes writing one field of
// consecutive records meet no bank conflict.
template <class S>
struct Rec64 {
  static constexpr int ZERO = 12 * S::NT, ONE = ZERO + 1, Y = ZERO + 2, R0 = ZERO + 3,
                       W = ZERO + 4, LEN = ZERO + 5;
  // nonzeros of a row of Phi~: a term's pair, or for an integral state the
  // pairs of its terms and itself
  static constexpr int NZ = S::NS == 0 ? 2 : 1 + 2 * (S::LAYOUT == 0 ? S::NT : 1);
};

// Row i of Phi~: the s-th nonzero's column and its place in the record.
template <class S>
GPSS_HD void phi_entry(int i, int s, int &col, int &off) {
  using R = Rec64<S>;
  col = 0;
  off = R::ZERO;
  if (i < 2 * S::NT) {
    if (s < 2) {
      col = (i & ~1) + s;
      off = 12 * (i >> 1) + 2 * (i & 1) + s;
    }
    return;
  }
  if (s == R::NZ - 1) {
    col = i;
    off = R::ONE;
    return;
  }
  const int t = S::LAYOUT == 0 ? s / 2 : (i - 2 * S::NT) % S::NT;
  col = 2 * t + (s & 1);
  off = 12 * t + 4 + (s & 1);
}

// Q~[i][j] (i <= j): the places of its (up to NT) terms in the record.
template <class S>
GPSS_HD int q_entry(int i, int j, int t) {
  constexpr int X = 2 * S::NT, ZERO = Rec64<S>::ZERO;
  const bool z_t = j >= X && (S::LAYOUT == 0 || (j - X) % S::NT == t);
  if (j < X) return (i >> 1) == t && (j >> 1) == t ? 12 * t + 6 + (i & 1) + (j & 1) : ZERO;
  if (!z_t) return ZERO;
  if (i < X) return (i >> 1) == t ? 12 * t + 9 + (i & 1) : ZERO;
  return S::LAYOUT == 0 || (i - X) % S::NT == t ? 12 * t + 11 : ZERO;
}

template <class S>
__global__ void __launch_bounds__(64) k_plain64(DevModel M, const float *__restrict__ theta,
                                                int per_series, double *__restrict__ ll_out,
                                                int *__restrict__ err) {
  using R = Rec64<S>;
  constexpr int D = S::D, NT = S::NT, NZ = R::NZ, X = 2 * NT;
  constexpr int NE = (D + 1) * D;        // entries of [P; m]
  constexpr int NR = (NE + 31) / 32;     // ... per lane
  __shared__ double rec[2][32][R::LEN];
  __shared__ double Sb[2][32], vb[2][32];
  __shared__ uint8_t tg[2][32];
  __shared__ double tab[NT][TAB64_LEN];
  __shared__ double cs[NT][TAB64_N + 2];
  __shared__ double Pm[NE], T[NE];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int v = blockIdx.x;
  const int s = per_series ? v : v % M.n_series;
  const int row = per_series ? v : v / M.n_series;
  TermC<double> tc[NT];
  double s2;
  load_terms<NT, double>(theta + (size_t)row * M.n_params, M.kinds, tc, s2);
  if (threadIdx.x < NT) {
#pragma unroll
    for (int t = 0; t < NT; ++t)
      if (t == (int)threadIdx.x) {
        const double unit = taylor64_unit(tc[t].r2);
        tab[t][6 * TAB64_N] = 1.0 / unit;
        taylor64_c(tc[t].a * unit, tc[t].w2 * unit * unit, cs[t]);
      }
  }
  if (threadIdx.x == 0) {
    // P0 = blkdiag(P_inf, I), m0 = 0
    for (int i = 0; i < NE; ++i) Pm[i] = 0.0;
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      Pm[2 * t * (D + 1)] = tc[t].var;
      Pm[(2 * t + 1) * (D + 1)] = tc[t].var * tc[t].w2;
    }
    for (int z = X; z < D; ++z) Pm[z * (D + 1)] = 1.0;
  }
  rec[warp][lane][R::ZERO] = 0.0;
  rec[warp][lane][R::ONE] = 1.0;
  __syncthreads();
  for (int i = threadIdx.x; i < NT * 6 * TAB64_N; i += 64) {
    const int t = i / (6 * TAB64_N), e = i % (6 * TAB64_N);
    tab[t][e] = taylor64_entry(cs[t], e / TAB64_N, e % TAB64_N);
  }
  __syncthreads();

  const int64_t e0 = M.ev_off[s], n_ev = M.ev_off[s + 1] - e0;
  const int64_t n_batch = (n_ev + 31) / 32;
  int64_t mi = M.meas_off[s];  // warp 1: first measurement of the next batch
  double sum_logS = 0.0, sum_q = 0.0;
  bool bad = false;

  auto produce = [&](int64_t b) {
    const int buf = (int)(b & 1);
    const int64_t k = b * 32 + lane;
    const bool in = k < n_ev;
    const uint8_t tag = in ? M.tag[e0 + k] : 0;
    const unsigned ends = __ballot_sync(0xffffffffu, tag & 1);
    if (in) {
      double *r = rec[buf][lane];
      const double dt = M.dt64[e0 + k];
#pragma unroll
      for (int t = 0; t < NT; ++t) {
        const Blocks<double> B = make_blocks(discretize_tab64(dt, tc[t], tab[t]), tc[t]);
        double *q = r + 12 * t;
        q[0] = B.p00; q[1] = B.p01; q[2] = B.p10; q[3] = B.p11; q[4] = B.pb0; q[5] = B.pb1;
        q[6] = B.q00; q[7] = B.q01; q[8] = B.q11; q[9] = B.qz0; q[10] = B.qz1; q[11] = B.qzz;
      }
      tg[buf][lane] = tag;
      if (tag & 1) {
        const int64_t i = mi + __popc(ends & ((1u << lane) - 1));
        r[R::Y] = M.meas64[3 * i];
        r[R::R0] = M.meas64[3 * i + 1];
        r[R::W] = M.meas64[3 * i + 2];
      }
    }
    mi += __popc(ends);
  };
  // S = 1, v = 0 stand for an event without a measurement (they add nothing)
  auto tally = [&](int64_t b) {
    if (b * 32 + lane >= n_ev) return;
    const double Sv = Sb[b & 1][lane], vv = vb[b & 1][lane];
    bad |= !(Sv > 0.0);
    sum_logS += log(Sv);
    sum_q += vv * vv / Sv;
  };

  // warp 0: this lane's entries of T (k, j) and of the packed P (i2, j2)
  int tcol[NR][NZ], toff[NR][NZ], tk[NR];
  int pcol[NZ], poff[NZ], qoff[NT], i2 = 0, j2 = lane;
#pragma unroll
  for (int q = 0; q < NR; ++q) {
    const int e = min(lane + 32 * q, NE - 1);
    tk[q] = (e / D) * D;
#pragma unroll
    for (int z = 0; z < NZ; ++z) phi_entry<S>(e % D, z, tcol[q][z], toff[q][z]);
  }
  while (i2 < D - 1 && j2 >= D - i2) {  // lane -> (i2, j2 - i2) of the upper triangle
    j2 -= D - i2;
    ++i2;
  }
  const bool has_p = lane < S::NP;
  j2 = min(i2 + j2, D - 1);
#pragma unroll
  for (int z = 0; z < NZ; ++z) phi_entry<S>(i2, z, pcol[z], poff[z]);
#pragma unroll
  for (int t = 0; t < NT; ++t) qoff[t] = q_entry<S>(i2, j2, t);
  const int l = min(lane, D - 1);

  auto consume = [&](int64_t b) {
    const int buf = (int)(b & 1);
    const int cnt = (int)(n_ev - b * 32 < 32 ? n_ev - b * 32 : 32);
    for (int kk = 0; kk < cnt; ++kk) {
      const double *r = rec[buf][kk];
      const uint8_t tag = tg[buf][kk];
#pragma unroll
      for (int q = 0; q < NR; ++q) {
        double acc = r[toff[q][0]] * Pm[tk[q] + tcol[q][0]];
#pragma unroll
        for (int z = 1; z < NZ; ++z)
          if (toff[q][z] != R::ZERO) acc = fma(r[toff[q][z]], Pm[tk[q] + tcol[q][z]], acc);
        if (lane + 32 * q < NE) T[lane + 32 * q] = acc;
      }
      __syncwarp();
      double p = r[qoff[0]];
#pragma unroll
      for (int t = 1; t < NT; ++t) p += r[qoff[t]];
#pragma unroll
      for (int z = 0; z < NZ; ++z)
        if (poff[z] != R::ZERO) p = fma(r[poff[z]], T[pcol[z] * D + j2], p);
      double m = T[D * D + l];
      const int slot = (tag >> 1) & 7;
      if (!(tag & 1)) {
        if constexpr (S::NS > 0) {
          if (S::zslot(j2) == slot && j2 >= X) p = 0.0;
          if (S::zslot(i2) == slot && i2 >= X) p = 0.0;
          if (S::zslot(l) == slot && l >= X) m = 0.0;
        }
        if (has_p) Pm[i2 * D + j2] = Pm[j2 * D + i2] = p;
        if (lane < D) Pm[D * D + lane] = m;
        if (lane == 0) {
          Sb[buf][kk] = 1.0;
          vb[buf][kk] = 0.0;
        }
        __syncwarp();
        continue;
      }
      if (has_p) Pm[i2 * D + j2] = Pm[j2 * D + i2] = p;
      if (lane < D) Pm[D * D + lane] = m;
      __syncwarp();
      // h selects columns c0 (and c1): the slot's integral states, or the latent
      const bool inst = S::NS == 0 || (tag & TAG_INSTANT);
      const int nz = S::LAYOUT == 0 ? 1 : NT;
      const int c0 = inst ? 0 : X + slot * nz;
      const int c1 = inst ? (NT > 1 ? 2 : -1) : (nz > 1 ? c0 + 1 : -1);
      const double w = inst ? 1.0 : r[R::W];
      auto col = [&](int i) {
        const double x = Pm[i * D + c0];
        return c1 < 0 ? x : x + Pm[i * D + c1];
      };
      const double ui = col(i2) * w, uj = col(j2) * w, ul = col(l) * w;
      const double hu = (c1 < 0 ? col(c0) : col(c0) + col(c1)) * w * w, hm = col(D) * w;
      const double Sv = hu + r[R::R0] + s2;
      const double vv = r[R::Y] - hm;
      const double iS = 1.0 / Sv;
      p -= ui * uj * iS;
      m += ul * (vv * iS);
      __syncwarp();
      if (has_p) Pm[i2 * D + j2] = Pm[j2 * D + i2] = p;
      if (lane < D) Pm[D * D + lane] = m;
      if (lane == 0) {
        Sb[buf][kk] = Sv;
        vb[buf][kk] = vv;
      }
      __syncwarp();
    }
  };

  if (warp == 1 && n_batch > 0) produce(0);
  __syncthreads();
  for (int64_t b = 0; b < n_batch; ++b) {
    if (warp == 0) {
      consume(b);
    } else {
      if (b > 0) tally(b - 1);
      if (b + 1 < n_batch) produce(b + 1);
    }
    __syncthreads();
  }
  if (warp == 0) return;
  if (n_batch > 0) tally(n_batch - 1);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    sum_logS += __shfl_down_sync(0xffffffffu, sum_logS, o);
    sum_q += __shfl_down_sync(0xffffffffu, sum_q, o);
  }
  bad = __any_sync(0xffffffffu, bad);
  if (lane == 0) {
    const double n_end = (double)(M.meas_off[s + 1] - M.meas_off[s]);
    const double ll = -0.5 * (n_end * LOG_2PI + sum_logS + sum_q);
    ll_out[v] = ll;
    if (bad || !isfinite(ll)) flag_error(err, v, 7);
  }
}

template <class S>
cudaError_t launch_plain64(const DevModel &M, const float *theta, int n_out, int per_series,
                           double *ll, int *err, cudaStream_t st) {
  if (n_out <= 0) return cudaSuccess;
  k_plain64<S><<<n_out, 64, 0, st>>>(M, theta, per_series, ll, err);
  GPSS_COUNT_LAUNCH();
  return cudaGetLastError();
}

}  // namespace gpss
