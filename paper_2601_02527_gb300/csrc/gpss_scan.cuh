// Parallel-in-time combination of chunk elements (Section 3.2.5 of
// arXiv 2601.02527; operator of Sarkka & Garcia-Fernandez 2021).
//
// An element E = (A, b, C, eta, J) describes one stretch of events: given the
// state x entering it, the filtered state leaving it is N(A x + b, C), and
// the stretch's data carry information (eta, J) about x.  Combining E_i
// (earlier) with E_j (later), with X = I + C_i J_j:
//   Y = X^{-1} A_i,  W = X^{-1} C_i,  w = X^{-1} (b_i + C_i eta_j)
//   A = A_j Y,  b = A_j w + b_j,  C = A_j W A_j^T + C_j,
//   eta = Y^T (eta_j - J_j b_i) + eta_i,  J = Y^T J_j A_i + J_i,
// which is the SG21 operator written with one factorisation of X (the
// (I + J_j C_i)^{-1} there equals X^{-T}).  The identity element is
// (I, 0, 0, 0, 0).  The first chunk of every series has A = 0 and
// eta = J = 0, so one unsegmented scan over all chunks of all series restarts
// at every series boundary in both directions.
//
// Scan structure (no inter-block waiting): for n elements and tiles of T,
//   1. k_tile_reduce   one block per tile folds its T elements (tree);
//   2. the tile totals are scanned recursively by the same three steps;
//   3. k_tile_scan     one block per tile: Blelloch exclusive scan in shared
//                      memory, then prefix-of-tile o exclusive o own element.
// rev = 1 runs the mirrored scan (suffixes), whose operator is the same
// combine with its arguments in time order.
#pragma once

#include "gpss_device.cuh"

namespace gpss {

template <class S>
struct Elem {
  static constexpr int D = S::D;
  static constexpr int NP = S::NP;
  static constexpr int A = 0;
  static constexpr int B = D * D;
  static constexpr int C = B + D;
  static constexpr int ETA = C + NP;
  static constexpr int J = ETA + D;
  static constexpr int NF = J + NP;
  // fields in shared memory where 16 lanes combine, padded to an odd count so
  // that the two groups of a warp read different banks
  static constexpr int ST = NF | 1;
};

// Element accessor over a strided field-major buffer of T (float, or double
// for the FP64 combination of chunk elements).
template <class T>
struct EViewT {
  T *p;
  int stride;
  GPSS_HD T &operator[](int f) const { return p[(size_t)f * stride]; }
};
using EView = EViewT<float>;

template <class S, class T>
GPSS_HD void set_identity(EViewT<T> e) {
  using L = Elem<S>;
#pragma unroll
  for (int f = 0; f < L::NF; ++f) e[f] = T(0);
#pragma unroll
  for (int i = 0; i < S::D; ++i) e[L::A + i * S::D + i] = T(1);
}

template <class S, class T>
GPSS_HD void copy_elem(EViewT<T> dst, EViewT<T> src) {
#pragma unroll 8
  for (int f = 0; f < Elem<S>::NF; ++f) dst[f] = src[f];
}

// out <- Ei o Ej (Ei earlier), in the arithmetic of T.  out may alias Ej (the
// operands are read into registers field by field before out is written, see
// ordering below).
//
// With WITH_C, field NF of each element is its log-normaliser c: the data of
// the stretch have likelihood exp(c + eta^T x - x^T J x / 2) as a function of
// the state x entering it (c = -(sum log S + gamma + n log 2 pi) / 2 for a
// chunk).  Integrating x' ~ N(A_i x + b_i, C_i) against the later stretch's
// likelihood gives
//   c = c_i + c_j - log det X / 2 + eta_j^T b_i - b_i^T J_j b_i / 2
//       + u^T X^{-1} C_i u / 2,   u = eta_j - J_j b_i,
// so for a series that starts from the prior (A = 0) the combination of all
// its stretches carries the series' log-likelihood in c.
template <class S, class T, bool WITH_C = false>
GPSS_HD void combine(EViewT<T> Ei, EViewT<T> Ej, EViewT<T> out) {
  using L = Elem<S>;
  constexpr int D = S::D;
  // X = I + C_i J_j ; right-hand sides [A_i | C_i | b_i + C_i eta_j]
  T X[D][D], R[D][2 * D + 1];
#pragma unroll
  for (int r = 0; r < D; ++r) {
    T ce = T(0);
#pragma unroll
    for (int k = 0; k < D; ++k) ce += Ei[L::C + S::pk(r, k)] * Ej[L::ETA + k];
    R[r][2 * D] = Ei[L::B + r] + ce;
#pragma unroll
    for (int c = 0; c < D; ++c) {
      T acc = (r == c) ? T(1) : T(0);
#pragma unroll
      for (int k = 0; k < D; ++k) acc += Ei[L::C + S::pk(r, k)] * Ej[L::J + S::pk(k, c)];
      X[r][c] = acc;
      R[r][c] = Ei[L::A + r * D + c];
      R[r][D + c] = Ei[L::C + S::pk(r, c)];
    }
  }
  const T logdet_x = solve_inplace<D, 2 * D + 1, T>(X, R);
  // R = [Y | W | w].  New (eta, J) first: they need b_i, A_i, J_j, eta_j.
  T u[D], eta_n[D];
  T c_n = T(0);
#pragma unroll
  for (int r = 0; r < D; ++r) {
    T jb = T(0);
#pragma unroll
    for (int k = 0; k < D; ++k) jb += Ej[L::J + S::pk(r, k)] * Ei[L::B + k];
    u[r] = Ej[L::ETA + r] - jb;
  }
  if constexpr (WITH_C) {
    T q = T(0);
#pragma unroll
    for (int r = 0; r < D; ++r) {
      const T bi = Ei[L::B + r];
      T wu = T(0), jb = T(0);
#pragma unroll
      for (int k = 0; k < D; ++k) {
        wu += R[r][D + k] * u[k];
        jb += Ej[L::J + S::pk(r, k)] * Ei[L::B + k];
      }
      q += Ej[L::ETA + r] * bi - T(0.5) * bi * jb + T(0.5) * u[r] * wu;
    }
    c_n = Ei[L::NF] + Ej[L::NF] - T(0.5) * logdet_x + q;
  }
#pragma unroll
  for (int r = 0; r < D; ++r) {
    T acc = Ei[L::ETA + r];
#pragma unroll
    for (int k = 0; k < D; ++k) acc += R[k][r] * u[k];
    eta_n[r] = acc;
  }
  // T = J_j A_i ; J = Y^T T + J_i
  T TT[D][D];
#pragma unroll
  for (int r = 0; r < D; ++r)
#pragma unroll
    for (int c = 0; c < D; ++c) {
      T acc = T(0);
#pragma unroll
      for (int k = 0; k < D; ++k) acc += Ej[L::J + S::pk(r, k)] * Ei[L::A + k * D + c];
      TT[r][c] = acc;
    }
  T J_n[S::NP];
#pragma unroll
  for (int r = 0; r < D; ++r)
#pragma unroll
    for (int c = r; c < D; ++c) {
      T a1 = T(0), a2 = T(0);
#pragma unroll
      for (int k = 0; k < D; ++k) {
        a1 += R[k][r] * TT[k][c];
        a2 += R[k][c] * TT[k][r];
      }
      J_n[S::pk(r, c)] = Ei[L::J + S::pk(r, c)] + T(0.5) * (a1 + a2);
    }
  // (A, b, C) with A_j
  T Aj[D][D];
#pragma unroll
  for (int r = 0; r < D; ++r)
#pragma unroll
    for (int c = 0; c < D; ++c) Aj[r][c] = Ej[L::A + r * D + c];
  T b_n[D], A_n[D][D], AW[D][D];
#pragma unroll
  for (int r = 0; r < D; ++r) {
    T acc = Ej[L::B + r];
#pragma unroll
    for (int k = 0; k < D; ++k) acc += Aj[r][k] * R[k][2 * D];
    b_n[r] = acc;
#pragma unroll
    for (int c = 0; c < D; ++c) {
      T a1 = T(0), a2 = T(0);
#pragma unroll
      for (int k = 0; k < D; ++k) {
        a1 += Aj[r][k] * R[k][c];
        a2 += Aj[r][k] * R[k][D + c];
      }
      A_n[r][c] = a1;
      AW[r][c] = a2;
    }
  }
  T C_n[S::NP];
#pragma unroll
  for (int r = 0; r < D; ++r)
#pragma unroll
    for (int c = r; c < D; ++c) {
      T a1 = T(0), a2 = T(0);
#pragma unroll
      for (int k = 0; k < D; ++k) {
        a1 += AW[r][k] * Aj[c][k];
        a2 += AW[c][k] * Aj[r][k];
      }
      C_n[S::pk(r, c)] = Ej[L::C + S::pk(r, c)] + T(0.5) * (a1 + a2);
    }
  // write
#pragma unroll
  for (int r = 0; r < D; ++r) {
#pragma unroll
    for (int c = 0; c < D; ++c) out[L::A + r * D + c] = A_n[r][c];
    out[L::B + r] = b_n[r];
    out[L::ETA + r] = eta_n[r];
  }
#pragma unroll
  for (int i = 0; i < S::NP; ++i) {
    out[L::C + i] = C_n[i];
    out[L::J + i] = J_n[i];
  }
  if constexpr (WITH_C) out[L::NF] = c_n;
}

// ---------------------------------------------------------------------------
// One combination by 16 lanes.  A thread that combines two elements alone runs
// some thousand dependent instructions, straight-line code larger than the
// instruction caches, and takes 5 to 6 us for states of 6 or 7; where there
// are too few combinations to fill the GPU that is their time.  Here each
// column of the right-hand sides (2 D + 1 <= 15) and of X is one lane's, the
// pivot column is broadcast, and the products run a column per lane.  Every
// value is formed by the same operations in the same order as in combine,
// state_through and info_through, so the results are the same bits.
// Elements in shared memory, field by field; all lanes of the warp take part
// (two groups of 16).  The caller synchronises before the results are read.
// ---------------------------------------------------------------------------
constexpr int COOP = 16;

template <int D, class T, int W>
__device__ __forceinline__ void coop_solve(T (&x)[D], T (&r)[D]) {
#pragma unroll
  for (int k = 0; k < D; ++k) {
    T col[D];
#pragma unroll
    for (int i = 0; i < D; ++i) col[i] = __shfl_sync(0xffffffffu, x[i], k, W);
    int piv = k;
    T best = fabs(col[k]);
#pragma unroll
    for (int i = k + 1; i < D; ++i) {
      const T v = fabs(col[i]);
      if (v > best) {
        best = v;
        piv = i;
      }
    }
#pragma unroll
    for (int i = k + 1; i < D; ++i) {
      const bool sw = piv == i;
      const T a = col[k], b = col[i], c = x[k], d = x[i], e = r[k], f = r[i];
      col[k] = sw ? b : a;
      col[i] = sw ? a : b;
      x[k] = sw ? d : c;
      x[i] = sw ? c : d;
      r[k] = sw ? f : e;
      r[i] = sw ? e : f;
    }
    const T ip = T(1) / col[k];
    x[k] *= ip;
    r[k] *= ip;
#pragma unroll
    for (int i = 0; i < D; ++i) {
      if (i == k) continue;
      x[i] -= col[i] * x[k];
      r[i] -= col[i] * r[k];
    }
  }
}

// out <- Ei o Ej (Ei earlier); out may alias either.
template <class S, class T>
__device__ __forceinline__ void combine_coop(const T *Ei, const T *Ej, T *out) {
  using L = Elem<S>;
  constexpr int D = S::D;
  static_assert(2 * D + 1 <= COOP, "a lane per right-hand side");
  const int lane = threadIdx.x & (COOP - 1);
  const int cl = lane < D ? lane : (lane < 2 * D ? lane - D : 0);  // column within its block
  // X = I + C_i J_j and the right-hand sides [A_i | C_i | b_i + C_i eta_j]
  T x[D], r[D], ai[D];
  {
    T v[D];
#pragma unroll
    for (int k = 0; k < D; ++k) v[k] = lane < D ? Ej[L::J + S::pk(k, cl)] : Ej[L::ETA + k];
#pragma unroll
    for (int i = 0; i < D; ++i) {
      T acc = (lane < D && i == cl) ? T(1) : T(0);
#pragma unroll
      for (int k = 0; k < D; ++k) acc += Ei[L::C + S::pk(i, k)] * v[k];
      x[i] = acc;
      ai[i] = Ei[L::A + i * D + cl];
      r[i] = lane < D ? ai[i] : (lane < 2 * D ? Ei[L::C + S::pk(i, cl)] : Ei[L::B + i] + acc);
    }
  }
  coop_solve<D, T, COOP>(x, r);  // lanes hold [Y | W | w]
  // u = eta_j - J_j b_i, then eta and column cl of T = J_j A_i
  T u = T(0), tt[D], eta = Ei[L::ETA + cl];
#pragma unroll
  for (int i = 0; i < D; ++i) {
    T jb = T(0), acc = T(0);
#pragma unroll
    for (int k = 0; k < D; ++k) {
      const T jik = Ej[L::J + S::pk(i, k)];
      jb += jik * Ei[L::B + k];
      acc += jik * ai[k];
    }
    tt[i] = acc;
    u = i == cl ? Ej[L::ETA + i] - jb : u;
  }
#pragma unroll
  for (int k = 0; k < D; ++k) eta += r[k] * __shfl_sync(0xffffffffu, u, k, COOP);
  // column cl of J = (Y^T T + T^T Y) / 2 + J_i
  T jn[D];
#pragma unroll
  for (int i = 0; i < D; ++i) {
    T a1 = T(0), a2 = T(0);
#pragma unroll
    for (int k = 0; k < D; ++k) {
      a1 += __shfl_sync(0xffffffffu, r[k], i, COOP) * tt[k];
      a2 += r[k] * __shfl_sync(0xffffffffu, tt[k], i, COOP);
    }
    jn[i] = Ei[L::J + S::pk(i, cl)] + T(0.5) * (a1 + a2);
  }
  // A_j [Y | W | w]: column of A, of A_j W, and b
  T o[D];
#pragma unroll
  for (int i = 0; i < D; ++i) {
    T acc = lane == 2 * D ? Ej[L::B + i] : T(0);
#pragma unroll
    for (int k = 0; k < D; ++k) acc += Ej[L::A + i * D + k] * r[k];
    o[i] = acc;
  }
  // column cl of C = (A_j W A_j^T + its transpose) / 2 + C_j
  T aj[D], awr[D], a1c[D], cn[D];
#pragma unroll
  for (int k = 0; k < D; ++k) aj[k] = Ej[L::A + cl * D + k];
#pragma unroll
  for (int i = 0; i < D; ++i) {
    T acc = T(0);
#pragma unroll
    for (int k = 0; k < D; ++k) {
      const T v = __shfl_sync(0xffffffffu, o[i], D + k, COOP);
      acc += v * aj[k];
      awr[k] = i == 0 || i == cl ? v : awr[k];
    }
    a1c[i] = acc;
  }
#pragma unroll
  for (int i = 0; i < D; ++i) {
    T acc = T(0);
#pragma unroll
    for (int k = 0; k < D; ++k) acc += awr[k] * Ej[L::A + i * D + k];
    cn[i] = Ej[L::C + S::pk(i, cl)] + T(0.5) * (a1c[i] + acc);
  }
  __syncwarp();  // both elements are read
  if (lane < D) {
#pragma unroll
    for (int i = 0; i < D; ++i) {
      out[L::A + i * D + cl] = o[i];
      if (i <= cl) {
        out[L::J + S::pk(i, cl)] = jn[i];
        out[L::C + S::pk(i, cl)] = cn[i];
      }
    }
    out[L::ETA + cl] = eta;
  } else if (lane == 2 * D) {
#pragma unroll
    for (int i = 0; i < D; ++i) out[L::B + i] = o[i];
  }
}

// Logical index i of a scan of n items -> physical position.
GPSS_HD int phys(int i, int n, int rev) { return rev ? n - 1 - i : i; }

// Combine in time order: with rev_op = 0 the logical order is time order;
// with rev_op = 1 the logical predecessor is later in time.
template <class S, class T>
GPSS_HD void combine_logical(EViewT<T> left, EViewT<T> right, EViewT<T> out, int rev_op) {
  if (rev_op)
    combine<S, T>(right, left, out);
  else
    combine<S, T>(left, right, out);
}

// Element fields of entry idx of a field-major buffer (stride = entries),
// converted to T.
template <class S, class T, class U>
GPSS_HD void load_elem_t(const U *src, size_t stride, size_t idx, T (&A)[S::D][S::D], T *b, T *C,
                         T *eta, T *J) {
  using L = Elem<S>;
  constexpr int D = S::D;
#pragma unroll
  for (int i = 0; i < D; ++i) {
#pragma unroll
    for (int j = 0; j < D; ++j) A[i][j] = T(src[(L::A + i * D + j) * stride + idx]);
    b[i] = T(src[(L::B + i) * stride + idx]);
    eta[i] = T(src[(L::ETA + i) * stride + idx]);
  }
#pragma unroll
  for (int i = 0; i < S::NP; ++i) {
    C[i] = T(src[(L::C + i) * stride + idx]);
    J[i] = T(src[(L::J + i) * stride + idx]);
  }
}

// Filtered state through an element: given the state N(m, P) entering it,
//   m <- A (I + P J)^{-1} (m + P eta) + b,  P <- A (I + P J)^{-1} P A^T + C
// (the combination of a state, an element with A = 0, with the element).
template <class S, class T>
GPSS_HD void state_through(const T (&A)[S::D][S::D], const T *b, const T *C, const T *eta,
                           const T *J, T *m, T *P) {
  constexpr int D = S::D;
  T X[D][D], R[D][D + 1];
#pragma unroll
  for (int i = 0; i < D; ++i) {
    T pe = T(0);
#pragma unroll
    for (int k = 0; k < D; ++k) pe += P[S::pk(i, k)] * eta[k];
    R[i][D] = m[i] + pe;
#pragma unroll
    for (int j = 0; j < D; ++j) {
      T acc = (i == j) ? T(1) : T(0);
#pragma unroll
      for (int k = 0; k < D; ++k) acc += P[S::pk(i, k)] * J[S::pk(k, j)];
      X[i][j] = acc;
      R[i][j] = P[S::pk(i, j)];
    }
  }
  solve_inplace<D, D + 1, T>(X, R);
  T TT[D][D];
#pragma unroll
  for (int i = 0; i < D; ++i) {
    T acc = b[i];
#pragma unroll
    for (int k = 0; k < D; ++k) acc += A[i][k] * R[k][D];
    m[i] = acc;
#pragma unroll
    for (int j = 0; j < D; ++j) {
      T a2 = T(0);
#pragma unroll
      for (int k = 0; k < D; ++k) a2 += A[i][k] * R[k][j];
      TT[i][j] = a2;
    }
  }
#pragma unroll
  for (int i = 0; i < D; ++i)
#pragma unroll
    for (int j = i; j < D; ++j) {
      T acc = C[S::pk(i, j)];
#pragma unroll
      for (int k = 0; k < D; ++k) acc += TT[i][k] * A[j][k];
      P[S::pk(i, j)] = acc;
    }
}

// Information about an element's end state (ie, iJ) carried back to the
// state entering it, plus the element's own information:
//   ie <- A^T (I + iJ C)^{-1} (ie - iJ b) + eta,  iJ <- A^T (I + iJ C)^{-1} iJ A + J.
template <class S, class T>
GPSS_HD void info_through(const T (&A)[S::D][S::D], const T *b, const T *C, const T *eta,
                          const T *J, T *ie, T *iJ) {
  constexpr int D = S::D;
  T X[D][D], R[D][D + 1];
#pragma unroll
  for (int i = 0; i < D; ++i) {
    T jb = T(0);
#pragma unroll
    for (int k = 0; k < D; ++k) jb += iJ[S::pk(i, k)] * b[k];
    R[i][D] = ie[i] - jb;
#pragma unroll
    for (int j = 0; j < D; ++j) {
      T acc = (i == j) ? T(1) : T(0), ja = T(0);
#pragma unroll
      for (int k = 0; k < D; ++k) {
        acc += iJ[S::pk(i, k)] * C[S::pk(k, j)];
        ja += iJ[S::pk(i, k)] * A[k][j];
      }
      X[i][j] = acc;
      R[i][j] = ja;
    }
  }
  solve_inplace<D, D + 1, T>(X, R);
#pragma unroll
  for (int i = 0; i < D; ++i) {
    T acc = eta[i];
#pragma unroll
    for (int k = 0; k < D; ++k) acc += A[k][i] * R[k][D];
    ie[i] = acc;
  }
#pragma unroll
  for (int i = 0; i < D; ++i)
#pragma unroll
    for (int j = i; j < D; ++j) {
      T a1 = T(0), a2 = T(0);
#pragma unroll
      for (int k = 0; k < D; ++k) {
        a1 += A[k][i] * R[k][j];
        a2 += A[k][j] * R[k][i];
      }
      iJ[S::pk(i, j)] = J[S::pk(i, j)] + T(0.5) * (a1 + a2);
    }
}

// Shared memory of the tile kernels: three regions of TL elements
// (working tree, own element, one temporary per thread).
template <class S, int TL, class T>
constexpr size_t tile_smem_bytes() {
  return (size_t)3 * TL * Elem<S>::NF * sizeof(T);
}

template <class S, int TL, class T>
__global__ void __launch_bounds__(TL) k_tile_reduce(const T *__restrict__ src, int n,
                                                    T *__restrict__ dst, int n_tiles,
                                                    int rev_index, int rev_op) {
  using L = Elem<S>;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  T *sm = reinterpret_cast<T *>(sm_raw);
  const int tile = blockIdx.x, tid = threadIdx.x;
  const int i0 = tile * TL;
  const int len = min(TL, n - i0);
  EViewT<T> mine{sm + tid, TL};
  if (tid < len) {
    const T *s = src + phys(i0 + tid, n, rev_index);
    for (int f = 0; f < L::NF; ++f) mine[f] = s[(size_t)f * n];
  }
  __syncthreads();
  for (int s = 1; s < TL; s <<= 1) {
    if ((tid % (2 * s)) == 0 && tid + s < len) {
      EViewT<T> right{sm + tid + s, TL};
      combine_logical<S, T>(mine, right, mine, rev_op);
    }
    __syncthreads();
  }
  if (tid == 0) {
    EViewT<T> out{dst + tile, n_tiles};
    copy_elem<S, T>(out, mine);
  }
}

// Inclusive scan of one tile (logical order) preceded by the inclusive scan
// of earlier tiles, pre[tile - 1] (full elements, logical order, stride
// n_pre; may be null).  Output mode 0: full elements to dst (logical order,
// stride n); mode 3: full elements at the physical position.
template <class S, int TL, class T>
__global__ void __launch_bounds__(TL) k_tile_scan(const T *__restrict__ src, int n,
                                                  const T *__restrict__ pre, int n_pre,
                                                  T *__restrict__ dst, int mode, int rev_index,
                                                  int rev_op) {
  using L = Elem<S>;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  T *sm = reinterpret_cast<T *>(sm_raw);
  const int tile = blockIdx.x, tid = threadIdx.x;
  const int i0 = tile * TL;
  const int len = min(TL, n - i0);
  EViewT<T> mine{sm + tid, TL};
  EViewT<T> own{sm + (size_t)TL * L::NF + tid, TL};
  EViewT<T> tmp{sm + (size_t)2 * TL * L::NF + tid, TL};
  if (tid < len) {
    const T *s = src + phys(i0 + tid, n, rev_index);
    for (int f = 0; f < L::NF; ++f) {
      const T v = s[(size_t)f * n];
      mine[f] = v;
      own[f] = v;
    }
  } else {
    set_identity<S, T>(mine);
    set_identity<S, T>(own);
  }
  __syncthreads();
  // Blelloch up-sweep
  for (int s = 1; s < TL; s <<= 1) {
    const int r = (tid + 1) * 2 * s - 1;
    if (r < TL) {
      EViewT<T> a{sm + r - s, TL}, b{sm + r, TL};
      combine_logical<S, T>(a, b, b, rev_op);
    }
    __syncthreads();
  }
  if (tid == 0) set_identity<S, T>(EViewT<T>{sm + TL - 1, TL});
  __syncthreads();
  // down-sweep: exclusive prefixes
  for (int s = TL / 2; s >= 1; s >>= 1) {
    const int r = (tid + 1) * 2 * s - 1;
    if (r < TL) {
      EViewT<T> a{sm + r - s, TL}, b{sm + r, TL};
      copy_elem<S, T>(tmp, a);  // left subtree total
      copy_elem<S, T>(a, b);    // left child gets the parent's prefix
      combine_logical<S, T>(b, tmp, b, rev_op);
    }
    __syncthreads();
  }
  if (tid >= len) return;
  combine_logical<S, T>(mine, own, own, rev_op);  // inclusive within the tile
  if (pre && tile > 0) {
    for (int f = 0; f < L::NF; ++f) tmp[f] = pre[(size_t)f * n_pre + tile - 1];
    combine_logical<S, T>(tmp, own, own, rev_op);
  }
  const int i = i0 + tid;
  EViewT<T> out{dst + (mode == 3 ? phys(i, n, rev_index) : i), n};
  copy_elem<S, T>(out, own);
}

// k_tile_scan with 16 lanes per combination (blocks of TL x 16 threads, a
// group per element): the same tree, hence the same bits.  One tile of states
// of 5: 47 -> 34 us, four of them 46 -> 39 us (k_tile_reduce, half of whose
// steps have one pair, takes 14 us either way).
template <class S, class T>
__device__ __forceinline__ void combine_coop_logical(const T *left, const T *right, T *out,
                                                     int rev_op) {
  combine_coop<S, T>(rev_op ? right : left, rev_op ? left : right, out);
}

template <class S, int TL>
__global__ void __launch_bounds__(TL *COOP) k_tile_scan_coop(const float *__restrict__ src, int n,
                                                             const float *__restrict__ pre,
                                                             int n_pre, float *__restrict__ dst,
                                                             int mode, int rev_index, int rev_op) {
  constexpr int NF = Elem<S>::NF, ST = Elem<S>::ST;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  float *sm = reinterpret_cast<float *>(sm_raw);  // working tree
  float *own = sm + TL * ST, *tmp = sm + 2 * TL * ST;
  const int tile = blockIdx.x, i0 = tile * TL, len = min(TL, n - i0);
  const int g = threadIdx.x / COOP, ln = threadIdx.x & (COOP - 1);
  for (int t = threadIdx.x; t < TL * NF; t += TL * COOP) {
    const int e = t % TL, f = t / TL;
    float v = (f < Elem<S>::B && f / S::D == f % S::D) ? 1.f : 0.f;  // the identity past the end
    if (e < len) v = src[(size_t)f * n + phys(i0 + e, n, rev_index)];
    sm[e * ST + f] = own[e * ST + f] = v;
  }
  __syncthreads();
  // Blelloch up-sweep (group g: the g-th pair of a level)
  for (int s = 1; s < TL; s <<= 1) {
    if (((g & ~1) + 1) * 2 * s - 1 < TL) {
      const int r = (g + 1) * 2 * s - 1;
      const bool act = r < TL;
      float *spare = tmp + g * ST;
      const float *a = act ? sm + (r - s) * ST : spare, *b = act ? sm + r * ST : spare;
      combine_coop_logical<S, float>(a, b, act ? sm + r * ST : spare, rev_op);
    }
    __syncthreads();
  }
  for (int f = threadIdx.x; f < NF; f += TL * COOP)
    sm[(TL - 1) * ST + f] = (f < Elem<S>::B && f / S::D == f % S::D) ? 1.f : 0.f;
  __syncthreads();
  // down-sweep: exclusive prefixes
  for (int s = TL / 2; s >= 1; s >>= 1) {
    if (((g & ~1) + 1) * 2 * s - 1 < TL) {
      const int r = (g + 1) * 2 * s - 1;
      const bool act = r < TL;
      float *a = act ? sm + (r - s) * ST : tmp + g * ST, *b = act ? sm + r * ST : tmp + g * ST;
      float *left = tmp + g * ST;
      if (act)
        for (int f = ln; f < NF; f += COOP) {
          left[f] = a[f];  // left subtree total
          a[f] = b[f];     // left child gets the parent's prefix
        }
      __syncwarp();
      combine_coop_logical<S, float>(b, left, b, rev_op);
    }
    __syncthreads();
  }
  // inclusive within the tile, then after the earlier tiles
  float *mine = sm + g * ST, *my = own + g * ST, *t = tmp + g * ST;
  combine_coop_logical<S, float>(mine, my, my, rev_op);
  __syncwarp();
  if (pre && tile > 0) {
    for (int f = ln; f < NF; f += COOP) t[f] = pre[(size_t)f * n_pre + tile - 1];
    __syncwarp();
    combine_coop_logical<S, float>(t, my, my, rev_op);
  }
  __syncthreads();
  for (int q = threadIdx.x; q < TL * NF; q += TL * COOP) {
    const int e = q % TL, f = q / TL;
    if (e < len)
      dst[(size_t)f * n + (mode == 3 ? phys(i0 + e, n, rev_index) : i0 + e)] = own[e * ST + f];
  }
}

template <class S, int TL>
constexpr size_t tile_coop_smem_bytes() {
  return (size_t)3 * TL * Elem<S>::ST * sizeof(float);
}

constexpr int SCAN_T = 64;

// Scratch entries of T needed by scan_elems for n elements.
template <class S>
size_t scan_scratch_count(int n) {
  size_t tot = 0;
  while (n > SCAN_T) {
    n = (n + SCAN_T - 1) / SCAN_T;
    tot += (size_t)2 * Elem<S>::NF * n;
  }
  return tot + 1;
}

// Inclusive scan of n elements (field-major, stride n) -> full elements (mode
// 0: logical order; mode 3: physical order).  Recursion depth is log_T(n).
template <class S, class T>
cudaError_t scan_elems(const T *src, int n, T *dst, int mode, int rev_index, int rev_op,
                       T *scratch, int n_sm, cudaStream_t st) {
  constexpr int TL = SCAN_T;
  // 16 lanes per combination for FP32 states of at least 5 while every tile's
  // block has an SM to itself
  constexpr bool LANES = sizeof(T) == sizeof(float) && S::D >= 5;
  const size_t smem = tile_smem_bytes<S, TL, T>();
  static bool attr = false;
  if (!attr) {
    cudaError_t e = cudaFuncSetAttribute(k_tile_scan<S, TL, T>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_tile_reduce<S, TL, T>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if constexpr (LANES) {
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_tile_scan_coop<S, TL>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)tile_coop_smem_bytes<S, TL>());
    }
    if (e != cudaSuccess) return e;
    attr = true;
  }
  if (n <= 0) return cudaSuccess;
  const int nt = (n + TL - 1) / TL;
  auto tiles = [&](const T *pre, int n_pre) {
    if constexpr (LANES) {
      if (nt <= n_sm) {
        k_tile_scan_coop<S, TL><<<nt, TL * COOP, tile_coop_smem_bytes<S, TL>(), st>>>(
            src, n, pre, n_pre, dst, mode, rev_index, rev_op);
        return;
      }
    }
    k_tile_scan<S, TL, T><<<nt, TL, smem, st>>>(src, n, pre, n_pre, dst, mode, rev_index, rev_op);
  };
  if (n <= TL) {
    tiles(nullptr, 0);
    GPSS_COUNT_LAUNCH();
    return cudaGetLastError();
  }
  T *agg = scratch, *aggscan = scratch + (size_t)Elem<S>::NF * nt;
  k_tile_reduce<S, TL, T><<<nt, TL, smem, st>>>(src, n, agg, nt, rev_index, rev_op);
  GPSS_COUNT_LAUNCH();
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  e = scan_elems<S, T>(agg, nt, aggscan, 0, 0, rev_op, aggscan + (size_t)Elem<S>::NF * nt, n_sm,
                       st);
  if (e != cudaSuccess) return e;
  tiles(aggscan, nt);
  GPSS_COUNT_LAUNCH();
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Warp-level combination.  The chunk plan gives every series a multiple of 32
// chunks, so each warp holds 32 consecutive chunks of one series.  Each warp
// scans its 32 elements in shared memory (Kogge-Stone, five steps, warp
// synchronous): inclusive prefixes (forward) and, for the gradient, inclusive
// suffixes (backward), plus the warp's total.  The warp totals -- 32x fewer
// than chunks -- are then scanned by scan_elems (or folded per series), and
// k_join combines the two levels per chunk.  T is the arithmetic of every
// combination (the chunk elements themselves are FP32).
//
// Bound by the instruction caches and the serial chain of a combination where
// warps are few, by instruction issue where they are many.  The directions
// are independent blocks (blockIdx.y) that share one copy of the combination's
// code: 357 warps, states of 5: 34 -> 21 us; 2430 warps, states of 6: 149 ->
// 132 us against one after the other, each with its own copy.
// ---------------------------------------------------------------------------
template <class S, class T>
constexpr size_t warp_scan_smem_bytes(int warps) {
  return (size_t)warps * 2 * 32 * Elem<S>::NF * sizeof(T);
}

template <class S, class T>
__global__ void __launch_bounds__(64) k_warp_scan(const float *__restrict__ ef, int n_vch,
                                                  T *__restrict__ pre_local,
                                                  T *__restrict__ suf_local,
                                                  T *__restrict__ wtot) {
  using L = Elem<S>;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  T *sm = reinterpret_cast<T *>(sm_raw);
  const int lane = threadIdx.x & 31;
  const int vc = blockIdx.x * blockDim.x + threadIdx.x;
  const int n_w = n_vch >> 5;
  const int w = vc >> 5;
  if (w >= n_w) return;  // whole warps only (n_vch is a multiple of 32)
  T *bufA = sm + (size_t)(threadIdx.x >> 5) * 2 * 32 * L::NF;
  T *bufB = bufA + 32 * L::NF;
  const int dir = blockIdx.y;  // 0: prefixes, 1: suffixes
  for (int f = 0; f < L::NF; ++f) bufA[f * 32 + lane] = T(ef[(size_t)f * n_vch + vc]);
  __syncwarp();
  T *src = bufA, *dst = bufB;
  for (int s = 1; s < 32; s <<= 1) {
    const bool act = dir == 0 ? lane >= s : lane + s < 32;
    if (act) {
      // one copy of the combination's code serves both directions
      T *early = src + (dir == 0 ? lane - s : lane), *late = src + (dir == 0 ? lane : lane + s);
      combine<S, T>(EViewT<T>{early, 32}, EViewT<T>{late, 32}, EViewT<T>{dst + lane, 32});
    } else {
      copy_elem<S, T>(EViewT<T>{dst + lane, 32}, EViewT<T>{src + lane, 32});
    }
    __syncwarp();
    T *t = src;
    src = dst;
    dst = t;
  }
  T *out = dir == 0 ? pre_local : suf_local;
  for (int f = 0; f < L::NF; ++f) out[(size_t)f * n_vch + vc] = src[f * 32 + lane];
  if (dir == 0 && lane == 31)
    for (int f = 0; f < L::NF; ++f) wtot[(size_t)f * n_w + w] = src[f * 32 + 31];
}

// The same scan with one block per warp of chunks and direction (blockIdx.y)
// and 16 lanes per combination: the same steps, hence the same bits.
template <class S>
__global__ void __launch_bounds__(32 * COOP) k_warp_scan_coop(const float *__restrict__ ef,
                                                              int n_vch,
                                                              float *__restrict__ pre_local,
                                                              float *__restrict__ suf_local,
                                                              float *__restrict__ wtot) {
  constexpr int NF = Elem<S>::NF, ST = Elem<S>::ST;
  __shared__ float buf[2][32 * ST];
  const int w = blockIdx.x, n_w = n_vch >> 5, dir = blockIdx.y;
  const int vc = w * 32 + (threadIdx.x & 31);
  for (int f = threadIdx.x >> 5; f < NF; f += COOP)
    buf[0][(threadIdx.x & 31) * ST + f] = ef[(size_t)f * n_vch + vc];
  __syncthreads();
  const int e = threadIdx.x / COOP;  // this group's element
  int at = 0;
  for (int s = 1; s < 32; s <<= 1) {
    const float *src = buf[at];
    float *dst = buf[at ^ 1] + e * ST;
    const int o = dir == 0 ? e - s : e + s;
    const bool act = o >= 0 && o < 32;
    // both groups of a warp run the combination; one without a partner on its
    // own element, and then copies it
    const int p = act ? o : e;
    combine_coop<S, float>(src + (dir == 0 ? p : e) * ST, src + (dir == 0 ? e : p) * ST, dst);
    __syncwarp();
    if (!act)
      for (int f = threadIdx.x & (COOP - 1); f < NF; f += COOP) dst[f] = src[e * ST + f];
    __syncthreads();
    at ^= 1;
  }
  float *out = dir == 0 ? pre_local : suf_local;
  for (int f = threadIdx.x >> 5; f < NF; f += COOP)
    out[(size_t)f * n_vch + vc] = buf[at][(threadIdx.x & 31) * ST + f];
  if (dir == 0)
    for (int f = threadIdx.x; f < NF; f += 32 * COOP)
      wtot[(size_t)f * n_w + w] = buf[at][31 * ST + f];
}

// Per chunk: filtered end state = (state entering the warp) o (warp-local
// inclusive prefix); information about the state entering the chunk from it
// and all later chunks of its series = (warp-local inclusive suffix) folded
// with the information from later warps.  wpre / wsuf: inclusive scans of
// the warp totals forward / backward (full elements, stride n_w).
// Records (vector D | packed NP) of T, stride n_vch.
template <class S, class T>
__global__ void __launch_bounds__(128) k_join(int n_vch, int n_chunks,
                                              const uint8_t *__restrict__ ch_flags,
                                              const T *__restrict__ pre_local,
                                              const T *__restrict__ suf_local,
                                              const T *__restrict__ wpre,
                                              const T *__restrict__ wsuf,
                                              T *__restrict__ state_end,
                                              T *__restrict__ info_incl) {
  using L = Elem<S>;
  constexpr int D = S::D;
  const int vc = blockIdx.x * blockDim.x + threadIdx.x;
  if (vc >= n_vch) return;
  const int n_w = n_vch >> 5;
  const int w = vc >> 5, lane = vc & 31;
  const int c0 = (vc - lane) % n_chunks;  // first chunk of this warp
  const bool first_warp = ch_flags[c0] & 1;
  // element of the warp-local prefix
  T A[D][D], b[D], C[S::NP], eta[D], J[S::NP];
  load_elem_t<S, T, T>(pre_local, n_vch, vc, A, b, C, eta, J);
  T m[D], P[S::NP];
  if (first_warp) {
#pragma unroll
    for (int i = 0; i < D; ++i) m[i] = b[i];
#pragma unroll
    for (int i = 0; i < S::NP; ++i) P[i] = C[i];
  } else {
    // state entering the warp: (b, C) of the inclusive warp prefix of w - 1
#pragma unroll
    for (int i = 0; i < D; ++i) m[i] = wpre[(size_t)(L::B + i) * n_w + w - 1];
#pragma unroll
    for (int i = 0; i < S::NP; ++i) P[i] = wpre[(size_t)(L::C + i) * n_w + w - 1];
    state_through<S, T>(A, b, C, eta, J, m, P);
  }
#pragma unroll
  for (int i = 0; i < D; ++i) state_end[(size_t)i * n_vch + vc] = m[i];
#pragma unroll
  for (int i = 0; i < S::NP; ++i) state_end[(size_t)(D + i) * n_vch + vc] = P[i];
  if (!info_incl) return;
  // backward: warp-local inclusive suffix folded with the information from
  // later warps (zero past the end of the series)
  load_elem_t<S, T, T>(suf_local, n_vch, vc, A, b, C, eta, J);
  T ie[D], iJ[S::NP];
  if (w + 1 < n_w) {
#pragma unroll
    for (int i = 0; i < D; ++i) ie[i] = wsuf[(size_t)(L::ETA + i) * n_w + w + 1];
#pragma unroll
    for (int i = 0; i < S::NP; ++i) iJ[i] = wsuf[(size_t)(L::J + i) * n_w + w + 1];
  } else {
#pragma unroll
    for (int i = 0; i < D; ++i) ie[i] = T(0);
#pragma unroll
    for (int i = 0; i < S::NP; ++i) iJ[i] = T(0);
  }
  info_through<S, T>(A, b, C, eta, J, ie, iJ);
#pragma unroll
  for (int i = 0; i < D; ++i) info_incl[(size_t)i * n_vch + vc] = ie[i];
#pragma unroll
  for (int i = 0; i < S::NP; ++i) info_incl[(size_t)(D + i) * n_vch + vc] = iJ[i];
}

// Sequential alternative to the scan of warp totals when every series spans
// only a few warps: one thread per (virtual) series folds its warp totals in
// time order.  Writes, in the field positions k_join reads, the filtered
// state at the end of each warp ((b, C) of wpre) and the information about
// the state entering each warp from it and all later warps of the series
// ((eta, J) of wsuf).
template <class S, class T>
__global__ void __launch_bounds__(64) k_warp_fold(int n_out, int per_series, int n_series,
                                                  int n_chunks,
                                                  const int32_t *__restrict__ ch_first,
                                                  const T *__restrict__ wtot, int n_w,
                                                  T *__restrict__ wpre, T *__restrict__ wsuf,
                                                  int want_info) {
  using L = Elem<S>;
  constexpr int D = S::D;
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n_out) return;
  const int s = per_series ? v : v % n_series;
  const int base = per_series ? 0 : (v / n_series) * n_chunks;
  const int w0 = (base + ch_first[s]) >> 5, w1 = (base + ch_first[s + 1]) >> 5;
  T m[D], P[S::NP];
  for (int w = w0; w < w1; ++w) {
    T A[D][D], b[D], C[S::NP], eta[D], J[S::NP];
    load_elem_t<S, T, T>(wtot, n_w, w, A, b, C, eta, J);
    if (w == w0) {
#pragma unroll
      for (int i = 0; i < D; ++i) m[i] = b[i];
#pragma unroll
      for (int i = 0; i < S::NP; ++i) P[i] = C[i];
    } else {
      state_through<S, T>(A, b, C, eta, J, m, P);
    }
#pragma unroll
    for (int i = 0; i < D; ++i) wpre[(size_t)(L::B + i) * n_w + w] = m[i];
#pragma unroll
    for (int i = 0; i < S::NP; ++i) wpre[(size_t)(L::C + i) * n_w + w] = P[i];
  }
  if (!want_info) return;
  T ie[D], iJ[S::NP];
#pragma unroll
  for (int i = 0; i < D; ++i) ie[i] = T(0);
#pragma unroll
  for (int i = 0; i < S::NP; ++i) iJ[i] = T(0);
  for (int w = w1 - 1; w >= w0; --w) {
    T A[D][D], b[D], C[S::NP], eta[D], J[S::NP];
    load_elem_t<S, T, T>(wtot, n_w, w, A, b, C, eta, J);
    info_through<S, T>(A, b, C, eta, J, ie, iJ);
#pragma unroll
    for (int i = 0; i < D; ++i) wsuf[(size_t)(L::ETA + i) * n_w + w] = ie[i];
#pragma unroll
    for (int i = 0; i < S::NP; ++i) wsuf[(size_t)(L::J + i) * n_w + w] = iJ[i];
  }
}

// The same fold with one warp per (virtual) series and direction (blockIdx.y:
// 0 forward, 1 backward): a lane per column of X and of the right-hand sides,
// the next warp total loaded while the current one is applied.  The same
// operations per value as state_through and info_through, hence the same bits.
// 48 series of 13 warps, states of 7, both directions: 149 -> 21 us; 1024
// series of 1 to 5 warps, states of 6: 20 -> 11 us.
template <class S>
__global__ void __launch_bounds__(32) k_warp_fold_coop(int per_series, int n_series, int n_chunks,
                                                       const int32_t *__restrict__ ch_first,
                                                       const float *__restrict__ wtot, int n_w,
                                                       float *__restrict__ wpre,
                                                       float *__restrict__ wsuf) {
  using T = float;
  using L = Elem<S>;
  constexpr int D = S::D, NF = L::NF, NV = (NF + 31) / 32;
  __shared__ T E[NF], st[D + S::NP];  // the warp total; the state or information
  const int v = blockIdx.x, lane = threadIdx.x, dir = blockIdx.y;
  const int s = per_series ? v : v % n_series;
  const int base = per_series ? 0 : (v / n_series) * n_chunks;
  const int w0 = (base + ch_first[s]) >> 5, w1 = (base + ch_first[s + 1]) >> 5;
  const int cl = lane < D ? lane : 0;
  T nx[NV];
  auto fetch = [&](int w) {
#pragma unroll
    for (int i = 0; i < NV; ++i)
      if (lane + 32 * i < NF) nx[i] = wtot[(size_t)(lane + 32 * i) * n_w + w];
  };
  const int step = dir ? -1 : 1;
  if (w1 > w0) fetch(dir ? w1 - 1 : w0);
  for (int i = lane; i < D + S::NP; i += 32) st[i] = T(0);
  for (int k0 = 0, w = dir ? w1 - 1 : w0; k0 < w1 - w0; ++k0, w += step) {
    __syncwarp();
#pragma unroll
    for (int i = 0; i < NV; ++i)
      if (lane + 32 * i < NF) E[lane + 32 * i] = nx[i];
    if (k0 + 1 < w1 - w0) fetch(w + step);
    __syncwarp();
    T x[D], r[D], o[D], nv[D];
    if (dir == 0) {
      if (k0 == 0) {
        // the series' first warp starts from the prior: its own (b, C)
        for (int i = lane; i < D; i += 32) st[i] = E[L::B + i];
        for (int i = lane; i < S::NP; i += 32) st[D + i] = E[L::C + i];
      } else {
        T q[D];
#pragma unroll
        for (int k = 0; k < D; ++k) q[k] = lane < D ? E[L::J + S::pk(k, cl)] : E[L::ETA + k];
#pragma unroll
        for (int i = 0; i < D; ++i) {
          T acc = (lane < D && i == cl) ? T(1) : T(0);
#pragma unroll
          for (int k = 0; k < D; ++k) acc += st[D + S::pk(i, k)] * q[k];
          x[i] = acc;
          r[i] = lane < D ? st[D + S::pk(i, cl)] : st[i] + acc;
        }
        coop_solve<D, T, 32>(x, r);
        T aj[D];
#pragma unroll
        for (int i = 0; i < D; ++i) {
          T acc = lane == D ? E[L::B + i] : T(0);
#pragma unroll
          for (int k = 0; k < D; ++k) acc += E[L::A + i * D + k] * r[k];
          o[i] = acc;
          aj[i] = E[L::A + cl * D + i];
        }
#pragma unroll
        for (int i = 0; i < D; ++i) {
          T acc = E[L::C + S::pk(i, cl)];
#pragma unroll
          for (int k = 0; k < D; ++k) acc += __shfl_sync(0xffffffffu, o[i], k) * aj[k];
          nv[i] = acc;
        }
      }
    } else {
      T q[D], ac[D];
#pragma unroll
      for (int k = 0; k < D; ++k) {
        q[k] = lane < D ? E[L::C + S::pk(k, cl)] : E[L::B + k];
        ac[k] = E[L::A + k * D + cl];
      }
#pragma unroll
      for (int i = 0; i < D; ++i) {
        T acc = (lane < D && i == cl) ? T(1) : T(0), ja = T(0);
#pragma unroll
        for (int k = 0; k < D; ++k) {
          const T jik = st[D + S::pk(i, k)];
          acc += jik * q[k];
          ja += jik * ac[k];
        }
        x[i] = acc;
        r[i] = lane < D ? ja : st[i] - acc;
      }
      coop_solve<D, T, 32>(x, r);
#pragma unroll
      for (int i = 0; i < D; ++i) {
        T a1 = lane == D ? E[L::ETA + i] : T(0), a2 = T(0);
#pragma unroll
        for (int k = 0; k < D; ++k) {
          a1 += E[L::A + k * D + i] * r[k];
          a2 += ac[k] * __shfl_sync(0xffffffffu, r[k], i);
        }
        o[i] = a1;
        nv[i] = E[L::J + S::pk(i, cl)] + T(0.5) * (a1 + a2);
      }
    }
    __syncwarp();  // the old state is read
    if (dir == 1 || k0 > 0) {
#pragma unroll
      for (int i = 0; i < D; ++i) {
        if (lane < D && i <= cl) st[D + S::pk(i, cl)] = nv[i];
        if (lane == D) st[i] = o[i];
      }
    }
    __syncwarp();
    float *out = dir ? wsuf : wpre;
    const int fv = dir ? L::ETA : L::B, fp = dir ? L::J : L::C;
    for (int i = lane; i < D; i += 32) out[(size_t)(fv + i) * n_w + w] = st[i];
    for (int i = lane; i < S::NP; i += 32) out[(size_t)(fp + i) * n_w + w] = st[D + i];
  }
}

}  // namespace gpss
