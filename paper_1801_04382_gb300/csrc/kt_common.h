// Internal definitions shared by the host runtime and the CUDA kernels.
#pragma once

#include <cmath>
#include <cstdint>

#ifdef __CUDACC__
#define KT_HD __host__ __device__ __forceinline__
#else
#define KT_HD inline
#endif

#define KT_MAX_NODES 8
#define KT_MAX_CTRL 8
#define KT_MAX_CTERMS 16  // control terms (a control acting on one node; two per control in Liouville space)
#define KT_MAX_LIND 4
#define KT_MAX_PAIRS 28
#define KT_MAX_NL 9       // local dimension of the cavity-structure kernels (atom x cavity, cutoff <= 2)
#define KT_MAX_S 4        // off-diagonal entries per row of a node-local generator factor
#define KT_MAX_SH 6       // entries per row of a control factor (update overlap)
#define KT_MAX_K 96       // Chebyshev terms
#define KT_MAX_T 32       // trajectories per tile
#define KT_MAX_ROUNDS 16  // jump-separated pieces of one interval in one kernel

// Kernel families timed by krotov_set_profiling (mirror KT_PROF_* in the public header).
#ifndef KT_PROF_FAMILIES
#define KT_PROF_FAMILIES 5
#define KT_PROF_FWD 0
#define KT_PROF_BWD 1
#define KT_PROF_GRAD 2
#define KT_PROF_CROSS 3
#define KT_PROF_FINISH 4
#endif

// Device status word values (first error wins); mirror kt_status.
#define KT_DEV_OK 0
#define KT_DEV_NONFINITE 5
#define KT_DEV_RECORD_FULL 6
#define KT_DEV_RANGE 8
#define KT_DEV_ZERO_JUMP 9
#define KT_DEV_TIMEOUT 4

// Chebyshev expansion of exp(-i G s) with G = c + r * Ghat (Ghat's spectrum in an ellipse
// around [-1, 1]):  exp(-i G s) = exp(-i c s) sum_k (2 - delta_k0) (-i)^k J_k(r s) T_k(Ghat).
//
// Bessel functions J_0..J_{n-1}(alpha) by Miller's backward recurrence
//   J_{k-1} = (2k / alpha) J_k - J_{k+1},
// started far above the wanted orders from (0, tiny) and normalised with the Neumann
// identity J_0 + 2 sum_{m >= 1} J_{2m} = 1 (J.C.P. Miller, 1952; Numerical Recipes' bessj).
// Values are rescaled whenever they grow past 1e150 so that tiny alpha cannot overflow.
template <typename F>
inline int kt_bessel_miller(F alpha, int n, F *out) {
  if (n < 1 || n > 256 || !(alpha >= 0)) return -1;
  if (alpha < (F)1e-290) {
    out[0] = 1;
    for (int k = 1; k < n; ++k) out[k] = 0;
    return 0;
  }
  int start = n + 20 + (int)(alpha);
  start += (start & 1);                 // even start keeps the Neumann sum bookkeeping simple
  for (int k = 0; k < n; ++k) out[k] = 0;
  F jp1 = 0, jk = (F)1e-200, norm = 0;
  const F inv = 2 / alpha;
  for (int k = start; k >= 1; --k) {
    F jm1 = (F)k * inv * jk - jp1;
    jp1 = jk;
    jk = jm1;                            // jk now holds J_{k-1}
    int km1 = k - 1;
    if (km1 < n) out[km1] = jk;
    if (km1 > 0 && (km1 & 1) == 0) norm += 2 * jk;
    if (jk > (F)1e150 || jk < (F)-1e150) {
      jk *= (F)1e-150; jp1 *= (F)1e-150; norm *= (F)1e-150;
      for (int q = km1; q < n; ++q) out[q] *= (F)1e-150;
    }
  }
  norm += jk;                            // + J_0
  const F s = 1 / norm;
  for (int k = 0; k < n; ++k) out[k] *= s;
  return 0;
}

// Coefficients m_k = (2 - delta_k0) J_k(r s) of a piece of an interval: Taylor series about the middle of the unit segment
// of r s, |x| <= 1/2, cut at KT_PIECE_DEG (what is left is below 2 (1/2)^16 / 16! = 1.5e-18).  The segment's middle is
// exact, so x = r s - middle is rounded at its own size and the value is as good as the table's: Miller's recurrence at
// the middle, in long double because its error grows with the argument (5e-15 at r s = 60 in double).  (Chebyshev series over the whole interval, summed by Clenshaw's recurrence, were off by
// 1.5e-15 ... 3e-15 up to K = 36 and 1.3e-14 at r dt = 60.)
#define KT_PIECE_DEG 15
inline int kt_piece_segments(double alpha_max) { return alpha_max > 1.0 ? (int)std::ceil(alpha_max) : 1; }
// out[segment][n][k], n <= KT_PIECE_DEG, k < K <= KT_MAX_K: with J_k' = (J_{k-1} - J_{k+1}) / 2,
// J_k^(n) = 2^-n sum_i (-1)^i C(n, i) J_{k-n+2i}, J_{-m} = (-1)^m J_m.
inline void kt_piece_table(int segs, int K, double *out) {
  long double L[KT_MAX_K + KT_PIECE_DEG + 1];
  double J[KT_MAX_K + KT_PIECE_DEG + 1];
  for (int q = 0; q < segs; ++q) {
    kt_bessel_miller<long double>(q + 0.5, K + KT_PIECE_DEG + 1, L);
    for (int k = 0; k <= K + KT_PIECE_DEG; ++k) J[k] = (double)L[k];
    for (int k = 0; k < K; ++k) {
      double scale = k == 0 ? 1 : 2;                    // over 2^n n!
      for (int n = 0; n <= KT_PIECE_DEG; ++n) {
        double c = 1, v = 0;                            // (-1)^i C(n, i)
        for (int i = 0; i <= n; ++i) {
          const int m = k - n + 2 * i;
          v += c * (m >= 0 ? J[m] : (m & 1 ? -J[-m] : J[-m]));
          c = -c * (n - i) / (i + 1);
        }
        out[((size_t)q * (KT_PIECE_DEG + 1) + n) * K + k] = scale * v;
        scale /= 2 * (n + 1);
      }
    }
  }
}
KT_HD double kt_piece_coef(const double *table, int segs, int K, int k, double r, double s) {
  const int q0 = (int)(r * s), q = q0 < segs ? q0 : segs - 1;
  const double x = fma(r, s, -(q + 0.5));
  const double *t = table + (size_t)q * (KT_PIECE_DEG + 1) * K + k;
  double v = t[KT_PIECE_DEG * K];
  for (int n = KT_PIECE_DEG - 1; n >= 0; --n) v = fma(v, x, t[n * K]);
  return v;
}

struct KtCplx { double re, im; };

// Problem geometry and constants passed to every kernel by value.
struct KtGeom {
  int n_nodes, n_loc, d, T;          // T = trajectories per tile (interleaved, element-major)
  int tile_elems;                    // complex elements per tile in global memory (>= d*T, multiple of 4)
  int n_tiles, M, M_pad, nthreads;
  int S, SH, n_pairs, n_ctrl, n_lind;
  int K;                             // Chebyshev terms of a full step
  int max_jumps, draws;              // jump cap and uniforms per trajectory and pass
  int prefetch_chi;                  // forward kernel keeps a third tile buffer for chi(t_j)
  int bwd_grid;                      // > 0: backward kernel CTAs looping over tiles, next input prefetched
  int fwd_grid;                      // > 0: the same for the forward kernel (psi and chi of the next tile prefetched)
  int first_order;                   // jump scheme: 0 jump times located in the interval, 1 at most one jump per interval, at its end
  int stride[KT_MAX_NODES];          // element stride of node i (n_loc^(N-1-i))
  int ctrl_node[KT_MAX_CTRL];        // node of control c (its ket node for a density matrix)
  int n_cterms;                      // control terms: control cterm_ctrl[t] acting on node cterm_node[t]
  int cterm_ctrl[KT_MAX_CTERMS];
  int cterm_node[KT_MAX_CTERMS];
  int density;                       // 1: the one "trajectory" is vec(rho) in Liouville space (no jumps, no normalisation)
  double M_norm;                     // M of the update's 1/M: all trajectories of the problem (M, or M_total when sharded)
  int inject_timeout;                // test of the failure path: the first wait for a bulk copy runs out
  double lam[KT_MAX_CTRL];
  double dt, eps_bound;
  double c_fwd, c_bwd, r;            // generator centre (per direction) and half width
};

// Precomputed (pulse independent) tables of one direction, FP64, in global memory: the generator G as
// B = -2i (G - c) / r, so that the series of exp(-i G s) is a real sum of y_k = (-i)^k T_k((G - c) / r) v with
// y_{k+1} = y_{k-1} + B y_k (see kt_device.cuh).
struct KtGenImage {
  const int *loc_dl;          // [N][n_loc][S] local column delta y - x (0 = no entry)
  const KtCplx *loc_base;     // [N][n_loc][S] drift part of B
  const KtCplx *ctrl_slot;    // [n_cterms][n_loc][S] per-unit-eps part of term t on node cterm_node[t]
  const KtCplx *diag_base;    // [N][n_loc] diagonal of B (node 0 also holds the shift by c)
  const KtCplx *ctrl_diag;    // [n_cterms][n_loc] per-unit-eps diagonal part
  const int *pair_off;        // [P][n_loc*n_loc] element offset (in elements, before *T); 0 = none
  const KtCplx *pair_val;     // [P][n_loc*n_loc]
  const double *cheb_full;    // [sets][K] full-step coefficients lambda_s (2 - delta_k0) J_k(r dt)
  const KtCplx *phase_full;   // [sets] exp(-i c dt) / lambda_s
  const double *piece;        // [piece_segs][KT_PIECE_DEG + 1][K] coefficients of a piece of an interval (kt_piece_coef)
  int piece_segs;
  int sets;                   // interval j takes set j % sets (a power of two)
  int quick_pulse;            // each node carries at most one control term and no control touches a diagonal
  const KtCplx *pair_coef;    // [P] coefficient of pair term p (value = coef * a^dag a entries)
  int pair_dst[KT_MAX_PAIRS]; // node raised by pair term p of this direction
  int pair_src[KT_MAX_PAIRS]; // node lowered by pair term p of this direction
  // Cavity-structure kernels with real / imaginary coupling classes: the pulse-independent
  // coefficients that every Chebyshev term reads, as kernel-parameter constants in both precisions
  // (the kernels then take them as constant-bank operands instead of shared-memory loads).
  float kd32[3 * KT_MAX_NL];  // last node's diagonal per local index: real part, imaginary part in two floats (kt_split)
  float ki32[KT_MAX_NL];      // its imaginary part in one float
  double kd64[2 * KT_MAX_NL]; // the same, (re, im)
  float kc32[2 * 2];          // last node's cavity couplings (imaginary): [n-1] row (r, n-1) <- (g, n), [NC + n-1] the reverse
  double kc64[2 * 2];
  float kp32[KT_MAX_PAIRS];   // pair coefficient p (real)
  double kp64[KT_MAX_PAIRS];
  // Block mapping: the pair coefficients by the kinds of their nodes.  Of the outer node i: kh[0][i] and kh[1][i]
  // of the hop that raises the middle / last node and lowers i, kh[2][i] and kh[3][i] of the reverse ones; of
  // the middle and the last node: kh[4][0] raising the last, kh[4][1] raising the middle one.
  float kh[5][2];
  float km[2][2][3];          // kh[0], kh[2] times the ladder values of both nodes: 1, sqrt 2 or 2
};

// FP32 coefficient sets of the y form.  A state that barely changes from one interval to the next meets the same
// roundings of the same coefficients each time, and they add up (up to 1e-7 per interval in the norm); scaling the
// coefficients by a different lambda_s from interval to interval, undone in the two-float phase, makes
// them random: norm off by 1e-6 ... 1e-5 -> 1e-7 ... 2.6e-6 after 100 intervals (d = 81, 216, eight pulses).
// Set 0 is not scaled (lambda_0 = 1): the T form uses it alone.
#define KT_COEF_SETS 32

// A diagonal value as a float on a 2^-21 grid and the float of what is left.  The dominant part of the
// diagonal's phase otherwise turns by its own rounding, 6e-8 r dt per interval and always the same way;
// the parts of different nodes add without rounding on the grid.
KT_HD void kt_split(double v, float *hi, float *lo) {
  const double h = (double)(long long)(v * 2097152.0 + (v < 0.0 ? -0.5 : 0.5)) * (1.0 / 2097152.0);
  *hi = (float)h;
  *lo = (float)(v - (double)*hi);
}

// Pulse-independent operators shared by both directions.
struct KtOps {
  const int *lo_dl;           // [n_loc] ladder factor a: row x -> column x + lo_dl[x]
  const KtCplx *lo_val;       // [n_loc] value (0 = empty row)
  const int *ra_dl;           // [n_loc] adjoint a^dag: row x -> column x + ra_dl[x]
  const KtCplx *ra_val;       // [n_loc]
  const KtCplx *lind_coef;    // [n_lind][N]
  const int *hc_dl;           // [n_cterms][n_loc][SH] control term factor (unscaled), column delta
  const KtCplx *hc_val;       // [n_cterms][n_loc][SH] (0 = no entry)
  const uint32_t *digits;     // [d] node digits of each basis index, node i in bits 4i..4i+3
  const KtCplx *tgt;          // [d] target state
};
