#pragma once
// CUDA kernels of the trajectory-parallel Krotov hot path (sm_103a).
//
// One CTA owns a tile of T trajectories for one time interval.  The tile's states sit in
// global memory as [d][T] complex (element-major, trajectories interleaved), so that a warp
// whose items share an element index (T = 32) runs the structured generator uniformly and
// reads its neighbours from consecutive shared-memory words.
//
// Per interval the CTA applies exp(-i G dt) by a Chebyshev series (paper Sec. 2.1: exact
// propagation over long steps, the basic operation being the matrix-vector product of
// Sec. 2.3), keeping y_{k-1}/y_{k+1} and y_k in two shared-memory buffers and the running
// sum in registers.  G is never formed: it is the sum of node-local factors, pair hops
// a_dst^dag a_src and a diagonal, all read from small per-interval tables in shared memory.
//
// The series is run in y_k = (-i)^k T_k((G - c) / r) v with B = -2i (G - c) / r in the tables:
//   y_0 = v,  y_1 = B v / 2,  y_{k+1} = y_{k-1} + B y_k,
//   exp(-i G s) v = exp(-i c s) sum_k m_k y_k,  m_k = (2 - delta_k0) J_k(r s) real.
// Against T_k with complex coefficients this saves two FMAs per element and term in the sum.  In FP32 a row is
// summed from its small terms up (couplings, then y_{k-1}, then the diagonal), and the diagonal's imaginary part
// and the phase are held as two floats: the error of Delta eps against 64 bits is 0.6e-6 ... 3.7e-6 where the T form's is
// 2.4e-6 ... 8.5e-6 (d = 216, 101 intervals, eight pulses), 0.8e-6 ... 3.2e-6 where it is 3.5e-6 ... 5.8e-6 (d = 81,
// 100 intervals).
//
// FP32 fibers and blocks run the T form all the same (t_form below), except in the sweeps that keep states for the
// gradient.  The norm of the FP32 state decides in which interval a trajectory jumps, a threshold can lie closer to
// the norm at t_j than its rounding, and a jump moved by an interval moves Delta eps by about 1 / M.  With hundreds of
// trajectories that happens in one sweep out of ten if the rounding of the norm changes by 5e-6, as it does between the
// two forms; with the T form the outcome of these problems is what it has always been.  It costs 3 % at d = 6561 and
// nothing at d = 729, where the shared-memory pipe is the bound.
#include <cuda_runtime.h>
#include <stdint.h>

#include "kt_common.h"
#include "kt_kernels.h"

namespace kt {

template <typename R> struct C2;
template <> struct C2<float> { typedef float2 T; };
template <> struct C2<double> { typedef double2 T; };

__device__ __forceinline__ float2 mkc(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ double2 mkc(double a, double b) { return make_double2(a, b); }

template <typename C> __device__ __forceinline__ C cmul(C a, C b) {
  return mkc(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
template <typename C> __device__ __forceinline__ C cfma(C a, C b, C c) {  // c + a*b
  c.x = fma(a.x, b.x, c.x);
  c.x = fma(-a.y, b.y, c.x);
  c.y = fma(a.x, b.y, c.y);
  c.y = fma(a.y, b.x, c.y);
  return c;
}

template <typename C> __device__ __forceinline__ C cmul_fma(C a, C b) {  // a*b with its roundings written out
  return mkc(fma(a.x, b.x, -(a.y * b.y)), fma(a.y, b.x, a.x * b.y));
}

// c + a*b for a purely real (rfma, a) or purely imaginary (ifma, i b) coefficient: the two
// FMAs of cfma whose coefficient part is nonzero, in cfma's order, so the result is bit-identical.
template <typename C, typename R> __device__ __forceinline__ C rfma(R a, C b, C c) {
  c.x = fma(a, b.x, c.x);
  c.y = fma(a, b.y, c.y);
  return c;
}
template <typename C, typename R> __device__ __forceinline__ C ifma(R bi, C b, C c) {
  c.x = fma(-bi, b.y, c.x);
  c.y = fma(bi, b.x, c.y);
  return c;
}

template <typename C> __device__ __forceinline__ C from_kc(KtCplx z) {
  typedef decltype(C().x) R;
  return mkc((R)z.re, (R)z.im);
}

__device__ __forceinline__ void set_status(int *status, int code) {
  atomicCAS(status, KT_DEV_OK, code);
}

// ---- bulk (TMA) copies between global and shared memory, completing on an mbarrier -------
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(unsigned long long *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// one thread: arm the barrier for `bytes` and start the copy global -> shared
// (addresses 16-byte aligned, size a multiple of 16)
__device__ __forceinline__ void bulk_load(void *dst_smem, const void *src_gmem, uint32_t bytes,
                                          unsigned long long *bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(smem_u32(dst_smem)), "l"(src_gmem), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(unsigned long long *bar, uint32_t phase) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(phase)
      : "memory");
  return ok != 0;
}

#define KT_WAIT_CYCLES 4000000000LL   // ~2 s of SM clock

// wait (one thread) for phase `phase` of the barrier, giving up after `budget` cycles of clock
__device__ __forceinline__ bool mbar_wait_bounded(unsigned long long *bar, uint32_t phase,
                                                  long long budget = KT_WAIT_CYCLES) {
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, phase))
    if (clock64() - t0 > budget) return false;
  return true;
}

// one thread: copy shared -> global (16-byte aligned, size a multiple of 16) as one bulk group
__device__ __forceinline__ void bulk_store(void *dst_gmem, const void *src_smem, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst_gmem), "r"(smem_u32(src_smem)),
               "r"(bytes)
               : "memory");
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
__device__ __forceinline__ void bulk_store_wait() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// Exchange of the update's tile partials within a whole-sweep launch.  Every interval has its own slots, filled
// with kNoValue before the launch and written once, so that a value carries its own arrival: a reader polls
// the slots it sums.  Nothing else passes between CTAs, so no fence is needed, and the exchange takes one store
// and one load through L2 where a counter barrier took two round trips, two fences and a second read
// (d = 81, 128
// trajectories, FP32: 13.7 -> 11.8 us per updating interval together with the merged reduction of norm and overlap).
constexpr unsigned long long kNoValue = ~0ull;   // a NaN that no arithmetic produces

__device__ __forceinline__ void put_partial(double *slot, double v) {
  unsigned long long b = (unsigned long long)__double_as_longlong(v);
  if (b == kNoValue) b = 0x7ff8000000000000ull;
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(slot), "l"(b) : "memory");
}
__device__ __forceinline__ unsigned long long get_partial(const double *slot) {
  unsigned long long b;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(b) : "l"(slot) : "memory");
  return b;
}

// Whole-tile load by the bulk engine: thread 0 waits (bounded, ~2 s) and the block learns the
// outcome.  On a timeout the status word gets KT_DEV_TIMEOUT, thread 0 waits once more (~2 s) so
// that the copy in flight lands before the block leaves, and false is returned to every thread.
// idle_bar (a test of this failure path, kt_config.inject_copy_timeout): the first wait watches a
// barrier nothing arrives at, for ~10 us, so that the timeout path runs deterministically.
__device__ __forceinline__ bool tile_wait(unsigned long long *bar, uint32_t phase, int *flag_slot, int *status,
                                          unsigned long long *idle_bar) {
  if (threadIdx.x == 0) {
    const bool ok = idle_bar ? mbar_wait_bounded(idle_bar, 0, 20000) : mbar_wait_bounded(bar, phase);
    if (!ok) {
      set_status(status, KT_DEV_TIMEOUT);
      mbar_wait_bounded(bar, phase);   // give the copy in flight a second bounded chance to land
    }
    *flag_slot = ok ? 1 : 0;
  }
  __syncthreads();
  return *flag_slot != 0;
}

// --------------------------------------------------------------------------------------
// Shared-memory carve-up (identical on host and device; see kt_smem_bytes).
struct Smem {
  void *bufA, *bufB;          // [tile_elems] complex each
  void *bufC;                 // [tile_elems] prefetched chi(t_j) (forward kernel, when it fits)
  void *bufD;                 // [tile_elems] the next tile's prefetched psi (forward kernel looping over tiles)
  unsigned long long *mbar;   // [4] transaction barriers of the bulk copies ([0], [3] psi, [1] chi); [2] never receives an arrival
  int *loc_off;               // [N*n_loc*S]  element offset * T (0 = no entry)
  void *loc_val;              // [N*n_loc*S]
  void *diag;                 // [N*n_loc] diagonal of B: real part, imaginary part (FP32: its first float)
  void *diag_lo;              // [N*n_loc] FP32: the imaginary part's second float
  int *pair_off;              // [P*n_loc^2]
  void *pair_val;             // [P*n_loc^2]
  int *hc_off;                // [n_cterms*n_loc*SH]
  void *hc_val;               // [n_cterms*n_loc*SH]
  void *coef;                 // [K][T] real; complex in the T form
  void *phase;                // [3][T] exp(-i c s) (FP32: in two floats, and r s / 2)
  double *red;                // [nwarps][T][8]
  double *tsc;                // per-trajectory scalars [TS_V0 + 8][T]
  int *tin;                   // per-trajectory ints [16][T]
  double *eps;                // [n_ctrl]
  int *flag;                  // [8] block flags
  void *ldense;               // [n_loc][n_loc] last node's factor, dense (cavity-structure path)
  void *lora;                 // [2][n_loc] ladder values a (row x) and a^dag (row x)
  void *pcoef;                // [P] scaled pair coefficients
};

__host__ __device__ inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

__host__ __device__ inline size_t carve(const KtGeom &g, int esz, char *base, Smem *s, bool with_c,
                                        bool with_d = false) {
  const int nl2 = g.n_loc * g.n_loc;
  const int nwarps = g.nthreads / 32;
  size_t off = 0;
  auto take = [&](size_t bytes) -> char * {
    off = align_up(off, 16);
    char *p = base ? base + off : nullptr;
    off += bytes;
    return p;
  };
  const size_t tile = (size_t)g.tile_elems * esz;
  char *a = take(tile), *b = take(tile);
  char *cbuf = with_c ? take(tile) : nullptr;
  char *dbuf = with_d ? take(tile) : nullptr;
  char *mb = take(4 * sizeof(unsigned long long));
  char *lo = take(sizeof(int) * g.n_nodes * g.n_loc * g.S);
  char *lv = take((size_t)esz * g.n_nodes * g.n_loc * g.S);
  char *dg = take((size_t)esz * g.n_nodes * g.n_loc);
  char *dgl = take((size_t)esz / 2 * g.n_nodes * g.n_loc);
  char *po = take(sizeof(int) * g.n_pairs * nl2);
  char *pv = take((size_t)esz * g.n_pairs * nl2);
  char *ho = take(sizeof(int) * g.n_cterms * g.n_loc * g.SH);
  char *hv = take((size_t)esz * g.n_cterms * g.n_loc * g.SH);
  char *cf = take((size_t)esz * g.K * g.T);
  char *phs = take((size_t)esz * 3 * g.T);
  char *rd = take(sizeof(double) * nwarps * g.T * 8);
  char *ts = take(sizeof(double) * 18 * g.T);
  char *ti = take(sizeof(int) * 16 * g.T);
  char *ep = take(sizeof(double) * KT_MAX_CTRL);
  char *fl = take(sizeof(int) * 8);
  char *ld = take((size_t)esz * g.n_loc * g.n_loc);
  char *lr = take((size_t)esz * 2 * g.n_loc);
  char *pc = take((size_t)esz * (g.n_pairs > 0 ? g.n_pairs : 1));
  if (s) {
    s->bufA = a; s->bufB = b; s->bufC = cbuf; s->bufD = dbuf; s->mbar = (unsigned long long *)mb; s->loc_off = (int *)lo; s->loc_val = lv; s->diag = dg; s->diag_lo = dgl;
    s->pair_off = (int *)po; s->pair_val = pv; s->hc_off = (int *)ho; s->hc_val = hv;
    s->coef = cf; s->phase = phs; s->red = (double *)rd; s->tsc = (double *)ts; s->tin = (int *)ti;
    s->eps = (double *)ep; s->flag = (int *)fl;
    s->ldense = ld; s->lora = lr; s->pcoef = pc;
  }
  return align_up(off, 16);
}

// per-trajectory scalar slots in Smem::tsc / Smem::tin
enum { TS_R = 0, TS_LO, TS_HI, TS_S0, TS_S, TS_PS, TS_PP, TS_C, TS_LEN, TS_X, TS_V0 };   // TS_V0: 8 values per trajectory
enum { TI_ACT = 0, TI_BUSY, TI_CH, TI_NJ, TI_J0, TI_J1, TI_J2, TI_J3, TI_J4, TI_J5, TI_J6, TI_J7,
       TI_J8, TI_J9, TI_J10, TI_J11 };

// --------------------------------------------------------------------------------------
// Per-trajectory block reduction: every thread holds NV partial sums of its trajectory
// (tau = tid % T); sums over lanes of equal tau by shuffles, then over warps in a fixed
// order.  Result in out[tau*NV + v].  Deterministic (FP64 throughout).
// For NV a power of two the first shuffle levels transpose: at offset o a lane sends half of its
// live values to its partner and adds the partner's other half, so each level halves the live
// values (8 values over 5 levels: 9 additions per lane instead of 40 -- FP64 runs at 1/64 of the
// FP32 rate on this GPU).  Slot q of lane l then holds value q + idx(l), idx from the lane bits of
// the transposing levels; the remaining levels add plainly.
template <int NV>
__device__ __forceinline__ void reduce_tau(double (&v)[NV], const KtGeom &g, double *red, double *out) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  int o = 16, live = NV, idx = 0, tmask = 0;
  if constexpr (NV > 1 && (NV & (NV - 1)) == 0) {
#pragma unroll
    for (int h = NV / 2; h >= 1; h >>= 1) {
      if (o >= g.T) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int q = 0; q < h; ++q) {
          const double send = up ? v[q] : v[q + h];
          const double keep = up ? v[q + h] : v[q];
          v[q] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
        if (up) idx += h;
        tmask |= o;
        live = h;
        o >>= 1;
      }
    }
  }
  for (; o >= g.T; o >>= 1) {
#pragma unroll
    for (int q = 0; q < NV; ++q)
      if (q < live) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
  }
  if (((lane & ~(g.T - 1)) & ~tmask) == 0) {
    const int tau = lane & (g.T - 1);
#pragma unroll
    for (int q = 0; q < NV; ++q)
      if (q < live) red[(warp * g.T + tau) * 8 + q + idx] = v[q];
  }
  __syncthreads();
  if ((NV & (NV - 1)) == 0 && g.T == 1) {
    // one trajectory: the warps' sums by a tree over one warp (one thread adding 23 of them took 1 us)
    if (threadIdx.x < 32) {
      const int q = lane % NV;
      double s = 0.0;
      for (int w = lane / NV; w < nwarps; w += 32 / NV) s += red[w * 8 + q];
#pragma unroll
      for (int h = NV; h < 32; h <<= 1) s += __shfl_xor_sync(0xffffffffu, s, h);
      if (lane < NV) out[q] = s;
    }
  } else {
    for (int t = threadIdx.x; t < g.T * NV; t += blockDim.x) {
      const int tau = t / NV, q = t % NV;
      double s = 0.0;
      for (int w = 0; w < nwarps; ++w) s += red[(w * g.T + tau) * 8 + q];
      out[tau * NV + q] = s;
    }
  }
  __syncthreads();
}

// --------------------------------------------------------------------------------------
// Diagonal of B: re + i (hi + lo), lo only in FP32 (kt_split).  diag_init starts a row's sum, diag_done
// adds y_{k-1} and the diagonal: in FP32 the smallest terms come first and only the last two additions
// round at the size of the result; in FP64 they come first, off the path from the neighbours' loads to the result.  lo turns an element by r s lo / 2 ~ 1e-7 over a series: apply_phase turns the
// result by it once (what the order of that turn and the couplings leaves out is a hundred times smaller).
template <typename R> struct Diag { R re, hi, lo; };

// T form of the series (FP32 fibers and blocks): T_{k+1} = 2 Ghat T_k - T_{k-1} with 2 Ghat = i B, and complex coefficients
// a_k = (2 - delta_k0) (-i)^k J_k(r s) exp(-i c s), one set for all intervals; a row is summed from the diagonal on (one
// float), then the last node, the other nodes in turn and the hops, every FMA written out.  The order and the roundings
// are part of the results (top of this file).  ACS 11, 12, 13: the mappings 3, 4, 5 in the y form.
template <typename R, int NL, int ACS> __host__ __device__ constexpr bool t_form() { return sizeof(R) == 4 && NL > 0 && ACS < 8; }
template <typename R, bool TF> struct CoefT { typedef R T; };
template <typename R> struct CoefT<R, true> { typedef typename C2<R>::T T; };
template <typename R, bool TF> using Coef = typename CoefT<R, TF>::T;
template <typename R, typename C> __device__ __forceinline__ C coef_mul(R a, C v) {
  if constexpr (sizeof(R) == sizeof(C)) return cmul_fma(a, v);
  else return mkc(a * v.x, a * v.y);
}
template <typename R, typename C> __device__ __forceinline__ C coef_fma(R a, C v, C c) {
  if constexpr (sizeof(R) == sizeof(C)) return cfma(a, v, c);
  else return rfma(a, v, c);
}
// c + i w v, c + w v, c + w v of an entry i w, w (real), w (complex) of B; T form: of 2 Ghat = i B
template <bool TF, typename R, typename C> __device__ __forceinline__ C add_im(R w, C v, C c) { return TF ? rfma(-w, v, c) : ifma(w, v, c); }
template <bool TF, typename R, typename C> __device__ __forceinline__ C add_re(R w, C v, C c) { return TF ? ifma(w, v, c) : rfma(w, v, c); }
template <bool TF, typename C> __device__ __forceinline__ C add_cx(C w, C v, C c) { return cfma(TF ? mkc(-w.y, w.x) : w, v, c); }

__device__ __forceinline__ void store_diag(const Smem &sm, int e, float2 *dg, double re, double im) {
  float hi, lo;
  kt_split(im, &hi, &lo);
  dg[e] = make_float2((float)re, hi);
  ((float *)sm.diag_lo)[e] = lo;
}
__device__ __forceinline__ void store_diag(const Smem &, int e, double2 *dg, double re, double im) {
  dg[e] = make_double2(re, im);
}
template <typename R, bool TF = false> __device__ __forceinline__ Diag<R> load_diag(const Smem &sm, int e) {
  const typename C2<R>::T v = ((const typename C2<R>::T *)sm.diag)[e];
  if constexpr (TF) return Diag<R>{v.x, v.y + ((const R *)sm.diag_lo)[e], (R)0};
  return Diag<R>{v.x, v.y, sizeof(R) == 4 ? ((const R *)sm.diag_lo)[e] : (R)0};
}
template <typename R> __device__ __forceinline__ Diag<R> add_diag(Diag<R> a, Diag<R> b) {
  return Diag<R>{a.re + b.re, a.hi + b.hi, sizeof(R) == 4 ? a.lo + b.lo : (R)0};
}
// Keeps the sums of D with a fiber's constants inside the loop: hoisted, they take two registers per element and spill.
__device__ __forceinline__ void keep_in_loop(Diag<float> &D) { asm volatile("" : "+f"(D.re), "+f"(D.hi)); }
__device__ __forceinline__ void keep_in_loop(Diag<double> &D) { asm volatile("" : "+d"(D.re), "+d"(D.hi)); }
template <bool TF = false, typename R, typename C> __device__ __forceinline__ C diag_init(Diag<R> D, C v, C old) {
  if constexpr (TF) return cmul_fma(mkc(-D.hi, D.re), v);
  else if constexpr (sizeof(R) == 4) return mkc(D.re * v.x, D.re * v.y);
  else return mkc(fma(-D.hi, v.y, fma(D.re, v.x, old.x)), fma(D.hi, v.x, fma(D.re, v.y, old.y)));
}
template <bool TF = false, typename R, typename C> __device__ __forceinline__ C diag_done(Diag<R> D, C v, C old, C s) {
  if constexpr (TF) {
    s.x -= old.x;
    s.y -= old.y;
  } else if constexpr (sizeof(R) == 4) {
    s.x += old.x;
    s.y += old.y;
    s.x = fma(-D.hi, v.y, s.x);
    s.y = fma(D.hi, v.x, s.y);
  }
  return s;
}

// acc times exp(-i c s) of trajectory tau and (FP32) 1 + i lo(q) r s / 2 of each element
// (T form: nothing, the phase is in the coefficients)
template <typename R, int N, bool TF = false, class LO>
__device__ __forceinline__ void apply_phase(const KtGeom &g, const Smem &sm, int tau, typename C2<R>::T (&acc)[N], LO lo_of) {
  typedef typename C2<R>::T C;
  if constexpr (TF) return;
  const C ph = ((const C *)sm.phase)[tau];
  if constexpr (sizeof(R) == 4) {
    const C lo = ((const C *)sm.phase)[g.T + tau];
    const R half = ((const C *)sm.phase)[2 * g.T + tau].x;
#pragma unroll
    for (int q = 0; q < N; ++q) {
      const R t = half * lo_of(q);
      const C z = mkc(lo.x - t * ph.y, lo.y + t * ph.x);
      acc[q] = cfma(ph, acc[q], cmul(z, acc[q]));
    }
  } else {
#pragma unroll
    for (int q = 0; q < N; ++q) acc[q] = cmul(ph, acc[q]);
  }
}
// phase of trajectory tau: exp(-i c s) (full steps: over lambda) in two floats, and r s / 2
template <typename R>
__device__ __forceinline__ void store_phase(const KtGeom &g, const Smem &sm, int tau, double re, double im, double s) {
  typedef typename C2<R>::T C;
  C *ph = (C *)sm.phase;
  const C hi = mkc((R)re, (R)im);
  ph[tau] = hi;
  if (sizeof(R) == 4) {
    ph[g.T + tau] = mkc((R)(re - (double)hi.x), (R)(im - (double)hi.y));
    ph[2 * g.T + tau] = mkc((R)(0.5 * g.r * s), (R)0);
  }
}

// --------------------------------------------------------------------------------------
// Per-interval tables: the factors of B for pulse eps, plus control factors for the update overlap.
template <typename R>
// pulse_only: the tables of a later interval of a whole sweep -- only the entries that depend on the
// pulse (node factors, diagonal, the last node's dense factor) are rebuilt, the rest is unchanged.
__device__ void build_tables(const KtGeom &g, const KtGenImage &im, const KtOps &ops, const Smem &sm,
                             const double *eps, bool with_hc, bool pulse_only = false) {
  typedef typename C2<R>::T C;
  C *lv = (C *)sm.loc_val;
  C *dg = (C *)sm.diag;
  C *pv = (C *)sm.pair_val;
  const int nls = g.n_loc * g.S;
  for (int e = threadIdx.x; e < g.n_nodes * nls; e += blockDim.x) {
    const int i = e / nls, rem = e % nls;
    double re = im.loc_base[e].re, imv = im.loc_base[e].im;
    for (int t = 0; t < g.n_cterms; ++t)
      if (g.cterm_node[t] == i) {
        re += eps[g.cterm_ctrl[t]] * im.ctrl_slot[t * nls + rem].re;
        imv += eps[g.cterm_ctrl[t]] * im.ctrl_slot[t * nls + rem].im;
      }
    lv[e] = mkc((R)re, (R)imv);
    if (!pulse_only) sm.loc_off[e] = im.loc_dl[e] * g.stride[i] * g.T;
  }
  for (int e = threadIdx.x; e < g.n_nodes * g.n_loc; e += blockDim.x) {
    const int i = e / g.n_loc, x = e % g.n_loc;
    double re = im.diag_base[e].re, imv = im.diag_base[e].im;
    for (int t = 0; t < g.n_cterms; ++t)
      if (g.cterm_node[t] == i) {
        re += eps[g.cterm_ctrl[t]] * im.ctrl_diag[t * g.n_loc + x].re;
        imv += eps[g.cterm_ctrl[t]] * im.ctrl_diag[t * g.n_loc + x].im;
      }
    store_diag(sm, e, dg, re, imv);
  }
  const int nl2 = g.n_loc * g.n_loc;
  if (!pulse_only)
    for (int e = threadIdx.x; e < g.n_pairs * nl2; e += blockDim.x) {
      sm.pair_off[e] = im.pair_off[e] * g.T;
      pv[e] = from_kc<C>(im.pair_val[e]);
    }
  {
    // last node's factor as a dense n_loc x n_loc table, ladder values, pair coefficients
    C *ld = (C *)sm.ldense;
    C *lr = (C *)sm.lora;
    C *pc = (C *)sm.pcoef;
    const int last = g.n_nodes - 1;
    for (int e = threadIdx.x; e < g.n_loc * g.n_loc; e += blockDim.x) ld[e] = mkc((R)0, (R)0);
    if (!pulse_only) {
      for (int e = threadIdx.x; e < g.n_loc; e += blockDim.x) {
        lr[e] = from_kc<C>(ops.lo_val[e]);
        lr[g.n_loc + e] = from_kc<C>(ops.ra_val[e]);
      }
      for (int e = threadIdx.x; e < g.n_pairs; e += blockDim.x) pc[e] = from_kc<C>(im.pair_coef[e]);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < g.n_loc * g.S; e += blockDim.x) {
      const int idx = last * nls + e, x = e / g.S, dl = im.loc_dl[idx];
      if (dl) ld[x * g.n_loc + x + dl] = lv[idx];
    }
  }
  if (with_hc && !pulse_only) {
    C *hv = (C *)sm.hc_val;
    const int nh = g.n_loc * g.SH;
    for (int e = threadIdx.x; e < g.n_cterms * nh; e += blockDim.x) {
      const int t = e / nh;
      sm.hc_off[e] = ops.hc_dl[e] * g.stride[g.cterm_node[t]] * g.T;
      hv[e] = from_kc<C>(ops.hc_val[e]);
    }
  }
}

// old + B v at one item (element x, trajectory tau) of tile vector v.
template <typename R>
__device__ __forceinline__ typename C2<R>::T apply_item(const KtGeom &g, const KtGenImage &im, const Smem &sm,
                                                        const typename C2<R>::T *__restrict__ v,
                                                        int item, uint32_t dig, Diag<R> D,
                                                        typename C2<R>::T old) {
  typedef typename C2<R>::T C;
  const C *lv = (const C *)sm.loc_val;
  const C *pv = (const C *)sm.pair_val;
  const C vi = v[item];
  C out = diag_init(D, vi, old);
  for (int i = 0; i < g.n_nodes; ++i) {
    const int xi = (dig >> (4 * i)) & 15;
    const int base = (i * g.n_loc + xi) * g.S;
    for (int s = 0; s < g.S; ++s) {
      const int off = sm.loc_off[base + s];
      if (off) out = cfma(lv[base + s], v[item + off], out);
    }
  }
  const int nl2 = g.n_loc * g.n_loc;
  for (int p = 0; p < g.n_pairs; ++p) {
    const int xd = (dig >> (4 * im.pair_dst[p])) & 15;
    const int xs = (dig >> (4 * im.pair_src[p])) & 15;
    const int idx = p * nl2 + xd * g.n_loc + xs;
    const int off = sm.pair_off[idx];
    if (off) out = cfma(pv[idx], v[item + off], out);
  }
  return diag_done(D, vi, old, out);
}

template <typename R>
__device__ __forceinline__ Diag<R> diag_of(const KtGeom &g, const Smem &sm, uint32_t dig) {
  Diag<R> s{(R)0, (R)0, (R)0};
  for (int i = 0; i < g.n_nodes; ++i) s = add_diag(s, load_diag<R>(sm, i * g.n_loc + ((dig >> (4 * i)) & 15)));
  return s;
}

// Items of this thread: item_q = tid + q * nthreads, valid while < d*T.
template <int EPT, bool FIBER>
struct ItemsT {
  // strided mapping: item_q = tid + q * nthreads
  int item_[EPT];
  uint32_t dig_[EPT];
  bool ok_[EPT];
  __device__ __forceinline__ int item(int q) const { return item_[q]; }
  __device__ __forceinline__ uint32_t dig(int q) const { return dig_[q]; }
  __device__ __forceinline__ bool ok(int q) const { return ok_[q]; }
};
template <int EPT>
struct ItemsT<EPT, true> {
  // fiber mapping: the thread's items run along the last node's digit, so everything follows
  // from the first item, the fiber's digits (last digit 0) and the tile width
  int base, T, shift;
  uint32_t fdig;
  bool okf;
  __device__ __forceinline__ int item(int q) const { return base + q * T; }
  __device__ __forceinline__ uint32_t dig(int q) const { return fdig + ((uint32_t)q << shift); }
  __device__ __forceinline__ bool ok(int) const { return okf; }
};
// block mapping: NP fibers per thread, the photon numbers of the middle node (the one before the last) at a
// fixed state of its atom -- EPT = NP * NL consecutive elements, tile width 1
template <int EPT, int NL>
struct ItemsB {
  int base, shift;
  uint32_t fdig;
  bool okf;
  __device__ __forceinline__ int item(int q) const { return base + q; }
  __device__ __forceinline__ uint32_t dig(int q) const {
    return fdig + ((uint32_t)(q / NL) << (shift - 4)) + ((uint32_t)(q % NL) << shift);
  }
  __device__ __forceinline__ bool ok(int) const { return okf; }
};
template <int EPT, int NL> struct ItemsSel { typedef ItemsB<EPT, NL> T; };
template <int EPT> struct ItemsSel<EPT, 0> { typedef ItemsT<EPT, false> T; };
template <int EPT> struct ItemsSel<EPT, EPT> { typedef ItemsT<EPT, true> T; };
template <int EPT, int NL>
using Items = typename ItemsSel<EPT, NL>::T;

template <int EPT, int NL>
__device__ __forceinline__ void load_items(const KtGeom &g, const KtOps &ops, Items<EPT, NL> &it) {
  if constexpr (NL > 0 && EPT > NL) {
    it.okf = (int)threadIdx.x < g.d / EPT;
    it.base = threadIdx.x * EPT;
    it.shift = 4 * (g.n_nodes - 1);
    it.fdig = it.okf ? ops.digits[it.base] : 0u;
  } else if constexpr (NL > 0) {
    // fiber mapping: thread -> (fiber f, trajectory tau); its NL items run along the last
    // node's digit (stride T in the interleaved tile), so node-local and pair coefficients of
    // the other nodes are fixed per thread and the last node's are uniform per item slot
    const int f = threadIdx.x / g.T, tau = threadIdx.x % g.T;
    it.okf = f < g.d / NL;
    it.base = f * NL * g.T + tau;
    it.T = g.T;
    it.shift = 4 * (g.n_nodes - 1);
    it.fdig = it.okf ? ops.digits[f * NL] : 0u;
  } else {
    const int n = g.d * g.T;
#pragma unroll
    for (int q = 0; q < EPT; ++q) {
      const int item = threadIdx.x + q * blockDim.x;
      it.item_[q] = item;
      it.ok_[q] = item < n;
      it.dig_[q] = it.ok_[q] ? ops.digits[item / g.T] : 0u;
    }
  }
}

// out[q] = old[q] + (B v)[item_q] for the whole fiber of this thread, q < NL, old[q] = prev[item_q] (PREV
// false: 0).  Coefficients of nodes other than the last are looked up once per fiber; those of the last
// node depend only on q and are the same for every lane.
template <typename R, int NL, bool PREV, bool TF>
__device__ __forceinline__ void apply_fiber(const KtGeom &g, const KtGenImage &im, const Smem &sm,
                                            const typename C2<R>::T *__restrict__ v,
                                            const typename C2<R>::T *prev, int base, uint32_t fdig, Diag<R> Df,
                                            typename C2<R>::T (&out)[NL]) {
  typedef typename C2<R>::T C;
  const C *lv = (const C *)sm.loc_val;
  const C *pv = (const C *)sm.pair_val;
  const int last = g.n_nodes - 1;
  const int T = g.T;
  const C zero = mkc((R)0, (R)0);
#pragma unroll
  for (int q = 0; q < NL; ++q)
    out[q] = diag_init<TF>(add_diag(Df, load_diag<R, TF>(sm, last * NL + q)), v[base + q * T], PREV ? prev[base + q * T] : zero);
  // last node: row q of its factor
#pragma unroll
  for (int q = 0; q < NL; ++q) {
    const int e0 = (last * NL + q) * g.S;
    for (int s = 0; s < g.S; ++s) {
      const int off = sm.loc_off[e0 + s];
      if (off) out[q] = add_cx<TF>(lv[e0 + s], v[base + q * T + off], out[q]);
    }
  }
  // other nodes: one row per fiber
  for (int i = 0; i < last; ++i) {
    const int e0 = (i * NL + ((fdig >> (4 * i)) & 15)) * g.S;
    for (int s = 0; s < g.S; ++s) {
      const int off = sm.loc_off[e0 + s];
      if (off) {
        const C w = lv[e0 + s];
#pragma unroll
        for (int q = 0; q < NL; ++q) out[q] = add_cx<TF>(w, v[base + q * T + off], out[q]);
      }
    }
  }
  // pair hops a_dst^dag a_src
  for (int p = 0; p < g.n_pairs; ++p) {
    const int pd = im.pair_dst[p], ps = im.pair_src[p];
    const int pb = p * NL * NL;
    if (pd != last && ps != last) {
      const int e = pb + ((fdig >> (4 * pd)) & 15) * NL + ((fdig >> (4 * ps)) & 15);
      const int off = sm.pair_off[e];
      if (off) {
        const C w = pv[e];
#pragma unroll
        for (int q = 0; q < NL; ++q) out[q] = add_cx<TF>(w, v[base + q * T + off], out[q]);
      }
    } else if (pd == last) {
      const int e0 = pb + ((fdig >> (4 * ps)) & 15);
#pragma unroll
      for (int q = 0; q < NL; ++q) {
        const int off = sm.pair_off[e0 + q * NL];
        if (off) out[q] = add_cx<TF>(pv[e0 + q * NL], v[base + q * T + off], out[q]);
      }
    } else {
      const int e0 = pb + ((fdig >> (4 * pd)) & 15) * NL;
#pragma unroll
      for (int q = 0; q < NL; ++q) {
        const int off = sm.pair_off[e0 + q];
        if (off) out[q] = add_cx<TF>(pv[e0 + q], v[base + q * T + off], out[q]);
      }
    }
  }
#pragma unroll
  for (int q = 0; q < NL; ++q)
    out[q] = diag_done<TF>(add_diag(Df, load_diag<R, TF>(sm, last * NL + q)), v[base + q * T], PREV ? prev[base + q * T] : zero,
                       out[q]);
}

// Chebyshev sum in fiber mapping (see cheb_run).
template <typename R, int NL, bool TF, class IT>
__device__ void cheb_run_fiber(const KtGeom &g, const KtGenImage &im, const Smem &sm, const IT &it, int K,
                               typename C2<R>::T (&acc)[NL]) {
  typedef typename C2<R>::T C;
  C *A = (C *)sm.bufA;
  C *B = (C *)sm.bufB;
  const Coef<R, TF> *cf = (const Coef<R, TF> *)sm.coef;
  const int tau = threadIdx.x % g.T;
  const bool ok = it.ok(0);
  const int base = it.item(0);
  const uint32_t fdig = it.dig(0);
  const int last = g.n_nodes - 1;
  Diag<R> Df{(R)0, (R)0, (R)0};
  for (int i = 0; i < last; ++i) Df = add_diag(Df, load_diag<R, TF>(sm, i * NL + ((fdig >> (4 * i)) & 15)));
  const Coef<R, TF> c0 = cf[tau];
#pragma unroll
  for (int q = 0; q < NL; ++q) {
    const C v = ok ? A[base + q * g.T] : mkc((R)0, (R)0);
    acc[q] = coef_mul(c0, v);
  }
  if (K > 1) {
    C t[NL];
    if (ok) {
      apply_fiber<R, NL, false, TF>(g, im, sm, A, A, base, fdig, Df, t);
      const Coef<R, TF> c1 = cf[g.T + tau];
#pragma unroll
      for (int q = 0; q < NL; ++q) {
        t[q] = mkc((R)0.5 * t[q].x, (R)0.5 * t[q].y);
        B[base + q * g.T] = t[q];
        acc[q] = coef_fma(c1, t[q], acc[q]);
      }
    }
    __syncthreads();
    C *P = A;   // holds y_{k-1}; receives y_{k+1}
    C *Q = B;   // holds y_k
    for (int k = 2; k < K; ++k) {
      if (ok) {
        const Coef<R, TF> a = cf[k * g.T + tau];
        apply_fiber<R, NL, true, TF>(g, im, sm, Q, P, base, fdig, Df, t);
#pragma unroll
        for (int q = 0; q < NL; ++q) {
          P[base + q * g.T] = t[q];
          acc[q] = coef_fma(a, t[q], acc[q]);
        }
      }
      __syncthreads();
      C *tmp = P; P = Q; Q = tmp;
    }
  } else {
    __syncthreads();
  }
  apply_phase<R, NL, TF>(g, sm, tau, acc, [&](int q) { return Df.lo + load_diag<R, TF>(sm, last * NL + q).lo; });
}

// Chebyshev sum: acc = exp(-i c s) sum_k coef[k][tau] y_k with y_0 = v in A on entry (synced).
// A and B are overwritten.  Ends synchronised.
template <typename R, int EPT, class IT>
__device__ void cheb_run(const KtGeom &g, const KtGenImage &im, const Smem &sm, const IT &it, int K,
                         typename C2<R>::T (&acc)[EPT]) {
  typedef typename C2<R>::T C;
  C *A = (C *)sm.bufA;
  C *B = (C *)sm.bufB;
  const R *cf = (const R *)sm.coef;
  const int tau = threadIdx.x % g.T;
  Diag<R> dv[EPT];
  const R c0 = cf[tau];
#pragma unroll
  for (int q = 0; q < EPT; ++q) {
    acc[q] = mkc((R)0, (R)0);
    if (!it.ok(q)) continue;
    dv[q] = diag_of<R>(g, sm, it.dig(q));
    const C v = A[it.item(q)];
    acc[q] = mkc(c0 * v.x, c0 * v.y);
  }
  if (K > 1) {
    const R c1 = cf[g.T + tau];
#pragma unroll
    for (int q = 0; q < EPT; ++q) {
      if (!it.ok(q)) continue;
      C t = apply_item<R>(g, im, sm, A, it.item(q), it.dig(q), dv[q], mkc((R)0, (R)0));
      t = mkc((R)0.5 * t.x, (R)0.5 * t.y);
      B[it.item(q)] = t;
      acc[q] = rfma(c1, t, acc[q]);
    }
    __syncthreads();
    C *P = A;   // holds y_{k-1}; receives y_{k+1}
    C *Q = B;   // holds y_k
    for (int k = 2; k < K; ++k) {
      const R a = cf[k * g.T + tau];
#pragma unroll
      for (int q = 0; q < EPT; ++q) {
        if (!it.ok(q)) continue;
        const C nv = apply_item<R>(g, im, sm, Q, it.item(q), it.dig(q), dv[q], P[it.item(q)]);
        P[it.item(q)] = nv;
        acc[q] = rfma(a, nv, acc[q]);
      }
      __syncthreads();
      C *tmp = P; P = Q; Q = tmp;
    }
  } else {
    __syncthreads();
  }
  apply_phase<R, EPT>(g, sm, tau, acc, [&](int q) { return it.ok(q) ? dv[q].lo : (R)0; });
}

// m (-i)^k (cs + i sn)
template <typename R> __device__ __forceinline__ typename C2<R>::T t_coef(int k, double m, double cs, double sn) {
  switch (k & 3) {
    case 0: return mkc((R)(m * cs), (R)(m * sn));
    case 1: return mkc((R)(m * sn), (R)(-m * cs));
    case 2: return mkc((R)(-m * cs), (R)(-m * sn));
  }
  return mkc((R)(-m * sn), (R)(m * cs));
}

// Coefficients of exp(-i G s) for every trajectory, s in sm.tsc[TS_X] (synchronised): m_k = (2 - delta_k0) J_k(r s) and the
// phase exp(-i c s).  Called by the whole block, one thread per coefficient: a Taylor series of 16 terms.  (One thread
// running Miller's recurrence for all orders took longer than a series of a small problem in FP64, where an
// instruction costs a warp 64 cycles however few of its lanes work: passes with several jumps per trajectory at d = 81
// 28.5 -> 25.3 ms, d = 216 FP32 9.9 -> 8.3 ms, d = 729 FP32 26.9 -> 25.4 ms.)
template <typename R, bool TF>
__device__ void piece_coefs(const KtGeom &g, const KtGenImage &im, const Smem &sm, double c_gen) {
  Coef<R, TF> *cf = (Coef<R, TF> *)sm.coef;
  for (int e = threadIdx.x; e < g.K * g.T; e += blockDim.x) {
    const int k = e / g.T;
    const double m = kt_piece_coef(im.piece, im.piece_segs, g.K, k, g.r, sm.tsc[TS_X * g.T + e % g.T]);
    if constexpr (TF) {
      double sn, cs;
      sincos(-c_gen * sm.tsc[TS_X * g.T + e % g.T], &sn, &cs);
      cf[e] = t_coef<R>(k, m, cs, sn);
    } else {
      cf[e] = (R)m;
    }
  }
  if constexpr (TF) return;
  const int t = blockDim.x - 1 - threadIdx.x;   // the phases on the last warp
  if (t < g.T) {
    const double s = sm.tsc[TS_X * g.T + t];
    double sn, cs;
    sincos(-c_gen * s, &sn, &cs);
    store_phase<R>(g, sm, t, cs, sn, s);
  }
}

template <typename R, bool TF>
__device__ void uniform_coefs(const KtGeom &g, const Smem &sm, const KtGenImage &im, int j) {
  Coef<R, TF> *cf = (Coef<R, TF> *)sm.coef;
  const int set = TF ? 0 : j & (im.sets - 1);   // set 0 is not scaled
  const double *full = im.cheb_full + (size_t)set * g.K;
  for (int e = threadIdx.x; e < g.K * g.T; e += blockDim.x) {
    if constexpr (TF) cf[e] = t_coef<R>(e / g.T, full[e / g.T], im.phase_full[0].re, im.phase_full[0].im);
    else cf[e] = (R)full[e / g.T];
  }
  if constexpr (TF) return;
  for (int t = threadIdx.x; t < g.T; t += blockDim.x)
    store_phase<R>(g, sm, t, im.phase_full[set].re, im.phase_full[set].im, g.dt);
}

// What a whole sweep keeps from interval to interval: its thread's entry of the node factors with the control term on
// it, and (tile width 1) the coefficient sets, behind the carve.  Rebuilding the tables from global memory, with the
// last node's dense factor and the two-float diagonal that the small problems' mappings do not use or that no control
// changes, and loading the coefficients again took a third of a d = 81 interval.
struct SweepKeep {
  double base_re, base_im, slot_re, slot_im;
  int ctrl;          // control of this thread's entry, -1: none (or no entry)
  bool quick, sets;
};

__host__ __device__ inline size_t sweep_keep_bytes(const KtGeom &g, int esz, int sets) {
  return g.T == 1 ? (size_t)esz / 2 * (((size_t)sets * g.K + 7) / 8 * 8) + (size_t)esz * 3 * sets : 0;
}

template <typename R>
__device__ __forceinline__ void sweep_keep_init(const KtGeom &g, const KtGenImage &im, char *extra, SweepKeep &kp) {
  typedef typename C2<R>::T C;
  const int nls = g.n_loc * g.S, e = threadIdx.x;
  kp.quick = im.quick_pulse && g.n_nodes * nls <= (int)blockDim.x;
  kp.sets = g.T == 1;
  kp.ctrl = -1;
  if (kp.quick && e < g.n_nodes * nls) {
    const int i = e / nls, rem = e % nls;
    kp.base_re = im.loc_base[e].re;
    kp.base_im = im.loc_base[e].im;
    for (int t = 0; t < g.n_cterms; ++t)
      if (g.cterm_node[t] == i) {
        kp.slot_re = im.ctrl_slot[t * nls + rem].re;
        kp.slot_im = im.ctrl_slot[t * nls + rem].im;
        if (kp.slot_re != 0.0 || kp.slot_im != 0.0) kp.ctrl = g.cterm_ctrl[t];
      }
  }
  if (kp.sets) {
    R *cf = (R *)extra;
    C *ph = (C *)(cf + (im.sets * g.K + 7) / 8 * 8);
    for (int q = threadIdx.x; q < im.sets * g.K; q += blockDim.x) cf[q] = (R)im.cheb_full[q];
    for (int q = threadIdx.x; q < im.sets; q += blockDim.x) {
      Smem t;
      t.phase = ph + 3 * q;
      store_phase<R>(g, t, 0, im.phase_full[q].re, im.phase_full[q].im, g.dt);
    }
  }
}

// Tables of the next interval (sm.eps is synchronised; a barrier must follow before they are read).
template <typename R>
__device__ __forceinline__ void sweep_tables(const KtGeom &g, const KtGenImage &im, const KtOps &ops, const Smem &sm,
                                             const SweepKeep &kp) {
  typedef typename C2<R>::T C;
  if (!kp.quick) {
    build_tables<R>(g, im, ops, sm, sm.eps, false, true);
  } else if (kp.ctrl >= 0) {
    const double e = sm.eps[kp.ctrl];
    ((C *)sm.loc_val)[threadIdx.x] = mkc((R)(kp.base_re + e * kp.slot_re), (R)(kp.base_im + e * kp.slot_im));
  }
}

// Full-step coefficients and phase of interval j: the kept set (in run, the copy of sm that the series takes: the jump
// phases write their coefficients through sm, and must not write over the sets), or loaded.
template <typename R>
__device__ __forceinline__ void sweep_coefs(const KtGeom &g, const KtGenImage &im, const Smem &sm, Smem &run,
                                            const SweepKeep &kp, char *extra, int j) {
  typedef typename C2<R>::T C;
  if (kp.sets) {
    const int set = j & (im.sets - 1);
    run.coef = (R *)extra + set * g.K;
    run.phase = (C *)((R *)extra + (im.sets * g.K + 7) / 8 * 8) + 3 * set;
  } else {
    uniform_coefs<R, false>(g, sm, im, j);
  }
}

template <typename R, int EPT, class IT>
__device__ __forceinline__ void load_tile(const KtGeom &g, const IT &it, const typename C2<R>::T *src,
                                          typename C2<R>::T *dst) {
#pragma unroll
  for (int q = 0; q < EPT; ++q)
    if (it.ok(q)) dst[it.item(q)] = src[it.item(q)];
}

// (sum_i coef_i a_i) v  (adj = 0)  or  (sum_i conj(coef_i) a_i^dag) v  (adj = 1) at one item.
template <typename R>
__device__ __forceinline__ typename C2<R>::T lind_item(const KtGeom &g, const KtOps &ops, int l, int adj,
                                                       const typename C2<R>::T *v, int item, uint32_t dig) {
  typedef typename C2<R>::T C;
  C out = mkc((R)0, (R)0);
  for (int i = 0; i < g.n_nodes; ++i) {
    const int xi = (dig >> (4 * i)) & 15;
    KtCplx lc = ops.lind_coef[l * g.n_nodes + i];
    KtCplx av = adj ? ops.ra_val[xi] : ops.lo_val[xi];
    const int dl = adj ? ops.ra_dl[xi] : ops.lo_dl[xi];
    if (av.re == 0.0 && av.im == 0.0) continue;
    if (lc.re == 0.0 && lc.im == 0.0) continue;
    if (adj) lc.im = -lc.im;
    const double wr = lc.re * av.re - lc.im * av.im, wi = lc.re * av.im + lc.im * av.re;
    out = cfma(mkc((R)wr, (R)wi), v[item + dl * g.stride[i] * g.T], out);
  }
  return out;
}

// --------------------------------------------------------------------------------------
// Cavity-structure fast path.  Valid when every node is a three-level atom {g, e, r} times a
// cavity with photon numbers 0..NC (local index atom * (NC+1) + n), the ladder factor is the
// cavity annihilation operator, and the last node's factor couples only (r, n-1) <-> (g, n)
// (cavity) and (r, n) <-> (e, n) (drive) besides its diagonal -- the node of Sec. 3.1.  Then
// every coupling inside a thread's fiber (which runs over the last node) has a position known
// at compile time: the fiber's own T_k stays in registers and the last node's factor and the
// pair hops that raise or lower its photon number become register-indexed FMAs.
// The fiber's rows of the other nodes' factors (at most three other nodes on the fiber path: the
// fiber of the last node holds n_loc^(N-1) <= 736 threads' worth of the tile), loaded once per
// Chebyshev series: element offsets of the two slots and their coefficients -- slot 0 a real entry of G
// (imaginary in B), slot 1 an imaginary one (real in B).
template <typename R>
struct RowCache {
  int off0[3], off1[3];
  R a[3], b[3];
};

template <typename R, int NL>
__device__ __forceinline__ void load_rows(const KtGeom &g, const Smem &sm, uint32_t fdig, RowCache<R> &rc) {
  typedef typename C2<R>::T C;
  const C *lv = (const C *)sm.loc_val;
  const int last = g.n_nodes - 1;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    rc.off0[i] = rc.off1[i] = 0;
    rc.a[i] = rc.b[i] = (R)0;
    if (i < last) {
      const int e0 = (i * NL + ((fdig >> (4 * i)) & 15)) * 2;
      rc.off0[i] = sm.loc_off[e0];
      rc.off1[i] = sm.loc_off[e0 + 1];
      rc.a[i] = lv[e0].y;
      rc.b[i] = lv[e0 + 1].x;
    }
  }
}

// Constants of the real / imaginary kernels (kernel parameters of the image, see KtGenImage).
template <typename R, bool TF = false> __device__ __forceinline__ Diag<R> acs_kd(const KtGenImage &im, int q) {
  if constexpr (sizeof(R) == 8) return Diag<R>{im.kd64[2 * q], im.kd64[2 * q + 1], 0.0};
  else if constexpr (TF) return Diag<R>{im.kd32[3 * q], im.ki32[q], 0.f};
  else return Diag<R>{im.kd32[3 * q], im.kd32[3 * q + 1], im.kd32[3 * q + 2]};
}
template <typename R> __device__ __forceinline__ const R *acs_kc(const KtGenImage &im);
template <> __device__ __forceinline__ const float *acs_kc<float>(const KtGenImage &im) { return im.kc32; }
template <> __device__ __forceinline__ const double *acs_kc<double>(const KtGenImage &im) { return im.kc64; }
template <typename R> __device__ __forceinline__ const R *acs_kp(const KtGenImage &im);
template <> __device__ __forceinline__ const float *acs_kp<float>(const KtGenImage &im) { return im.kp32; }
template <> __device__ __forceinline__ const double *acs_kp<double>(const KtGenImage &im) { return im.kp64; }
// sqrt(n) for the photon numbers n <= 2 of the cavity-structure node (<n-1|a|n>; the host has
// checked that the ladder factor holds exactly these values)
template <typename R>
__device__ __forceinline__ R sqrt_n(int n) {
  return n >= 2 ? (R)1.4142135623730951 : (n == 1 ? (R)1 : (R)0);
}

// out[q] = old[q] + (B v)[base + q T] for the thread's fiber, vk its own values of v, old[q] = prev[base + q T]
// (PREV false: 0).
// RI: the couplings are purely real or imaginary by class (host check: node rows of G hold
// [real, imaginary] slots, last-node cavity real and drive imaginary, pair coefficients imaginary --
// in B = -2i G the classes change places --
// ladder values sqrt(n), no control on the last node's diagonal or cavity couplings), applied with
// two FMAs each; the pulse-independent coefficients (last node's diagonal and cavity couplings,
// pair coefficients, ladder values) are kernel-parameter or compile-time constants, so only the
// drive couplings, the other nodes' pair tables and the states are read from shared memory.
// CACHE: the other nodes' rows come from rc (registers, the reverse gradient) instead of the shared tables.
template <typename R, int NC, int TT, bool RI, bool CACHE, bool PREV, bool TF>
__device__ __forceinline__ void apply_acs(const KtGeom &g, const KtGenImage &im, const Smem &sm,
                                          const typename C2<R>::T *__restrict__ v,
                                          const typename C2<R>::T *prev, int base, uint32_t fdig, Diag<R> Df,
                                          const typename C2<R>::T (&vk)[3 * (NC + 1)],
                                          typename C2<R>::T (&out)[3 * (NC + 1)], const RowCache<R> &rc) {
  typedef typename C2<R>::T C;
  constexpr int NP = NC + 1, NL = 3 * NP;
  const C *lv = (const C *)sm.loc_val;
  const C *pv = (const C *)sm.pair_val;
  const C *ld = (const C *)sm.ldense;
  const C *lo = (const C *)sm.lora;
  const C *ra = lo + NL;
  const C *pc = (const C *)sm.pcoef;
  const int last = g.n_nodes - 1;
  const int T = TT > 0 ? TT : g.T;   // TT > 0: tile width fixed at compile time
  auto diag = [&](int q) -> Diag<R> {
    if constexpr (RI) return add_diag(Df, acs_kd<R, TF>(im, q));
    else return add_diag(Df, load_diag<R, TF>(sm, last * NL + q));
  };
  const C zero = mkc((R)0, (R)0);
#pragma unroll
  for (int q = 0; q < NL; ++q) out[q] = diag_init<TF>(diag(q), vk[q], PREV ? prev[base + q * T] : zero);
  // last node: cavity (r, n-1) <-> (g, n) and drive (r, n) <-> (e, n)
#pragma unroll
  for (int n = 1; n <= NC; ++n) {
    const int qr = 2 * NP + n - 1, qg = n;
    if constexpr (RI) {
      out[qr] = add_im<TF>(acs_kc<R>(im)[n - 1], vk[qg], out[qr]);
      out[qg] = add_im<TF>(acs_kc<R>(im)[NC + n - 1], vk[qr], out[qg]);
    } else {
      out[qr] = add_cx<TF>(ld[qr * NL + qg], vk[qg], out[qr]);
      out[qg] = add_cx<TF>(ld[qg * NL + qr], vk[qr], out[qg]);
    }
  }
#pragma unroll
  for (int n = 0; n <= NC; ++n) {
    const int qr = 2 * NP + n, qe = NP + n;
    if constexpr (RI) {
      out[qr] = add_re<TF>(ld[qr * NL + qe].x, vk[qe], out[qr]);
      out[qe] = add_re<TF>(ld[qe * NL + qr].x, vk[qr], out[qe]);
    } else {
      out[qr] = add_cx<TF>(ld[qr * NL + qe], vk[qe], out[qr]);
      out[qe] = add_cx<TF>(ld[qe * NL + qr], vk[qr], out[qe]);
    }
  }
  // other nodes: one row per fiber, each entry one neighbouring fiber
  if constexpr (RI && !CACHE) {
    for (int i = 0; i < last; ++i) {
      const int e0 = (i * NL + ((fdig >> (4 * i)) & 15)) * 2;
      const int off0 = sm.loc_off[e0], off1 = sm.loc_off[e0 + 1];
      if (off0) {
        const R a = lv[e0].y;
#pragma unroll
        for (int q = 0; q < NL; ++q) out[q] = add_im<TF>(a, v[base + off0 + q * T], out[q]);
      }
      if (off1) {
        const R b = lv[e0 + 1].x;
#pragma unroll
        for (int q = 0; q < NL; ++q) out[q] = add_re<TF>(b, v[base + off1 + q * T], out[q]);
      }
    }
  } else if constexpr (RI) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      if (rc.off0[i]) {
#pragma unroll
        for (int q = 0; q < NL; ++q) out[q] = add_im<TF>(rc.a[i], v[base + rc.off0[i] + q * T], out[q]);
      }
      if (rc.off1[i]) {
#pragma unroll
        for (int q = 0; q < NL; ++q) out[q] = add_re<TF>(rc.b[i], v[base + rc.off1[i] + q * T], out[q]);
      }
    }
  } else {
    for (int i = 0; i < last; ++i) {
      const int e0 = (i * NL + ((fdig >> (4 * i)) & 15)) * g.S;
      for (int s = 0; s < g.S; ++s) {
        const int off = sm.loc_off[e0 + s];
        if (off) {
          const C w = lv[e0 + s];
#pragma unroll
          for (int q = 0; q < NL; ++q) out[q] = add_cx<TF>(w, v[base + off + q * T], out[q]);
        }
      }
    }
  }
  // pair hops coef a_dst^dag a_src
  for (int p = 0; p < g.n_pairs; ++p) {
    const int pd = im.pair_dst[p], ps = im.pair_src[p];
    if (pd != last && ps != last) {
      const int e = p * NL * NL + ((fdig >> (4 * pd)) & 15) * NL + ((fdig >> (4 * ps)) & 15);
      const int off = sm.pair_off[e];
      if (off) {
        if constexpr (RI) {
          const R b = pv[e].x;
#pragma unroll
          for (int q = 0; q < NL; ++q) out[q] = add_re<TF>(b, v[base + off + q * T], out[q]);
        } else {
          const C w = pv[e];
#pragma unroll
          for (int q = 0; q < NL; ++q) out[q] = add_cx<TF>(w, v[base + off + q * T], out[q]);
        }
      }
    } else if (pd == last) {
      // raise the last node (q <- q-1, n_q >= 1), lower node ps (x_s -> x_s + 1, n_s < NC)
      const int xs = (fdig >> (4 * ps)) & 15;
      if (xs % NP < NC) {
        const int off = g.stride[ps] * T;
        if constexpr (RI) {
          const R cb = acs_kp<R>(im)[p] * sqrt_n<R>(xs % NP + 1);
#pragma unroll
          for (int q = 0; q < NL; ++q) {
            if (q % NP == 0) continue;
            out[q] = add_re<TF>(cb * sqrt_n<R>(q % NP), v[base + off + (q - 1) * T], out[q]);
          }
        } else {
          const C cf = cmul(pc[p], lo[xs]);
#pragma unroll
          for (int q = 0; q < NL; ++q) {
            if (q % NP == 0) continue;
            out[q] = add_cx<TF>(cmul(cf, ra[q]), v[base + off + (q - 1) * T], out[q]);
          }
        }
      }
    } else {
      // lower the last node (q <- q+1, n_q < NC), raise node pd (x_d -> x_d - 1, n_d >= 1)
      const int xd = (fdig >> (4 * pd)) & 15;
      if (xd % NP >= 1) {
        const int off = -g.stride[pd] * T;
        if constexpr (RI) {
          const R cb = acs_kp<R>(im)[p] * sqrt_n<R>(xd % NP);
#pragma unroll
          for (int q = 0; q < NL; ++q) {
            if (q % NP == NC) continue;
            out[q] = add_re<TF>(cb * sqrt_n<R>(q % NP + 1), v[base + off + (q + 1) * T], out[q]);
          }
        } else {
          const C cf = cmul(pc[p], ra[xd]);
#pragma unroll
          for (int q = 0; q < NL; ++q) {
            if (q % NP == NC) continue;
            out[q] = add_cx<TF>(cmul(cf, lo[q]), v[base + off + (q + 1) * T], out[q]);
          }
        }
      }
    }
  }
#pragma unroll
  for (int q = 0; q < NL; ++q) out[q] = diag_done<TF>(diag(q), vk[q], PREV ? prev[base + q * T] : zero, out[q]);
}

template <typename R, int NC, int TT, bool RI, bool TF, class IT>
__device__ void cheb_run_acs(const KtGeom &g, const KtGenImage &im, const Smem &sm, const IT &it,
                             int K, typename C2<R>::T (&acc)[3 * (NC + 1)]) {
  typedef typename C2<R>::T C;
  constexpr int NL = 3 * (NC + 1);
  C *A = (C *)sm.bufA;
  C *B = (C *)sm.bufB;
  const Coef<R, TF> *cf = (const Coef<R, TF> *)sm.coef;
  const int T = TT > 0 ? TT : g.T;
  const int tau = TT == 1 ? 0 : (int)(threadIdx.x % T);
  const bool ok = it.ok(0);
  const int base = it.item(0);
  const uint32_t fdig = it.dig(0);
  const int last = g.n_nodes - 1;
  Diag<R> Df{(R)0, (R)0, (R)0};
  for (int i = 0; i < last; ++i) Df = add_diag(Df, load_diag<R, TF>(sm, i * NL + ((fdig >> (4 * i)) & 15)));
  const RowCache<R> rc{};   // not read: the other nodes' rows come from the tables
  C vk[NL];
  const Coef<R, TF> c0 = cf[tau];
#pragma unroll
  for (int q = 0; q < NL; ++q) {
    vk[q] = ok ? A[base + q * T] : mkc((R)0, (R)0);
    acc[q] = coef_mul(c0, vk[q]);
  }
  if (K > 1) {
    C t[NL];
    if (ok) {
      apply_acs<R, NC, TT, RI, false, false, TF>(g, im, sm, A, A, base, fdig, Df, vk, t, rc);
      const Coef<R, TF> c1 = cf[T + tau];
#pragma unroll
      for (int q = 0; q < NL; ++q) {
        vk[q] = mkc((R)0.5 * t[q].x, (R)0.5 * t[q].y);
        B[base + q * T] = vk[q];
        acc[q] = coef_fma(c1, vk[q], acc[q]);
      }
    }
    __syncthreads();
    C *P = A;   // holds y_{k-1}; receives y_{k+1}
    C *Q = B;   // holds y_k (this thread's fiber also in vk)
    for (int k = 2; k < K; ++k) {
      if (ok) {
        const Coef<R, TF> a = cf[k * T + tau];
        if constexpr (RI) keep_in_loop(Df);
        apply_acs<R, NC, TT, RI, false, true, TF>(g, im, sm, Q, P, base, fdig, Df, vk, t, rc);
#pragma unroll
        for (int q = 0; q < NL; ++q) {
          P[base + q * T] = t[q];
          acc[q] = coef_fma(a, t[q], acc[q]);
          vk[q] = t[q];
        }
      }
      __syncthreads();
      C *tmp = P; P = Q; Q = tmp;
    }
  } else {
    __syncthreads();
  }
  apply_phase<R, NL, TF>(g, sm, tau, acc, [&](int q) {
    if constexpr (RI) return Df.lo + acs_kd<R, TF>(im, q).lo;
    else return Df.lo + load_diag<R, TF>(sm, last * NL + q).lo;
  });
}

// --------------------------------------------------------------------------------------
// Block mapping (FP32, tile width 1, real / imaginary cavity structure on the middle and the last node): a
// thread owns NP fibers, the photon numbers 0..NC of the middle node at a fixed state of its atom.  What bounds
// the series is the shared-memory pipe: one fiber per thread executes 10.3 loads and stores per element and term
// at d = 6561 (6 neighbours needed, the rest lanes that a branch leaves idle) and twelve table lookups
// and branches per fiber, with 23 warps of 80 registers to hide them.  Here a neighbour's block serves the
// hops onto the middle and onto the last node at once, a hop between those two stays in registers, and every
// offset and coefficient is shared by 27 elements, with 8 warps of 255 registers whose 27 independent
// rows cover the latency.  1024 trajectories of d = 6561, per interval: forward with update 370 -> 345 us, backward 313 -> 294 us.
template <typename R, int NP>
struct BlkCache {
  int off0[2], off1[2];   // outer nodes: element offsets of the two slots (0 = none)
  R a[2], b[2];           // and their coefficients (imaginary, real)
  int moff0[NP], moff1;   // middle node: cavity offset per photon number, drive offset
  R ma[NP], mb[NP];
  int hoff[2];            // hops between the outer nodes
  R hop[2];
  R up[2], dn[2];         // sqrt(n_i + 1) (0: cutoff reached), sqrt(n_i) of the outer nodes
};

template <typename R, int NC>
__device__ __forceinline__ void load_blk(const KtGeom &g, const KtGenImage &im, const Smem &sm, uint32_t fdig,
                                         BlkCache<R, NC + 1> &rc) {
  typedef typename C2<R>::T C;
  constexpr int NP = NC + 1, NL = 3 * NP;
  const C *lv = (const C *)sm.loc_val;
  const int outer = g.n_nodes - 2;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    rc.off0[i] = rc.off1[i] = 0;
    rc.a[i] = rc.b[i] = rc.up[i] = rc.dn[i] = (R)0;
    rc.hoff[i] = 0;
    rc.hop[i] = (R)0;
    if (i < outer) {
      const int x = (fdig >> (4 * i)) & 15, e0 = (i * NL + x) * 2;
      rc.off0[i] = sm.loc_off[e0];
      rc.off1[i] = sm.loc_off[e0 + 1];
      rc.a[i] = lv[e0].y;
      rc.b[i] = lv[e0 + 1].x;
      rc.up[i] = x % NP < NC ? sqrt_n<R>(x % NP + 1) : (R)0;
      rc.dn[i] = sqrt_n<R>(x % NP);
    }
  }
  const int xm = (fdig >> (4 * outer)) & 15;
#pragma unroll
  for (int n = 0; n < NP; ++n) {
    const int e0 = (outer * NL + xm + n) * 2;
    rc.moff0[n] = sm.loc_off[e0];
    rc.ma[n] = lv[e0].y;
    rc.mb[n] = lv[e0 + 1].x;
  }
  rc.moff1 = sm.loc_off[(outer * NL + xm) * 2 + 1];
  int h = 0;
  for (int p = 0; p < g.n_pairs && outer == 2; ++p) {
    const int pd = im.pair_dst[p], ps = im.pair_src[p];
    if (pd >= outer || ps >= outer) continue;
    const int e = p * NL * NL + ((fdig >> (4 * pd)) & 15) * NL + ((fdig >> (4 * ps)) & 15);
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (i == h) {
        rc.hoff[i] = sm.pair_off[e];
        rc.hop[i] = ((const C *)sm.pair_val)[e].x;
      }
    ++h;
  }
}

// out[q] = prev[base + q] + (B v)[base + q] for the thread's block, as apply_acs.  Every element's terms come in the order of
// the fiber mapping (for the hops as long as a pair of nodes hops one way only, as a cascade does), with its coefficients.
template <typename R, int NC, bool TF>
__device__ __forceinline__ void apply_blk(const KtGeom &g, const KtGenImage &im, const Smem &sm,
                                          const typename C2<R>::T *__restrict__ v, const typename C2<R>::T *prev,
                                          int base, const Diag<R> (&Df)[NC + 1],
                                          const typename C2<R>::T (&vk)[3 * (NC + 1) * (NC + 1)],
                                          typename C2<R>::T (&out)[3 * (NC + 1) * (NC + 1)],
                                          const BlkCache<R, NC + 1> &rc) {
  typedef typename C2<R>::T C;
  constexpr int NP = NC + 1, NL = 3 * NP, E = NP * NL;
  const C *ld = (const C *)sm.ldense;
  const C zero = mkc((R)0, (R)0);
#pragma unroll
  for (int q = 0; q < E; ++q) out[q] = diag_init<TF>(add_diag(Df[q / NL], acs_kd<R, TF>(im, q % NL)), vk[q], zero);
  // last node
#pragma unroll
  for (int m = 0; m < NP; ++m) {
#pragma unroll
    for (int n = 1; n <= NC; ++n) {
      const int qr = m * NL + 2 * NP + n - 1, qg = m * NL + n;
      out[qr] = add_im<TF>(acs_kc<R>(im)[n - 1], vk[qg], out[qr]);
      out[qg] = add_im<TF>(acs_kc<R>(im)[NC + n - 1], vk[qr], out[qg]);
    }
#pragma unroll
    for (int n = 0; n <= NC; ++n) {
      const int r = 2 * NP + n, e = NP + n;
      out[m * NL + r] = add_re<TF>(ld[r * NL + e].x, vk[m * NL + e], out[m * NL + r]);
      out[m * NL + e] = add_re<TF>(ld[e * NL + r].x, vk[m * NL + r], out[m * NL + e]);
    }
  }
  // outer nodes' rows
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    if (rc.off0[i]) {
#pragma unroll
      for (int q = 0; q < E; ++q) out[q] = add_im<TF>(rc.a[i], v[base + rc.off0[i] + q], out[q]);
    }
    if (rc.off1[i]) {
#pragma unroll
      for (int q = 0; q < E; ++q) out[q] = add_re<TF>(rc.b[i], v[base + rc.off1[i] + q], out[q]);
    }
  }
  // middle node's rows
#pragma unroll
  for (int m = 0; m < NP; ++m)
    if (rc.moff0[m]) {
#pragma unroll
      for (int q = 0; q < NL; ++q) out[m * NL + q] = add_im<TF>(rc.ma[m], v[base + rc.moff0[m] + m * NL + q], out[m * NL + q]);
    }
  if (rc.moff1) {
#pragma unroll
    for (int q = 0; q < E; ++q) out[q] = add_re<TF>(rc.mb[q / NL], v[base + rc.moff1 + q], out[q]);
  }
  // hops between the outer nodes
#pragma unroll
  for (int i = 0; i < 2; ++i)
    if (rc.hoff[i]) {
#pragma unroll
      for (int q = 0; q < E; ++q) out[q] = add_re<TF>(rc.hop[i], v[base + rc.hoff[i] + q], out[q]);
    }
  // hops between an outer node and the middle and the last one
#pragma unroll
  for (int i = 0; i < 2; ++i)
    if (i < g.n_nodes - 2) {
      const int s = g.stride[i];
      // middle or last node raised, node i lowered: the block with one photon more in node i
      if (rc.up[i] != (R)0 && (im.kh[0][i] != 0.f || im.kh[1][i] != 0.f)) {
        const bool two = rc.up[i] > (R)1;
        const R cm1 = two ? im.km[0][i][1] : im.km[0][i][0], cm2 = two ? im.km[0][i][2] : im.km[0][i][1];
        const R cl = (R)im.kh[1][i] * rc.up[i];
#pragma unroll
        for (int m = 0; m < NP; ++m)
#pragma unroll
          for (int q = 0; q < NL; ++q) {
            if (m == NC && q % NP == NC) continue;
            const C w = v[base + s + m * NL + q];
            if (m < NC) out[(m + 1) * NL + q] = add_re<TF>(m == 1 ? cm2 : cm1, w, out[(m + 1) * NL + q]);
            if (q % NP < NC) out[m * NL + q + 1] = add_re<TF>(cl * sqrt_n<R>(q % NP + 1), w, out[m * NL + q + 1]);
          }
      }
      // node i raised, middle or last node lowered
      if (rc.dn[i] != (R)0 && (im.kh[2][i] != 0.f || im.kh[3][i] != 0.f)) {
        const bool two = rc.dn[i] > (R)1;
        const R cm1 = two ? im.km[1][i][1] : im.km[1][i][0], cm2 = two ? im.km[1][i][2] : im.km[1][i][1];
        const R cl = (R)im.kh[3][i] * rc.dn[i];
#pragma unroll
        for (int m = NC; m >= 0; --m)
#pragma unroll
          for (int q = 0; q < NL; ++q) {
            if (m == 0 && q % NP == 0) continue;
            const C w = v[base - s + m * NL + q];
            if (m >= 1) out[(m - 1) * NL + q] = add_re<TF>(m == 2 ? cm2 : cm1, w, out[(m - 1) * NL + q]);
            if (q % NP >= 1) out[m * NL + q - 1] = add_re<TF>(cl * sqrt_n<R>(q % NP), w, out[m * NL + q - 1]);
          }
      }
    }
  // hops between the middle and the last node
  {
    const R cl = (R)im.kh[4][0], cm = (R)im.kh[4][1];
    if (cl != (R)0) {
#pragma unroll
      for (int m = 0; m < NC; ++m)
#pragma unroll
        for (int q = 0; q < NL; ++q)
          if (q % NP >= 1)
            out[m * NL + q] = add_re<TF>((cl * sqrt_n<R>(m + 1)) * sqrt_n<R>(q % NP), vk[(m + 1) * NL + q - 1], out[m * NL + q]);
    }
    if (cm != (R)0) {
#pragma unroll
      for (int m = 1; m <= NC; ++m)
#pragma unroll
        for (int q = 0; q < NL; ++q)
          if (q % NP < NC)
            out[m * NL + q] = add_re<TF>((cm * sqrt_n<R>(m)) * sqrt_n<R>(q % NP + 1), vk[(m - 1) * NL + q + 1], out[m * NL + q]);
    }
  }
#pragma unroll
  for (int q = 0; q < E; ++q)
    out[q] = diag_done<TF>(add_diag(Df[q / NL], acs_kd<R, TF>(im, q % NL)), vk[q], prev[base + q], out[q]);
}

template <typename R, int NC, bool TF, class IT>
__device__ void cheb_run_blk(const KtGeom &g, const KtGenImage &im, const Smem &sm, const IT &it, int K,
                             typename C2<R>::T (&acc)[3 * (NC + 1) * (NC + 1)]) {
  typedef typename C2<R>::T C;
  constexpr int NP = NC + 1, NL = 3 * NP, E = NP * NL;
  C *P = (C *)sm.bufB;   // holds y_{k-1}; receives y_{k+1}
  C *Q = (C *)sm.bufA;   // holds y_k (this thread's block also in vk)
  const Coef<R, TF> *cf = (const Coef<R, TF> *)sm.coef;
  const bool ok = it.ok(0);
  const int base = it.item(0), outer = g.n_nodes - 2;
  const uint32_t fdig = it.dig(0);
  Diag<R> Df[NP];
  BlkCache<R, NP> rc;
  C vk[E], out[E];
  const Coef<R, TF> c0 = cf[0];
  if (ok) {
    load_blk<R, NC>(g, im, sm, fdig, rc);
    Diag<R> D{(R)0, (R)0, (R)0};
    for (int i = 0; i < outer; ++i) D = add_diag(D, load_diag<R, TF>(sm, i * NL + ((fdig >> (4 * i)) & 15)));
#pragma unroll
    for (int m = 0; m < NP; ++m) Df[m] = add_diag(D, load_diag<R, TF>(sm, outer * NL + ((fdig >> (4 * outer)) & 15) + m));
  }
#pragma unroll
  for (int q = 0; q < E; ++q) {
    vk[q] = ok ? Q[base + q] : mkc((R)0, (R)0);
    acc[q] = coef_mul(c0, vk[q]);
  }
  for (int k = 1; k < K; ++k) {
    if (ok) {
      // y_1 = B y_0 / 2: the first round finds zeros for y_{-1} and halves the result
      if (k == 1) {
#pragma unroll
        for (int q = 0; q < E; ++q) P[base + q] = mkc((R)0, (R)0);
      }
      apply_blk<R, NC, TF>(g, im, sm, Q, P, base, Df, vk, out, rc);
      const Coef<R, TF> a = cf[k];
      const R h = k == 1 ? (R)0.5 : (R)1;
#pragma unroll
      for (int q = 0; q < E; ++q) {
        vk[q] = mkc(h * out[q].x, h * out[q].y);
        P[base + q] = vk[q];
        acc[q] = coef_fma(a, vk[q], acc[q]);
      }
    }
    __syncthreads();
    C *tmp = P; P = Q; Q = tmp;
  }
  if (K == 1) __syncthreads();
  apply_phase<R, E, TF>(g, sm, 0, acc, [&](int q) { return Df[q / NL].lo + acs_kd<R, TF>(im, q % NL).lo; });
}

// --------------------------------------------------------------------------------------
// Row mapping: one element per thread, its row of B in registers (real / imaginary coupling classes, at most NN
// nodes with two slots each and NPR pair terms).  Small problems are bound by the latency of a term, not by
// any pipe: the table-driven apply_item walks 2 N + P dependent table lookups and branches per
// term, 0.55 us at d = 81 with one trajectory per CTA; with offsets and coefficients in registers a term is 2 N + P
// independent loads, two FMAs each, and a barrier.  y_{k-1} and y_k of the thread's own element stay in
// registers too.  Measured per interval, forward with update / backward, against the
// mapping of one item or one fiber per thread with tables: d = 81, 128 trajectories 25.8 / 11.2 -> 12.2 / 5.8 us (FP32), 51 /
// 48 -> 32 / 25 us (FP64); d = 81, 1024 trajectories 66 / 14.7 -> 51 / 7.7 us (FP32), 219 / 163 -> 132 / 122 us (FP64);
// d = 144, 100 trajectories 64 / 50 -> 12.8 / 6.2 us; d = 216, 333 trajectories 37 / 27 -> 20 / 9.2 us.  At d = 729 a
// thread per element executes 85 instructions per term where a fiber shares them among nine (1024 trajectories: 64
// against 49 us backward), so the fiber mapping stays there.
template <typename R, int NN, int NPR>
struct RowRegs {
  int off[2 * NN + NPR];
  R w[2 * NN + NPR];
};

template <typename R, int NN, int NPR>
__device__ __forceinline__ void load_row(const KtGeom &g, const KtGenImage &im, const Smem &sm, uint32_t dig,
                                         RowRegs<R, NN, NPR> &r) {
  typedef typename C2<R>::T C;
  const C *lv = (const C *)sm.loc_val;
#pragma unroll
  for (int i = 0; i < NN; ++i) {
    r.off[2 * i] = r.off[2 * i + 1] = 0;
    r.w[2 * i] = r.w[2 * i + 1] = (R)0;
    if (i < g.n_nodes) {
      const int e0 = (i * g.n_loc + ((dig >> (4 * i)) & 15)) * 2;
      r.off[2 * i] = sm.loc_off[e0];
      r.w[2 * i] = lv[e0].y;              // slot 0: real in G, imaginary in B
      r.off[2 * i + 1] = sm.loc_off[e0 + 1];
      r.w[2 * i + 1] = lv[e0 + 1].x;      // slot 1: imaginary in G, real in B
    }
  }
#pragma unroll
  for (int p = 0; p < NPR; ++p) {
    r.off[2 * NN + p] = 0;
    r.w[2 * NN + p] = (R)0;
    if (p < g.n_pairs) {
      const int xd = (dig >> (4 * im.pair_dst[p])) & 15, xs = (dig >> (4 * im.pair_src[p])) & 15;
      const int e = (p * g.n_loc + xd) * g.n_loc + xs;
      r.off[2 * NN + p] = sm.pair_off[e];
      r.w[2 * NN + p] = ((const C *)sm.pair_val)[e].x;
    }
  }
}

// v = base[off] where off != 0, else 0, without a branch: all of a row's loads are in flight before the first is
// used (behind branches they wait for one another), and lanes
// without an entry cause no bank conflicts.  Volatile: ordered with the barriers around it.
__device__ __forceinline__ float2 ld_if(const float2 *base, int off) {
  float2 v;
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %3, 0;\n\tmov.f32 %0, 0f00000000;\n\tmov.f32 %1, 0f00000000;\n\t"
               "@p ld.shared.v2.f32 {%0, %1}, [%2];\n\t}"
               : "=&f"(v.x), "=&f"(v.y) : "r"(smem_u32(base + off)), "r"(off) : "memory");
  return v;
}
__device__ __forceinline__ double2 ld_if(const double2 *base, int off) {
  double2 v;
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %3, 0;\n\tmov.f64 %0, 0d0000000000000000;\n\t"
               "mov.f64 %1, 0d0000000000000000;\n\t@p ld.shared.v2.f64 {%0, %1}, [%2];\n\t}"
               : "=&d"(v.x), "=&d"(v.y) : "r"(smem_u32(base + off)), "r"(off) : "memory");
  return v;
}

template <typename R, int NN, int NPR, class IT>
__device__ void cheb_run_row(const KtGeom &g, const KtGenImage &im, const Smem &sm, const IT &it, int K,
                             typename C2<R>::T (&acc)[1]) {
  typedef typename C2<R>::T C;
  C *P = (C *)sm.bufB, *Q = (C *)sm.bufA;
  const R *cf = (const R *)sm.coef;
  const int tau = threadIdx.x % g.T, item = it.item(0);
  const bool ok = it.ok(0);
  RowRegs<R, NN, NPR> r;
  Diag<R> D{(R)0, (R)0, (R)0};
  C cur = mkc((R)0, (R)0), prev = cur;
  if (ok) {
    load_row<R, NN, NPR>(g, im, sm, it.dig(0), r);
    D = diag_of<R>(g, sm, it.dig(0));
    cur = Q[item];
  }
  if (!ok) {
#pragma unroll
    for (int e = 0; e < 2 * NN + NPR; ++e) r.off[e] = 0;
  }
  unsigned any = 0;
  if (sizeof(R) == 8 && NN >= 3) {
#pragma unroll
    for (int e = 0; e < 2 * NN + NPR; ++e) any |= (__any_sync(0xffffffffu, r.off[e] != 0) ? 1u : 0u) << e;
  }
  const R c0 = cf[tau];
  acc[0] = mkc(c0 * cur.x, c0 * cur.y);
  R a = K > 1 ? cf[g.T + tau] : (R)0;
  C s = diag_init(D, cur, prev);   // of the next term: formed before the barrier, from the thread's own values
  for (int k = 1; k < K; ++k) {
    if (ok) {
      C v[2 * NN + NPR];
#pragma unroll
      for (int e = 0; e < 2 * NN + NPR; ++e) v[e] = ld_if(Q + item, r.off[e]);
      if constexpr (sizeof(R) == 4) {
        C z = mkc((R)0, (R)0);   // two chains, for latency
#pragma unroll
        for (int e = 0; e < 2 * NN; e += 2) {
          s = ifma(r.w[e], v[e], s);
          z = rfma(r.w[e + 1], v[e + 1], z);
        }
#pragma unroll
        for (int e = 2 * NN; e < 2 * NN + NPR; ++e) z = rfma(r.w[e], v[e], z);
        s.x += z.x;
        s.y += z.y;
      } else {
        // FP64: an FMA takes a warp 64 cycles of its scheduler's share of the FP64 unit, so the count decides; with three
        // nodes most warps have slots that no lane needs
#pragma unroll
        for (int e = 0; e < 2 * NN + NPR; ++e)
          if (NN < 3 || (any >> e & 1)) s = (e < 2 * NN && e % 2 == 0) ? ifma(r.w[e], v[e], s) : rfma(r.w[e], v[e], s);
      }
      s = diag_done(D, cur, prev, s);
      if (k == 1) s = mkc((R)0.5 * s.x, (R)0.5 * s.y);
      P[item] = s;
      prev = cur;
      cur = s;
      acc[0] = rfma(a, cur, acc[0]);
      s = diag_init(D, cur, prev);
    }
    a = k + 1 < K ? cf[(k + 1) * g.T + tau] : (R)0;
    __syncthreads();
    C *tmp = P; P = Q; Q = tmp;
  }
  if (K == 1) __syncthreads();
  apply_phase<R, 1>(g, sm, tau, acc, [&](int) { return D.lo; });
}

template <typename R, int EPT, int NL, int ACS, class IT>
__device__ __forceinline__ void cheb_dispatch(const KtGeom &g, const KtGenImage &im, const Smem &sm,
                                              const IT &it, int K, typename C2<R>::T (&acc)[EPT]) {
  // ACS: 1 cavity structure, 2 the same with T = 1, 3 with real / imaginary couplings, 4 both
  // 5 block mapping; 6, 7 row mapping (up to two nodes and one pair, three nodes and three pairs); 11, 12, 13: 3, 4, 5 in the y form
  constexpr int A = ACS >= 8 ? ACS - 8 : ACS;
  constexpr bool TF = t_form<R, NL, ACS>();
  if constexpr (A == 6) cheb_run_row<R, 2, 1>(g, im, sm, it, K, acc);
  else if constexpr (A == 7) cheb_run_row<R, 3, 3>(g, im, sm, it, K, acc);
  else if constexpr (A == 5) cheb_run_blk<R, NL / 3 - 1, TF>(g, im, sm, it, K, acc);
  else if constexpr (A) cheb_run_acs<R, NL / 3 - 1, (A == 2 || A == 4) ? 1 : 0, (A >= 3), TF>(g, im, sm, it, K, acc);
  else if constexpr (NL > 0) cheb_run_fiber<R, NL, TF>(g, im, sm, it, K, acc);
  else cheb_run<R, EPT>(g, im, sm, it, K, acc);
}

// End of a tile in the forward kernel looping over tiles: the generic-proxy writes of the tile are
// ordered before the bulk copies that will overwrite its buffers, then the prefetched psi (fourth
// buffer) becomes the next tile's input and the old input buffer (maybe still being stored) the next
// prefetch target.
__device__ __forceinline__ void end_fwd_tile(Smem &sm, bool persist) {
  if (!persist) return;
  fence_proxy_async_smem();
  __syncthreads();
  void *t = sm.bufA;
  sm.bufA = sm.bufD;
  sm.bufD = t;
}

// CTAs per SM that the register allocation leaves room for: FP32 fibers in small CTAs at 80 registers (with 104,
// 18 warps instead of 24 per SM: 71 instead of 54 us per backward interval at d = 729, 1024 trajectories); one row
// per thread at 80 (small CTAs) or 40.
__host__ __device__ constexpr int kt_min_ctas(int rsize, int ept, int nl, int maxt) {
  if (rsize != 4) return nl == 0 && ept == 1 && maxt == 256 ? 2 : 1;
  if (nl > 0 && ept == nl && maxt == 256) return 3;
  if (nl == 0 && ept == 1 && maxt == 256) return 3;
  return nl == 0 && ept == 1 && maxt == 768 ? 2 : 1;
}

// --------------------------------------------------------------------------------------
// Forward interval kernel.  One Chebyshev call site serves every phase:
//   MAIN    full interval from psi(t_{j-1}) (uniform coefficients),
//   ROOT    Newton's method for n(s) = ||exp(-i G s) start||^2 = r of the flagged trajectories,
//   SSTAR   the state at the located jump time s*, then collapse (Sec. 2.1, steps 3-5),
//   REST    the remainder of the interval from the collapsed state, tested again.
// The jump time: the norm falls at the loss rate, dn/ds = -p(s), p = sum_l ||L_l psi(s)||^2, so each trial
// series gives value and slope.  The first trial is the root of the cubic through (n, p) at both ends of
// the piece, whose error is of order dt^4; a step is taken as the answer once its own error, curvature times
// its square, is below tol, and a step that leaves the bracket is replaced by the bracket's middle.  The state at the
// time taken, which the collapse needs anyway, has to have the norm r; else the search goes on from there.  One or two
// series where the bisection to 2^-48 dt (2^-40 in FP32) took 48 (40): a Krotov pass over d = 81 with 128 trajectories
// of several jumps each in FP64 fell from 201 to 24 ms, 100 intervals of d = 729 with 3 % of 1024 trajectories
// jumping from 82 to 27 ms.
enum { PH_MAIN = 0, PH_ROOT, PH_SSTAR, PH_REST, PH_DONE };

// This thread's part of its trajectory's norm^2: summed over a fiber (at most 16 elements) in the state precision, over a
// block's fibers in FP64.
template <typename R, int EPT, int NL, class IT>
__device__ __forceinline__ double norm_part(const IT &it, const typename C2<R>::T (&v)[EPT]) {
  constexpr int FB = NL > 0 ? NL : EPT;
  double n = 0.0;
#pragma unroll
  for (int f = 0; f < EPT; f += FB) {
    R s = 0;
#pragma unroll
    for (int q = f; q < f + FB; ++q)
      if (it.ok(q)) s += v[q].x * v[q].x + v[q].y * v[q].y;
    n = f == 0 ? (double)s : n + (double)s;
  }
  return n;
}
template <typename R, bool WIDE> struct SumT { typedef R T; };
template <typename R> struct SumT<R, true> { typedef double T; };

// Root of the cubic Hermite interpolant of a decreasing n on [0, len] with n(0) = n0 >= r >= n(len) = n1
// and slopes -p0, -p1.
__device__ __forceinline__ double hermite_root(double n0, double n1, double p0, double p1, double len, double r) {
  const double D = n0 - n1;
  if (!(D > 0.0) || !(len > 0.0)) return 0.5 * len;
  const double m0 = p0 * len / D, m1 = p1 * len / D, y = (n0 - r) / D;   // fall h(u) = (n0 - n) / D from 0 to 1
  double u = y;
  for (int i = 0; i < 4; ++i) {
    // h(u) = m0 u + (3 - 2 m0 - m1) u^2 + (m0 + m1 - 2) u^3
    const double c2 = 3.0 - 2.0 * m0 - m1, c3 = m0 + m1 - 2.0;
    const double f = ((c3 * u + c2) * u + m0) * u - y, df = (3.0 * c3 * u + 2.0 * c2) * u + m0;
    if (!(df > 0.0)) break;
    u -= f / df;
    u = u < 0.0 ? 0.0 : (u > 1.0 ? 1.0 : u);
  }
  return u * len;
}

template <typename R, int EPT, int NL, int ACS, bool SWEEP, int MAXT>
__global__ void __launch_bounds__(MAXT, kt_min_ctas(sizeof(R), EPT, NL, MAXT)) fwd_kernel(KtGeom g, KtGenImage im, KtOps ops, FwdArgs a) {
  typedef typename C2<R>::T C;
  extern __shared__ __align__(16) char smem_raw[];
  Smem sm;
  // with g.fwd_grid > 0 the CTAs loop over tiles blockIdx.x, blockIdx.x + gridDim.x, ...: the tables and
  // the item mapping are built once, and the next tile's psi (fourth buffer, barriers [0] / [3] in turn)
  // and chi (third buffer) arrive by bulk copy while the current tile is propagated.
  // SWEEP (a.sweep): one launch runs intervals a.j .. nt of one tile per CTA (see FwdArgs);
  // a compile-time switch, so that the per-interval kernels carry none of the sweep's state.
  constexpr bool sweep = SWEEP;
  const bool persist = !sweep && g.fwd_grid > 0;
  char *const extra = smem_raw + carve(g, sizeof(C), smem_raw, &sm, g.prefetch_chi != 0, persist);
  const int tau = threadIdx.x % g.T;
  // error allowed to the jump time: 2^-50 dt in FP64 (near the rounding of the FP64 norm that decides it),
  // 2^-32 dt in FP32-mixed (the FP32 norm's rounding, 2^-24 and more over a loss of 1e-3 ... 1e-2 per interval, leaves
  // the time uncertain by 1e-5 dt: steps do not get smaller than that, and 2^-40 dt was not reached in 60 trials)
  const double tol = (sizeof(R) == 8 ? 0x1p-50 : 0x1p-32) * g.dt;
  int j = a.j;

  if (threadIdx.x < g.n_ctrl) {
    const int c = threadIdx.x;
    double e = 0.0;
    if (j >= 1) {
      e = a.eps_old[c * a.nt + (j - 1)];
      if (a.update) e += a.deps[c * a.nt + (j - 1)];
    }
    sm.eps[c] = e;
  }
  if (threadIdx.x < 8) sm.flag[threadIdx.x] = 0;
  if (threadIdx.x == 0) {
    mbar_init(&sm.mbar[0], 1);
    mbar_init(&sm.mbar[1], 1);
    mbar_init(&sm.mbar[2], 1);
    mbar_init(&sm.mbar[3], 1);
    fence_mbar_init();
  }
  __syncthreads();
  const uint32_t tile_bytes = (uint32_t)(g.tile_elems * sizeof(C));
  // co-states chi(t_i) of interval i's update overlap
  auto chi_of = [&](int i, int t) -> const C * {
    const C *base = sweep ? (const C *)((const char *)a.chi_slots + (size_t)i * a.slot_bytes) : (const C *)a.chi_t;
    return base + (size_t)t * g.tile_elems;
  };
  // the bulk engine brings psi(t_{j-1}) (and chi(t_j) when there is room) while the tables are built
  if (threadIdx.x == 0) {
    bulk_load(sm.bufA, (const C *)a.psi_in + (size_t)blockIdx.x * g.tile_elems, tile_bytes, &sm.mbar[0]);
    if (a.overlap && j < a.nt && g.prefetch_chi) bulk_load(sm.bufC, chi_of(j, blockIdx.x), tile_bytes, &sm.mbar[1]);
  }
  build_tables<R>(g, im, ops, sm, sm.eps, a.overlap != 0);
  Items<EPT, NL> it;
  load_items<EPT, NL>(g, ops, it);
  SweepKeep keep;
  if constexpr (SWEEP) sweep_keep_init<R>(g, im, extra, keep);
  bool store_pending = false;
  unsigned nchi = 0;        // chi loads waited for on barrier [1] (the n-th completes phase n & 1)
  C acc[EPT];
  double eps_ahead = 0.0;   // guess sweep: the next interval's pulse, read an interval ahead
  for (;; ++j) {            // intervals: one unless sweep
    const bool need_chi = a.overlap && j < a.nt;
    // sweep: the update's pulse-independent factors for the finisher, read now, off its critical path
    // (the per-interval kernels read them in the finisher: registers held across the tiles spill there)
    const double eps_next = eps_ahead;
    if (sweep && !a.update && j < a.nt && threadIdx.x < g.n_ctrl) eps_ahead = a.eps_old[threadIdx.x * a.nt + j];
    double fin_scale = 0.0, fin_eold = 0.0;
    if (sweep && need_chi && threadIdx.x < g.n_ctrl) {
      const size_t idx = (size_t)threadIdx.x * a.nt + j;   // interval j+1 (0-based index j)
      fin_scale = a.shape[idx] / (g.lam[threadIdx.x] * g.M_norm);
      fin_eold = a.eps_old[idx];
    }
    if (j != a.j) {
      // sweep: the next interval.  Its pulse is in sm.eps (guess sweep: eps_old; updating: the value
      // the exchange's finisher formed), its chi goes to the third buffer once every thread is done
      // with the previous one, and the tables are rebuilt for the new pulse.
      if (!a.update && threadIdx.x < g.n_ctrl) sm.eps[threadIdx.x] = eps_next;
      fence_proxy_async_smem();
      __syncthreads();
      if (threadIdx.x == 0 && need_chi && g.prefetch_chi)
        bulk_load(sm.bufC, chi_of(j, blockIdx.x), tile_bytes, &sm.mbar[1]);
      if constexpr (SWEEP) sweep_tables<R>(g, im, ops, sm, keep);
    }
    int tile = blockIdx.x;
    for (int use = 0; tile < g.n_tiles; tile += gridDim.x, ++use) {
      const int next = tile + (int)gridDim.x;
      const C *psi_in = (const C *)((!sweep || j <= 1) ? a.psi_in : a.psi_ring[(j - 1) & 1]) + (size_t)tile * g.tile_elems;
      C *psi_out = (C *)(sweep ? a.psi_ring[j & 1] : a.psi_out) + (size_t)tile * g.tile_elems;
      const C *chi_g = need_chi ? chi_of(j, tile) : nullptr;
      // the trajectory's current threshold, read now so that its latency is off the path after the series
      const double r_start = (threadIdx.x < g.T) ? a.rstate[(size_t)tile * g.T + threadIdx.x] : 0.0;
      if (threadIdx.x == 0) {
        sm.flag[0] = 0;
        sm.flag[1] = 0;
        sm.flag[2] = 0;
      }
      C *A = (C *)sm.bufA;
      C *B = (C *)sm.bufB;
      if (sweep && j != a.j) {
        // sweep: psi(t_{j-1}) is the previous interval's result, still in registers
    #pragma unroll
        for (int q = 0; q < EPT; ++q)
          if (it.ok(q)) A[it.item(q)] = acc[q];   // synchronised before the series
      } else if (!tile_wait((use & 1) ? &sm.mbar[3] : &sm.mbar[0], (use >> 1) & 1, &sm.flag[4], a.status,
                            g.inject_timeout ? &sm.mbar[2] : nullptr)) {
        // psi of this tile: load number `use`, barrier [0] / [3] in turn, phase parity (use >> 1) & 1
        if (threadIdx.x == 0) {
          if (need_chi && g.prefetch_chi) mbar_wait_bounded(&sm.mbar[1], nchi & 1);
          if (store_pending) bulk_store_wait();
        }
        return;
      }
      if (persist && next < g.n_tiles) {
        // the fourth buffer fed the previous tile's bulk store: let that finish, then prefetch into it
        if (threadIdx.x == 0) {
          if (store_pending) bulk_store_wait();
          bulk_load(sm.bufD, (const C *)a.psi_in + (size_t)next * g.tile_elems, tile_bytes,
                    (use & 1) ? &sm.mbar[0] : &sm.mbar[3]);
        }
        store_pending = false;
      }
      bool jumped = false, stored = false;

      // |L_l v|^2 at this thread's elements of tile vector v, summed over a fiber in the state precision (norm_part)
      // (the jump phases' loops stay rolled where an element's place is arithmetic: they are rare, and unrolled they
      // cost the series registers)
      constexpr int UJ = NL > 0 ? 1 : EPT;
      auto channel = [&](int l, const C *v) -> double {
        double n = 0.0;
        R s = 0;
    #pragma unroll UJ
        for (int q = 0; q < EPT; ++q) {
          if (it.ok(q)) {
            const C y = lind_item<R>(g, ops, l, 0, v, it.item(q), it.dig(q));
            s += y.x * y.x + y.y * y.y;
          }
          if (NL > 0 && EPT > NL && q % (NL > 0 ? NL : 1) == NL - 1) {
            n += (double)s;
            s = 0;
          }
        }
        return NL > 0 && EPT > NL ? n : (double)s;
      };
      auto loss = [&](const C *v) -> double {
        double p = 0.0;
        for (int l = 0; l < g.n_lind; ++l) p += channel(l, v);
        return p;
      };
      // One step of the root search of trajectory t from n - r = f and the loss rate p at the trial time TS_S, kept inside
      // the bracket: the next trial, or (TI_BUSY 0) the time taken, in TS_S.
      auto newton = [&](int t, double f, double p) {
        const double s0 = sm.tsc[TS_S * g.T + t], ps = sm.tsc[TS_PS * g.T + t], pp = sm.tsc[TS_PP * g.T + t];
        double lo = sm.tsc[TS_LO * g.T + t], hi = sm.tsc[TS_HI * g.T + t];
        if (f <= 0.0) hi = s0;
        else lo = s0;
        const double step = f / p, next = s0 + step, mid = 0.5 * (lo + hi);
        const int tries = sm.tin[TI_CH * g.T + t] + 1;
        const bool in = p > 0.0 && next >= lo && next <= hi;
        // what Newton's step leaves: |n'' / (2 n')| step^2, n'' from the two latest slopes
        const double left = fabs((p - pp) / (s0 - ps)) * step * step / p;
        const bool small = in && (left <= tol || fabs(step) <= tol), spent = hi - lo <= tol || tries >= 60;
        sm.tsc[TS_LO * g.T + t] = lo;
        sm.tsc[TS_HI * g.T + t] = hi;
        sm.tsc[TS_PS * g.T + t] = s0;
        sm.tsc[TS_PP * g.T + t] = p;
        sm.tsc[TS_S * g.T + t] = in ? next : (spent ? hi : mid);
        sm.tin[TI_BUSY * g.T + t] = !small && !spent;
        sm.tin[TI_CH * g.T + t] = spent ? 60 : tries;    // 60: nothing left to try
      };
      int phase = (j >= 1) ? PH_MAIN : PH_DONE;
      if (phase == PH_DONE) {
    #pragma unroll
        for (int q = 0; q < EPT; ++q) acc[q] = it.ok(q) ? A[it.item(q)] : mkc((R)0, (R)0);
      }
      int guard = 0;
      bool chi_here = false, chi_failed = false;
      int vstride = 8, voff = 1;
      for (;;) {
        if (phase != PH_DONE) {
          Smem run = sm;
          // ---- choose the propagation of this round
          if (phase == PH_ROOT) {
            if (threadIdx.x == 0) sm.flag[1] = 0;
            __syncthreads();
            if (threadIdx.x < g.T && sm.tin[TI_ACT * g.T + threadIdx.x] && sm.tin[TI_BUSY * g.T + threadIdx.x])
              atomicAdd(&sm.flag[1], 1);
            __syncthreads();
            if (sm.flag[1] == 0) phase = PH_SSTAR;
          }
          if (phase == PH_MAIN) {
            if constexpr (SWEEP) sweep_coefs<R>(g, im, sm, run, keep, extra, j);
            else uniform_coefs<R, t_form<R, NL, ACS>()>(g, sm, im, j);
          } else {
            if (threadIdx.x < g.T) {
              const int t = threadIdx.x;
              const bool act = sm.tin[TI_ACT * g.T + t] != 0;
              double len = 0.0;
              if (phase == PH_ROOT) len = act && sm.tin[TI_BUSY * g.T + t] ? sm.tsc[TS_S * g.T + t] : 0.0;
              else if (phase == PH_SSTAR) len = act ? sm.tsc[TS_S * g.T + t] : 0.0;
              else len = act ? g.dt - sm.tsc[TS_S0 * g.T + t] : 0.0;
              sm.tsc[TS_X * g.T + t] = len;
            }
            load_tile<R, EPT>(g, it, psi_out, A);   // the main round's tile came by bulk copy
            __syncthreads();
            piece_coefs<R, t_form<R, NL, ACS>()>(g, im, sm, g.c_fwd);
          }
          __syncthreads();
          cheb_dispatch<R, EPT, NL, ACS>(g, im, run, it, g.K, acc);
        }
        if (phase == PH_MAIN || phase == PH_DONE) {
          // ---- norm of the result and update overlap at t_j, g_c = sum_k Im <chi_k|hc_c|psi_k>, in one reduction.
          // After the main round the overlap is formed on the chance that no trajectory jumps (it then is the
          // final one), when chi(t_j) has a buffer of its own.
          if (phase == PH_MAIN || jumped) {
    #pragma unroll
            for (int q = 0; q < EPT; ++q)
              if (it.ok(q)) A[it.item(q)] = acc[q];
          }
          fence_proxy_async_smem();      // A is stored by the bulk engine, B may be loaded by it
          const bool sum = need_chi && (phase == PH_DONE || g.prefetch_chi);
          const C *chi = (const C *)(g.prefetch_chi ? sm.bufC : sm.bufB);
          if (sum && !chi_here) {
            if (!g.prefetch_chi) {
              __syncthreads();
              if (threadIdx.x == 0) bulk_load(B, chi_g, tile_bytes, &sm.mbar[1]);
            }
            chi_here = true;
            if (!tile_wait(&sm.mbar[1], nchi & 1, &sm.flag[5], a.status, g.inject_timeout ? &sm.mbar[2] : nullptr)) {
              chi_failed = true;
              break;
            }
            ++nchi;
          } else {
            __syncthreads();
          }
          const double ns = norm_part<R, EPT, NL>(it, acc);
          // per-thread sums per control in the state precision, a fiber at a time (a trajectory problem has one term per
          // control; a density matrix a ket and a bra term), converted to FP64 for the reduction
          constexpr int FB = NL > 0 ? NL : EPT;                    // elements summed in the state precision
          typedef typename SumT<R, (EPT > FB)>::T S;
          S sc[KT_MAX_CTRL];
    #pragma unroll
          for (int c = 0; c < KT_MAX_CTRL; ++c) sc[c] = (S)0;
          for (int t = 0; t < g.n_cterms && sum; ++t) {
            const int node = g.cterm_node[t];
            const C *hv = (const C *)sm.hc_val;
            S s = 0;
            // one pass per entry of a factor row, without branches (an empty entry has weight and offset zero), so
            // that the loads of all elements are in flight together
            for (int e = 0; e < g.SH; ++e) {
              if (NL > 0 && node < g.n_nodes - (EPT > NL ? 2 : 1)) {
                // fiber and block mapping, control on another node: one factor row serves the whole fiber (block)
                if (it.ok(0)) {
                  const int b = (t * g.n_loc + ((it.dig(0) >> (4 * node)) & 15)) * g.SH + e, off = sm.hc_off[b];
                  const C w = hv[b];
    #pragma unroll
                  for (int f = 0; f < EPT; f += FB) {
                    R sf = 0;
    #pragma unroll
                    for (int q = f; q < f + FB; ++q) {
                      const C x = chi[it.item(q)], h = cmul(w, A[it.item(q) + off]);
                      sf += x.x * h.y - x.y * h.x;       // Im(conj(chi) * h)
                    }
                    s += (S)sf;
                  }
                }
              } else {
    #pragma unroll
                for (int f = 0; f < EPT; f += FB) {
                  R sf = 0;
    #pragma unroll
                  for (int q = f; q < f + FB; ++q) {
                    if (!it.ok(q)) continue;
                    const int b = (t * g.n_loc + ((it.dig(q) >> (4 * node)) & 15)) * g.SH + e;
                    const C x = chi[it.item(q)], h = cmul(hv[b], A[it.item(q) + sm.hc_off[b]]);
                    sf += x.x * h.y - x.y * h.x;
                  }
                  s += (S)sf;
                }
              }
            }
            const int ct = g.cterm_ctrl[t];
    #pragma unroll
            for (int c = 0; c < KT_MAX_CTRL; ++c)
              if (c == ct) sc[c] += s;
          }
          // FP64 block reduction: the norm and the controls, four values when there are at most three controls
          // (FP64 runs at 1/64 of the FP32 rate here, and every slot costs additions in each lane)
          double nrm_t = 0.0;
          if (!sum) {
            double v[1] = {ns};
            reduce_tau<1>(v, g, sm.red, sm.tsc + TS_V0 * g.T);
            vstride = 1;
          } else if (g.n_ctrl <= 3) {
            double v[4] = {ns, (double)sc[0], (double)sc[1], (double)sc[2]};
            reduce_tau<4>(v, g, sm.red, sm.tsc + TS_V0 * g.T);
            vstride = 4;
          } else if (g.n_ctrl < KT_MAX_CTRL) {
            double v[8];
            v[0] = ns;
    #pragma unroll
            for (int c = 1; c < 8; ++c) v[c] = (double)sc[c - 1];
            reduce_tau<8>(v, g, sm.red, sm.tsc + TS_V0 * g.T);
            vstride = 8;
          } else {
            double n1[1] = {ns};
            reduce_tau<1>(n1, g, sm.red, sm.tsc + TS_V0 * g.T);
            if (threadIdx.x < g.T) nrm_t = sm.tsc[TS_V0 * g.T + threadIdx.x];
            __syncthreads();
            double v[8];
    #pragma unroll
            for (int c = 0; c < 8; ++c) v[c] = (double)sc[c];
            reduce_tau<8>(v, g, sm.red, sm.tsc + TS_V0 * g.T);
            vstride = 8;
            voff = 0;
          }
          if (phase == PH_DONE) break;
          if (threadIdx.x < g.T) {
            const int t = threadIdx.x, k = tile * g.T + t;
            const double nrm = voff ? sm.tsc[TS_V0 * g.T + t * vstride] : nrm_t;
            const double r = r_start;                        // padding trajectories carry r = -1
            if (!isfinite(nrm)) set_status(a.status, KT_DEV_NONFINITE);
            const int act = (k < g.M) && (nrm <= r);         // jump iff ||psi||^2 <= r
            sm.tin[TI_ACT * g.T + t] = act;
            if (act) {
              sm.tsc[TS_R * g.T + t] = r;
              sm.tsc[TS_S0 * g.T + t] = 0.0;
              sm.tsc[TS_LEN * g.T + t] = g.dt;
              sm.tsc[TS_PP * g.T + t] = nrm;                 // n at the end of the piece, until the root search is set up
              atomicAdd(&sm.flag[0], 1);
            }
          }
          __syncthreads();
          if (sm.flag[0] == 0) {
            if (need_chi && !sum) {
              phase = PH_DONE;           // chi(t_j) takes the buffer that the series has left
              continue;
            }
            break;
          }
          // a jump: the tile's results go to psi_out now (coalesced), and flagged trajectories
          // restart from psi(t_{j-1}), kept in psi_out
          jumped = true;
          for (int e = threadIdx.x; e < g.d * g.T; e += blockDim.x) psi_out[e] = A[e];
          __syncthreads();
    #pragma unroll
          for (int q = 0; q < EPT; ++q)
            if (it.ok(q) && sm.tin[TI_ACT * g.T + tau]) psi_out[it.item(q)] = psi_in[it.item(q)];
          __syncthreads();
          phase = PH_REST;               // set the root search up below
        } else if (phase == PH_ROOT) {
          // n and p at the trial time: one Newton step, kept inside the bracket
          double v[2];
    #pragma unroll
          for (int q = 0; q < EPT; ++q)
            if (it.ok(q)) A[it.item(q)] = acc[q];
          __syncthreads();
          v[0] = norm_part<R, EPT, NL>(it, acc);
          v[1] = loss(A);
          reduce_tau<2>(v, g, sm.red, sm.tsc + TS_V0 * g.T);
          if (threadIdx.x < g.T) {
            const int t = threadIdx.x;
            if (sm.tin[TI_ACT * g.T + t] && sm.tin[TI_BUSY * g.T + t])
              newton(t, sm.tsc[TS_V0 * g.T + 2 * t] - sm.tsc[TS_R * g.T + t], sm.tsc[TS_V0 * g.T + 2 * t + 1]);
          }
          __syncthreads();
          continue;
        } else if (phase == PH_SSTAR) {
    #pragma unroll
          for (int q = 0; q < EPT; ++q)
            if (it.ok(q)) A[it.item(q)] = acc[q];
          if (threadIdx.x == 0) sm.flag[1] = 0;
          __syncthreads();
          double nv[1] = {norm_part<R, EPT, NL>(it, acc)};
          reduce_tau<1>(nv, g, sm.red, sm.tsc + TS_V0 * g.T);
          const double nstar = threadIdx.x < g.T ? sm.tsc[TS_V0 * g.T + threadIdx.x] : 0.0;
          __syncthreads();
          // channel probabilities p_l = ||L_l phi||^2
          double v[KT_MAX_LIND];
          for (int l = 0; l < KT_MAX_LIND; ++l) v[l] = l < g.n_lind ? channel(l, A) : 0.0;
          reduce_tau<KT_MAX_LIND>(v, g, sm.red, sm.tsc + TS_V0 * g.T);
          // the norm there is r to its own rounding (one of its type per term), or this was a trial like the others: the
          // estimate of what a step leaves can be wrong, two slopes may agree by chance
          if (threadIdx.x < g.T && sm.tin[TI_ACT * g.T + threadIdx.x] && !g.first_order) {
            const int t = threadIdx.x;
            const double f = nstar - sm.tsc[TS_R * g.T + t];
            if (fabs(f) > (sizeof(R) == 8 ? 0x1p-52 : 0x1p-23) * g.K && sm.tin[TI_CH * g.T + t] < 60) {
              double p = 0.0;
              for (int l = 0; l < g.n_lind; ++l) p += sm.tsc[TS_V0 * g.T + t * KT_MAX_LIND + l];
              newton(t, f, p);
              sm.flag[1] = 1;
            }
          }
          __syncthreads();
          if (sm.flag[1]) {
            phase = PH_ROOT;
            continue;
          }
          if (threadIdx.x < g.T) {
            const int t = threadIdx.x, k = tile * g.T + t;
            int ch = -1;
            if (sm.tin[TI_ACT * g.T + t]) {
              const double *p = sm.tsc + TS_V0 * g.T + t * KT_MAX_LIND;
              const int m = a.jcount[k] + 1;
              if (m > g.max_jumps) {
                set_status(a.status, KT_DEV_RECORD_FULL);
                sm.tin[TI_ACT * g.T + t] = 0;
              } else if (g.n_lind == 0) {
                set_status(a.status, KT_DEV_ZERO_JUMP);      // norm loss without any jump operator
                sm.tin[TI_ACT * g.T + t] = 0;
              } else {
                const double *U = a.U + ((size_t)*a.pass_row * g.M + k) * g.draws;
                double tot = 0.0;
                for (int l = 0; l < g.n_lind; ++l) tot += p[l];
                const double target = U[2 * m - 1] * tot;   // first channel whose cumulative p reaches u * sum p
                ch = g.n_lind - 1;
                double cum = 0.0;
                for (int l = 0; l < g.n_lind; ++l) {
                  cum += p[l];
                  if (cum >= target) { ch = l; break; }
                }
                if (!(p[ch] > 0.0)) {
                  set_status(a.status, KT_DEV_ZERO_JUMP);
                  sm.tin[TI_ACT * g.T + t] = 0;
                  ch = -1;
                } else {
                  const double cnorm = 1.0 / sqrt(p[ch]);
                  const double sstar = sm.tsc[TS_S0 * g.T + t] + sm.tsc[TS_S * g.T + t];
                  const size_t ri = (size_t)k * g.max_jumps + (m - 1);
                  a.rec_step[ri] = j;
                  a.rec_ch[ri] = ch;
                  a.rec_s[ri] = sstar;
                  a.rec_c[ri] = cnorm;
                  a.jcount[k] = m;
                  const double rn = U[2 * m];
                  a.rstate[k] = rn;
                  sm.tsc[TS_R * g.T + t] = rn;
                  sm.tsc[TS_S0 * g.T + t] = sstar;
                  sm.tsc[TS_C * g.T + t] = cnorm;
                }
              }
            }
            sm.tin[TI_NJ * g.T + t] = ch;
          }
          __syncthreads();
          // collapse: start <- c L_ch phi
          const int ch = sm.tin[TI_NJ * g.T + tau];
          if (ch >= 0) {
            const R cn = (R)sm.tsc[TS_C * g.T + tau];
    #pragma unroll UJ
            for (int q = 0; q < EPT; ++q) {
              if (!it.ok(q)) continue;
              const C y = lind_item<R>(g, ops, ch, 0, A, it.item(q), it.dig(q));
              psi_out[it.item(q)] = mkc(cn * y.x, cn * y.y);
            }
          }
          __syncthreads();
          phase = PH_REST;
          continue;
        } else {  // PH_REST
          double v[1] = {norm_part<R, EPT, NL>(it, acc)};
          if (threadIdx.x == 0) sm.flag[2] = 0;
          reduce_tau<1>(v, g, sm.red, sm.tsc + TS_V0 * g.T);
          if (threadIdx.x < g.T) {
            const int t = threadIdx.x;
            int done = 0;
            if (sm.tin[TI_ACT * g.T + t]) {
              const double nrm = sm.tsc[TS_V0 * g.T + t];
              if (nrm > sm.tsc[TS_R * g.T + t]) done = 1;
              else {
                atomicAdd(&sm.flag[2], 1);      // another jump inside the remainder
                sm.tsc[TS_LEN * g.T + t] = g.dt - sm.tsc[TS_S0 * g.T + t];
                sm.tsc[TS_PP * g.T + t] = nrm;
              }
            }
            sm.tin[TI_BUSY * g.T + t] = done;
          }
          __syncthreads();
    #pragma unroll
          for (int q = 0; q < EPT; ++q)
            if (it.ok(q) && sm.tin[TI_BUSY * g.T + tau]) psi_out[it.item(q)] = acc[q];
          __syncthreads();
          if (threadIdx.x < g.T && sm.tin[TI_BUSY * g.T + threadIdx.x]) sm.tin[TI_ACT * g.T + threadIdx.x] = 0;
          __syncthreads();
          ++guard;
          if (sm.flag[2] == 0 || guard > g.max_jumps + 1) {
            // final states of the whole tile
    #pragma unroll
            for (int q = 0; q < EPT; ++q)
              if (it.ok(q)) acc[q] = psi_out[it.item(q)];
            __syncthreads();
            phase = PH_DONE;
            if (j == a.nt || !a.overlap) break;
            continue;
          }
    #pragma unroll
          for (int q = 0; q < EPT; ++q)
            if (it.ok(q)) A[it.item(q)] = acc[q];    // the states at the end of the piece, for the slope there
          __syncthreads();
        }
        // ---- set the root search of the flagged trajectories up: slopes at both ends, norm at the start (A holds
        // the states at the end of the piece, psi_out those at its start)
        {
          double v[4];
          v[0] = loss(A);
          __syncthreads();
          load_tile<R, EPT>(g, it, psi_out, A);
          __syncthreads();
    #pragma unroll
          for (int q = 0; q < EPT; ++q)
            if (it.ok(q)) acc[q] = A[it.item(q)];
          v[1] = norm_part<R, EPT, NL>(it, acc);
          v[2] = loss(A);
          v[3] = 0.0;
          reduce_tau<4>(v, g, sm.red, sm.tsc + TS_V0 * g.T);
          if (threadIdx.x < g.T && sm.tin[TI_ACT * g.T + threadIdx.x]) {
            const int t = threadIdx.x;
            const double len = sm.tsc[TS_LEN * g.T + t], n1 = sm.tsc[TS_PP * g.T + t];
            const double *o = sm.tsc + TS_V0 * g.T + 4 * t;
            sm.tsc[TS_LO * g.T + t] = 0.0;
            sm.tsc[TS_HI * g.T + t] = len;
            sm.tsc[TS_S * g.T + t] = g.first_order ? len : hermite_root(o[1], n1, o[2], o[0], len, sm.tsc[TS_R * g.T + t]);
            sm.tsc[TS_PS * g.T + t] = len;
            sm.tsc[TS_PP * g.T + t] = o[0];
            sm.tin[TI_CH * g.T + t] = 0;                     // trials of the root search
            sm.tin[TI_BUSY * g.T + t] = !g.first_order;      // first-order scheme: the jump is applied at dt
          }
          __syncthreads();
          phase = PH_ROOT;
        }
      }
      if (chi_failed) {
        if (threadIdx.x == 0) {
          if (store_pending || stored) bulk_store_wait();
          // the next tile's psi is on its way into the fourth buffer: let it land before leaving
          if (persist && next < g.n_tiles) mbar_wait_bounded((use & 1) ? &sm.mbar[0] : &sm.mbar[3], ((use + 1) >> 1) & 1);
        }
        return;
      }

      if (j >= 1 && !jumped) {
        if (sweep) {
          // sweep: plain stores, read back by the next interval's jump restarts after a CTA barrier
    #pragma unroll
          for (int q = 0; q < EPT; ++q)
            if (it.ok(q)) psi_out[it.item(q)] = acc[q];
        } else {
          // psi(t_j) of the whole tile is in A (fenced and synchronised above): one bulk store to psi_out
          if (threadIdx.x == 0) bulk_store(psi_out, A, tile_bytes);
          stored = true;
        }
      }

      // ---------------- end of the sweep: tau_k = <tgt|psi_k>/||psi_k|| ----------------
      if (j == a.nt) {
        double v[3] = {0.0, 0.0, 0.0};
    #pragma unroll
        for (int q = 0; q < EPT; ++q) {
          if (!it.ok(q)) continue;
          const KtCplx t = ops.tgt[it.item(q) / g.T];
          const double xr = (double)acc[q].x, xi = (double)acc[q].y;
          v[0] += t.re * xr + t.im * xi;   // conj(tgt) * psi
          v[1] += t.re * xi - t.im * xr;
          v[2] += xr * xr + xi * xi;
        }
        reduce_tau<3>(v, g, sm.red, sm.tsc + TS_V0 * g.T);
        if (threadIdx.x < g.T) {
          const int k = tile * g.T + threadIdx.x;
          const double *o = sm.tsc + TS_V0 * g.T + threadIdx.x * 3;
          const double nrm = o[2];
          // a trajectory's overlap is taken with the normalised state; a density matrix's
          // <<P_tgt|rho(T)>> is linear in rho and is not normalised
          const double inv = g.density ? 1.0 : (nrm > 0.0 ? 1.0 / sqrt(nrm) : 0.0);
          a.tau[k].re = o[0] * inv;
          a.tau[k].im = o[1] * inv;
          a.norm2[k] = nrm;
          if (!isfinite(nrm) || !isfinite(o[0]) || !isfinite(o[1])) set_status(a.status, KT_DEV_NONFINITE);
        }
        store_pending = store_pending || stored;
        end_fwd_tile(sm, persist);
        continue;
      }

      // ---------------- this tile's part of the update overlap at t_j ----------------
      if (!a.overlap) {
        store_pending = store_pending || stored;
        end_fwd_tile(sm, persist);
        continue;
      }
      if (threadIdx.x < g.n_ctrl) {
        double s = 0.0;
        for (int t = 0; t < g.T; ++t) s += sm.tsc[TS_V0 * g.T + t * vstride + voff + threadIdx.x];
        if (sweep) put_partial(a.partials + ((size_t)j * g.n_tiles + tile) * g.n_ctrl + threadIdx.x, s);
        else a.partials[(size_t)tile * g.n_ctrl + threadIdx.x] = s;
      }
      store_pending = store_pending || stored;
      end_fwd_tile(sm, persist);
      // every thread is done with this tile's chi (the barrier above): the third buffer takes the next tile's
      if (persist && need_chi && g.prefetch_chi && next < g.n_tiles && threadIdx.x == 0)
        bulk_load(sm.bufC, (const C *)a.chi_t + (size_t)next * g.tile_elems, tile_bytes, &sm.mbar[1]);
    }   // tiles of this CTA
    // Delta eps of interval j+1 from the partials of all tiles: every thread adds a fixed, contiguous
    // chunk of the tiles and a fixed shuffle/warp tree adds the chunks -- the same order on every run
    // for a given tile count and block size.  The new pulse value goes to sm.eps (the next interval of
    // a sweep) and, with write_out, to deps / eps_new.
    auto finish_update = [&](const double *part, bool write_out) -> bool {
      const int chunk = (g.n_tiles + (int)blockDim.x - 1) / (int)blockDim.x;
      const int t0 = threadIdx.x * chunk, t1 = min(g.n_tiles, t0 + chunk);
      bool late = false;
      for (int c = 0; c < g.n_ctrl; ++c) {
        double v = 0.0;
        if (sweep) {
          // poll the chunk's slots until every value is there
          const long long clk = clock64();
          for (bool all = false; !all && !late;) {
            all = true;
            v = 0.0;
            for (int t = t0; t < t1; ++t) {
              const unsigned long long b = get_partial(part + (size_t)t * g.n_ctrl + c);
              all = all && b != kNoValue;
              v += __longlong_as_double((long long)b);
            }
            late = !all && clock64() - clk > KT_WAIT_CYCLES;
          }
        } else {
          for (int t = t0; t < t1; ++t) v += __ldcg(part + (size_t)t * g.n_ctrl + c);
        }
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0) sm.red[(threadIdx.x >> 5) * 8 + c] = v;
      }
      if (late) {
        set_status(a.status, KT_DEV_TIMEOUT);
        sm.flag[6] = 1;
      }
      __syncthreads();
      if (threadIdx.x < g.n_ctrl) {
        const int c = threadIdx.x;
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += sm.red[w * 8 + c];
        const size_t idx = (size_t)c * a.nt + j;   // interval j+1 (0-based index j)
        const double de = (sweep ? fin_scale : a.shape[idx] / (g.lam[c] * g.M_norm)) * s;
        const double en = (sweep ? fin_eold : a.eps_old[idx]) + de;
        if (write_out) {
          a.deps[idx] = de;
          a.eps_new[idx] = en;
          if (!isfinite(de)) set_status(a.status, KT_DEV_NONFINITE);
          if (fabs(en) > g.eps_bound) set_status(a.status, KT_DEV_RANGE);
        }
        sm.eps[c] = en;
      }
      return sm.flag[6] == 0;
    };
    if (sweep) {
      if (j == a.nt) break;
      if (!need_chi) continue;                 // guess sweep: nothing to exchange between intervals
      if (!finish_update(a.partials + (size_t)j * g.n_tiles * g.n_ctrl, blockIdx.x == 0)) break;   // timed out: results void
      continue;
    }
    if (!a.overlap || j == a.nt || !a.finish) {   // no update sum here (a shard sums after its exchange)
      if (threadIdx.x == 0 && store_pending) bulk_store_wait();
      return;
    }
    // ---------------- last CTA: Delta eps of interval j+1, summed in tile order ----------------
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
      const unsigned ticket = atomicAdd(a.counter, 1u);
      sm.flag[3] = (ticket == (unsigned)(gridDim.x - 1));
    }
    __syncthreads();
    if (threadIdx.x == 0 && store_pending) bulk_store_wait();
    if (!sm.flag[3]) return;
    __threadfence();
    finish_update(a.partials, true);
    if (threadIdx.x == 0) *a.counter = 0u;
    return;
  }   // intervals
  if (threadIdx.x == 0 && store_pending) bulk_store_wait();
}

// --------------------------------------------------------------------------------------
// Backward interval kernel: chi(t_{j-1}) = U_j^dag chi(t_j) along each trajectory's record.
// Round rnd propagates piece rnd of the interval (backwards: dt - s_m, s_m - s_{m-1}, ..., s_1)
// and then applies conj(c) L^dag of the jump that bounds it.  One Chebyshev call site.
// With a.forward_replay the same kernel replays a recorded forward pass instead: the image is
// the forward generator's, pieces run forwards (s_1, s_2 - s_1, ..., dt - s_m) and each is
// followed by c L of its jump -- the frozen-record map U_j of the gradient (no bisection).
// Tiles: with g.bwd_grid > 0 the grid holds that many CTAs, each looping over tiles blockIdx.x,
// blockIdx.x + gridDim.x, ...: the tables and the item mapping (which depend on the interval only)
// are built once, and the next tile's input arrives by bulk copy in a third buffer while the current
// tile's series runs (loads alternate between two transaction barriers).  Otherwise one tile per CTA.
// With a.sweep one launch runs the whole backward sweep of its tile, intervals a.j down to 1 (the
// co-states of different trajectories never meet, so the CTAs need no synchronisation): the state
// stays in shared memory from one interval to the next, and each interval's result is stored to its
// co-state slot.
template <typename R, int EPT, int NL, int ACS, bool SWEEP, int MAXT>
__global__ void __launch_bounds__(MAXT, kt_min_ctas(sizeof(R), EPT, NL, MAXT)) bwd_kernel(KtGeom g, KtGenImage im, KtOps ops, BwdArgs a) {
  typedef typename C2<R>::T C;
  extern __shared__ __align__(16) char smem_raw[];
  Smem sm;
  constexpr bool sweep = SWEEP;   // a.sweep, compiled in
  const bool persist = !sweep && g.bwd_grid > 0;
  char *const extra = smem_raw + carve(g, sizeof(C), smem_raw, &sm, persist);
  const int tau = threadIdx.x % g.T;
  const int j_first = a.j, j_last = sweep ? 1 : a.j;
  if (threadIdx.x < g.n_ctrl) sm.eps[threadIdx.x] = a.eps[threadIdx.x * a.nt + (j_first - 1)];
  if (threadIdx.x < 8) sm.flag[threadIdx.x] = 0;
  if (threadIdx.x == 0) {
    mbar_init(&sm.mbar[0], 1);
    mbar_init(&sm.mbar[1], 1);
    mbar_init(&sm.mbar[2], 1);
    fence_mbar_init();
  }
  __syncthreads();
  const uint32_t tile_bytes = (uint32_t)(g.tile_elems * sizeof(C));
  int tile = blockIdx.x;
  if (threadIdx.x == 0)
    bulk_load(sm.bufB, (const C *)a.chi_in + (size_t)tile * g.tile_elems, tile_bytes, &sm.mbar[0]);
  build_tables<R>(g, im, ops, sm, sm.eps, false);
  const bool fw = a.forward_replay != 0;
  Items<EPT, NL> it;
  load_items<EPT, NL>(g, ops, it);
  SweepKeep keep;
  if constexpr (SWEEP) sweep_keep_init<R>(g, im, extra, keep);
  int cur = -1, cur_step = 0;      // the trajectory's latest unprocessed record (forward replay: the next) and its interval
  double eps_ahead = 0.0;          // sweep: the next interval's pulse
  bool store_pending = false;
  for (int use = 0; tile < g.n_tiles; tile += gridDim.x, ++use) {
    // this tile's input: load number `use`, on barrier use & 1 with phase parity (use >> 1) & 1
    if (!tile_wait(&sm.mbar[use & 1], (use >> 1) & 1, &sm.flag[4], a.status,
                   g.inject_timeout ? &sm.mbar[2] : nullptr)) {
      if (threadIdx.x == 0 && store_pending) bulk_store_wait();
      return;
    }
    const int next = tile + (int)gridDim.x;
    if (persist && next < g.n_tiles && threadIdx.x == 0)   // the third buffer is free: prefetch the next input
      bulk_load(sm.bufC, (const C *)a.chi_in + (size_t)next * g.tile_elems, tile_bytes, &sm.mbar[(use + 1) & 1]);
    for (int j = j_first; j >= j_last; --j) {
      C *chi_out = sweep ? (C *)((char *)a.chi_slots + (size_t)(j - 1) * a.slot_bytes) + (size_t)tile * g.tile_elems
                         : (C *)a.chi_out + (size_t)tile * g.tile_elems;
      if (sweep && threadIdx.x < g.n_ctrl) {
        if (j != j_first) sm.eps[threadIdx.x] = eps_ahead;
        if (j > 1) eps_ahead = a.eps[threadIdx.x * a.nt + (j - 2)];
      }
      if (threadIdx.x == 0) sm.flag[0] = 0;
      if (threadIdx.x == 0 && store_pending) bulk_store_wait();   // A still feeds the previous tile's store
      store_pending = false;
      int nj = 0;
      if (threadIdx.x < g.T) {
        const int t = threadIdx.x, k = tile * g.T + t;
        if (k < g.M) {
          const int cnt = fw ? a.jcount[k] : 0;
          auto held = [&]() { return fw ? cur < cnt : cur >= 0; };
          if (j == j_first) {
            cur = a.cursor[k];
            cur_step = held() ? a.rec_step[(size_t)k * g.max_jumps + cur] : 0;
          }
          while (held() && cur_step == j && nj < 12) {
            sm.tin[(TI_J0 + nj) * g.T + t] = cur;   // forward replay ascending in time, backward descending
            ++nj;
            cur += fw ? 1 : -1;
            cur_step = held() ? a.rec_step[(size_t)k * g.max_jumps + cur] : 0;
          }
          if (held() && cur_step == j) set_status(a.status, KT_DEV_RECORD_FULL);
          if (a.advance_cursor && j == j_last) a.cursor[k] = cur;
        }
        sm.tin[TI_NJ * g.T + t] = nj;
      }
      // most intervals hold no jump: one barrier then says so (and covers the pulse and flag[0] above)
      int rounds = __syncthreads_or(nj);
      if (rounds) {
        if (threadIdx.x < g.T) atomicMax(&sm.flag[0], nj);
        __syncthreads();
        rounds = sm.flag[0];
      }
      if constexpr (SWEEP) {
        // the next interval's tables (every read of the previous one's ended with its series)
        if (j != j_first) sweep_tables<R>(g, im, ops, sm, keep);
      }
      C *A = (C *)sm.bufA;
      C *B = (C *)sm.bufB;
      C acc[EPT];
      for (int rnd = 0; rnd <= rounds; ++rnd) {
        Smem run = sm;
        if (rounds == 0) {
          if constexpr (SWEEP) sweep_coefs<R>(g, im, sm, run, keep, extra, j);
          else uniform_coefs<R, t_form<R, NL, ACS>()>(g, sm, im, j);
        } else if (threadIdx.x < g.T) {
          const int t = threadIdx.x, k = tile * g.T + t;
          double len = 0.0;
          if (rnd <= nj) {
            const double *rs = a.rec_s + (size_t)k * g.max_jumps;
            if (fw) {   // pieces forwards: s_1 - 0, s_2 - s_1, ..., dt - s_m
              const double lo = (rnd == 0) ? 0.0 : rs[sm.tin[(TI_J0 + rnd - 1) * g.T + t]];
              const double hi = (rnd < nj) ? rs[sm.tin[(TI_J0 + rnd) * g.T + t]] : g.dt;
              len = hi - lo;
            } else {    // pieces backwards: dt - s_m, s_m - s_{m-1}, ..., s_1 - 0
              const double hi = (rnd == 0) ? g.dt : rs[sm.tin[(TI_J0 + rnd - 1) * g.T + t]];
              const double lo = (rnd < nj) ? rs[sm.tin[(TI_J0 + rnd) * g.T + t]] : 0.0;
              len = hi - lo;
            }
          }
          sm.tsc[TS_X * g.T + t] = len;
        }
        if (rounds > 0) {
          __syncthreads();
          piece_coefs<R, t_form<R, NL, ACS>()>(g, im, sm, fw ? g.c_fwd : g.c_bwd);
        }
        // B holds the vector to propagate (a sweep's later intervals start with it in A)
        if (!sweep || j == j_first || rnd > 0) {
  #pragma unroll
          for (int q = 0; q < EPT; ++q)
            if (it.ok(q)) A[it.item(q)] = B[it.item(q)];
        }
        __syncthreads();
        cheb_dispatch<R, EPT, NL, ACS>(g, im, run, it, g.K, acc);
        if (rnd == rounds) break;
  #pragma unroll
        for (int q = 0; q < EPT; ++q)
          if (it.ok(q)) A[it.item(q)] = acc[q];
        __syncthreads();
        const int njt = sm.tin[TI_NJ * g.T + tau];
        const int k = tile * g.T + tau;
  #pragma unroll (NL > 0 ? 1 : EPT)
        for (int q = 0; q < EPT; ++q) {
          if (!it.ok(q)) continue;
          C y = A[it.item(q)];
          if (rnd < njt) {
            const size_t ri = (size_t)k * g.max_jumps + sm.tin[(TI_J0 + rnd) * g.T + tau];
            const C z = lind_item<R>(g, ops, a.rec_ch[ri], fw ? 0 : 1, A, it.item(q), it.dig(q));
            const R cn = (R)a.rec_c[ri];
            y = mkc(cn * z.x, cn * z.y);
          }
          B[it.item(q)] = y;
        }
        __syncthreads();
      }
      // chi(t_{j-1}) of the whole tile: into A, then one bulk store (completed before A is reused); a sweep starts its
      // next interval from A and stores from its registers, which nothing has to wait for
  #pragma unroll
      for (int q = 0; q < EPT; ++q)
        if (it.ok(q)) {
          A[it.item(q)] = acc[q];
          if (sweep) chi_out[it.item(q)] = acc[q];
        }
      if (!sweep) {
        fence_proxy_async_smem();
        __syncthreads();
        if (threadIdx.x == 0) bulk_store(chi_out, A, tile_bytes);
        store_pending = true;
      }
    }   // intervals
    // the prefetched input becomes this CTA's input buffer; the old one (free) the next prefetch target
    void *tmp = sm.bufB;
    sm.bufB = sm.bufC;
    sm.bufC = tmp;
  }
  if (threadIdx.x == 0 && store_pending) bulk_store_wait();
}

}  // namespace kt
