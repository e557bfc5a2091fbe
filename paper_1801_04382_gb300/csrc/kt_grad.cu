// Gradient of the trajectory functional with respect to the piecewise-constant controls, with
// the jump record of the forward pass held fixed (the differentiable object defined by freezing
// (interval, s*, channel, c) of every jump; J_T is invariant to the c's).
//
//   dJ_T/deps_ij = -(2/M) sum_k Re <chi~_k(t_j)| dU_kj/deps_i |psi_k(t_{j-1})>,
//
// U_kj = P(tau_m) c_m L ... c_1 L P(tau_0) the trajectory's map over interval j (pieces between its
// recorded jumps), chi~ the co-state of the exact boundary propagated backwards along the same
// record.  By the product rule the bracket is a sum over pieces q of <W_q| dP(tau_q) |Z_q>, Z_q the
// state at the start of piece q and W_q the co-state at its end.  dP(tau)/deps_i is evaluated
// exactly with the Chebyshev series of the block-triangular generator [[G, H_i], [0, G]] applied
// to [0; Z]: T_k of that block matrix carries dT_k(Ghat)/deps in its upper-right block, so the
// recurrences z_{k+1} = z_{k-1} + B z_k and y_{k+1} = y_{k-1} + B y_k + B_i z_k (B = -2i (G - c) / r as in
// kt_device.cuh, B_i = -2i H_i / r its derivative; z_1 = B z_0 / 2, y_0 = 0, y_1 = B_i z_0 / 2) give
// dP/deps_i Z = exp(-i c tau) sum_k m_k y_k with the propagator's own coefficients (the same constants c, r:
// only B depends on eps).
//
// That costs 2 n_ctrl generator applications per term.  Where the generator has the cavity structure with real /
// imaginary classes and the controls are its drives, grad_adj_kernel differentiates the series in reverse instead:
// with Wt = exp(-i c tau)^* W,
//   b_k = m_k Wt + b_{k+2} + B^dag b_{k+1}  (b_K = 0; the last step, k = 0, with B^dag b_1 / 2),
//   Re <W| dP/deps_i |Z> = Re sum_{k >= 1} <b_{k+1}| B_i |z_k> + Re <b_1| B_i |z_0> / 2,   b_0 = P^dag W,
// two applications per term whatever the number of controls, and b_0 is the co-state at the start of the piece, so the
// backward interval kernel is not launched.  B_i has the drive's entries only: its bilinear forms take the neighbour
// values that B^dag loads anyway.  The z_k of a thread's own fiber wait in global memory (K states; written and
// read back once, coalesced, mostly in L2).  Per interval, gradient, backward and replay launches of before together against
// this one: d = 729, 1024 trajectories, three controls, FP32 572 -> 189 us; d = 6561, 64 trajectories 2084 -> 182 us; d = 216,
// 200 trajectories 362 -> 50 us; d = 81, 100 trajectories, FP64 693 -> 382 us.
//
// One CTA per trajectory, gathered from the problem's interleaved tile layout.
#include "kt_device.cuh"

namespace kt {

__host__ __device__ inline size_t grad_carve(const KtGeom &g1, int esz, char *base, Smem *s, void **D) {
  size_t off = carve(g1, esz, base, s, true);
  off = align_up(off, 16);
  if (D) *D = base ? base + off : nullptr;
  off += (size_t)g1.tile_elems * esz;
  return align_up(off, 16);
}

// trajectory k of a tile-layout array (T_layout interleaved) -> dst[x]
template <typename R, int EPT, class IT>
__device__ __forceinline__ void gather_traj(const IT &it, const typename C2<R>::T *tiles, int k, int T_layout,
                                            int tel, typename C2<R>::T *dst) {
  const typename C2<R>::T *src = tiles + (size_t)(k / T_layout) * tel + (k % T_layout);
#pragma unroll
  for (int q = 0; q < EPT; ++q)
    if (it.ok(q)) dst[it.item(q)] = src[(size_t)it.item(q) * T_layout];
}

// B_c v = -2i H_c / r v at one item
template <typename R>
__device__ __forceinline__ typename C2<R>::T hc_item(const KtGeom &g, const Smem &sm, int c,
                                                     const typename C2<R>::T *v, int item, uint32_t dig, R invr) {
  typedef typename C2<R>::T C;
  const C *hv = (const C *)sm.hc_val;
  const int xi = (dig >> (4 * g.ctrl_node[c])) & 15;
  const int base = (c * g.n_loc + xi) * g.SH;
  C h = mkc((R)0, (R)0);
  for (int e = 0; e < g.SH; ++e) {
    const C w = hv[base + e];
    if (w.x != (R)0 || w.y != (R)0) h = cfma(w, v[item + sm.hc_off[base + e]], h);
  }
  return mkc((R)2 * h.y * invr, (R)-2 * h.x * invr);
}

// acc = exp(-i c s) sum_k m_k y_k, the derivative along control c of the propagator's series on z0 (z0 in A, synced).
// Uses A, B (z recurrence) and C, D (y recurrence).  Ends synchronised.
template <typename R, int EPT, class IT>
__device__ void aug_run(const KtGeom &g, const KtGenImage &im, const Smem &sm, const IT &it, int K, int c,
                        typename C2<R>::T *Dbuf, typename C2<R>::T (&acc)[EPT]) {
  typedef typename C2<R>::T C;
  C *A = (C *)sm.bufA, *B = (C *)sm.bufB, *Cb = (C *)sm.bufC, *D = Dbuf;
  const R *cf = (const R *)sm.coef;
  const R invr = (R)(1.0 / g.r);
  const C zero = mkc((R)0, (R)0);
  Diag<R> dv[EPT];
#pragma unroll
  for (int q = 0; q < EPT; ++q) {
    acc[q] = zero;
    if (!it.ok(q)) continue;
    dv[q] = diag_of<R>(g, sm, it.dig(q));
    Cb[it.item(q)] = zero;   // y_0 = 0
  }
  if (K < 2) { __syncthreads(); return; }
  const R c1 = cf[1];
#pragma unroll
  for (int q = 0; q < EPT; ++q) {
    if (!it.ok(q)) continue;
    const int i = it.item(q);
    const C z1 = apply_item<R>(g, im, sm, A, i, it.dig(q), dv[q], zero);
    const C y1 = hc_item<R>(g, sm, c, A, i, it.dig(q), invr);
    B[i] = mkc((R)0.5 * z1.x, (R)0.5 * z1.y);
    D[i] = mkc((R)0.5 * y1.x, (R)0.5 * y1.y);
    acc[q] = rfma(c1, D[i], acc[q]);
  }
  __syncthreads();
  C *Pz = A, *Qz = B, *Py = Cb, *Qy = D;
  for (int k = 2; k < K; ++k) {
    const R ak = cf[k];
#pragma unroll
    for (int q = 0; q < EPT; ++q) {
      if (!it.ok(q)) continue;
      const int i = it.item(q);
      const C hz = hc_item<R>(g, sm, c, Qz, i, it.dig(q), invr);
      const C oy = Py[i];
      const C ny = apply_item<R>(g, im, sm, Qy, i, it.dig(q), dv[q], mkc(oy.x + hz.x, oy.y + hz.y));
      Pz[i] = apply_item<R>(g, im, sm, Qz, i, it.dig(q), dv[q], Pz[i]);
      Py[i] = ny;
      acc[q] = rfma(ak, ny, acc[q]);
    }
    __syncthreads();
    C *t1 = Pz; Pz = Qz; Qz = t1;
    C *t2 = Py; Py = Qy; Qy = t2;
  }
  apply_phase<R, EPT>(g, sm, 0, acc, [&](int q) { return it.ok(q) ? dv[q].lo : (R)0; });
}

// The CTA's sums per control and, in the last CTA, dJ_T/deps of interval j.
__device__ __forceinline__ void grad_finish(const KtGeom &g, const Smem &sm, const GradArgs &a, double (&part)[KT_MAX_CTRL]) {
  const int k = blockIdx.x, j = a.j;
  reduce_tau<KT_MAX_CTRL>(part, g, sm.red, sm.tsc + TS_V0 * g.T);
  if (threadIdx.x < g.n_ctrl) a.partials[(size_t)k * g.n_ctrl + threadIdx.x] = sm.tsc[TS_V0 * g.T + threadIdx.x];
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned ticket = atomicAdd(a.counter, 1u);
    sm.flag[3] = (ticket == (unsigned)(gridDim.x - 1));
  }
  __syncthreads();
  if (!sm.flag[3]) return;
  __threadfence();
  const int chunk = ((int)gridDim.x + blockDim.x - 1) / blockDim.x;
  const int t0 = threadIdx.x * chunk, t1 = min((int)gridDim.x, t0 + chunk);
  for (int c = 0; c < g.n_ctrl; ++c) {
    double v = 0.0;
    for (int t = t0; t < t1; ++t) v += __ldcg(a.partials + (size_t)t * g.n_ctrl + c);
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) sm.red[(threadIdx.x >> 5) * 8 + c] = v;
  }
  __syncthreads();
  if (threadIdx.x < g.n_ctrl) {
    double s = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += sm.red[w * 8 + threadIdx.x];
    const double gr = -2.0 / (double)g.M * s;
    a.grad[(size_t)threadIdx.x * a.nt + (j - 1)] = gr;
    if (!isfinite(gr)) set_status(a.status, KT_DEV_NONFINITE);
  }
  if (threadIdx.x == 0) *a.counter = 0u;
}

// A sum over the terms and pieces of an interval.  FP32: in two floats (Knuth's two-sum), the rounding errors of the first
// collected in the second -- seven FP32 additions where one to FP64 would take a warp 128 cycles; what is added at a
// time is a sum over at most nine elements.  Against sums in single floats: d = 729, 1024 trajectories 183 -> 189 us, d = 6561, 64
// trajectories 160 -> 182 us (80 registers).
template <typename R> struct Wide;
template <> struct Wide<double> {
  double s = 0.0;
  __device__ __forceinline__ void add(double x) { s += x; }
  __device__ __forceinline__ double value() const { return s; }
};
template <> struct Wide<float> {
  float s = 0.f, e = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float t = s + x, z = t - s;
    e += (s - (t - z)) + (x - z);
    s = t;
  }
  __device__ __forceinline__ double value() const { return (double)s + (double)e; }
};

// One step of the reverse series on the thread's fiber (tile width 1): out[q] = h (B^dag b)[q] + add[q], b's own values
// in bk, add[q] = m W[q] + prev[base + q]; and dot[i] += h sum_q Re(conj(b at the drive neighbour of node i) y[q]) for the
// outer nodes, dl[.] the same for the last node, one slot per e_n and r_n row.
template <typename R, int NC>
__device__ __forceinline__ void adj_step(const KtGeom &g, const KtGenImage &im, const Smem &sm,
                                         const typename C2<R>::T *__restrict__ v, const typename C2<R>::T *prev, int base,
                                         uint32_t fdig, Diag<R> Df, const RowCache<R> &rc, R h, R m,
                                         const typename C2<R>::T (&w)[3 * (NC + 1)], typename C2<R>::T (&bk)[3 * (NC + 1)],
                                         const typename C2<R>::T *__restrict__ ysrc, int ystride, Wide<R> (&dot)[3],
                                         Wide<R> (&dl)[2 * (NC + 1)]) {
  typedef typename C2<R>::T C;
  constexpr int NP = NC + 1, NL = 3 * NP;
  const C *pv = (const C *)sm.pair_val;
  const C *ld = (const C *)sm.ldense;
  const int last = g.n_nodes - 1;
  C y[NL], out[NL];
#pragma unroll
  for (int q = 0; q < NL; ++q) y[q] = ysrc[(size_t)q * ystride];
#pragma unroll
  for (int q = 0; q < NL; ++q) {
    const R re = Df.re + acs_kd<R>(im, q).re;
    out[q] = mkc(re * bk[q].x, re * bk[q].y);
  }
#pragma unroll
  for (int n = 1; n <= NC; ++n) {
    const int qr = 2 * NP + n - 1, qg = n;
    out[qr] = ifma(acs_kc<R>(im)[n - 1], bk[qg], out[qr]);
    out[qg] = ifma(acs_kc<R>(im)[NC + n - 1], bk[qr], out[qg]);
  }
#pragma unroll
  for (int n = 0; n <= NC; ++n) {
    const int qr = 2 * NP + n, qe = NP + n;
    out[qr] = rfma(ld[qr * NL + qe].x, bk[qe], out[qr]);
    out[qe] = rfma(ld[qe * NL + qr].x, bk[qr], out[qe]);
    dl[n].add(h * fma(bk[qr].y, y[qe].y, bk[qr].x * y[qe].x));             // row e_n, neighbour r_n
    dl[NP + n].add(h * fma(bk[qe].y, y[qr].y, bk[qe].x * y[qr].x));        // row r_n, neighbour e_n
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    if (rc.off0[i]) {
#pragma unroll
      for (int q = 0; q < NL; ++q) out[q] = ifma(rc.a[i], v[base + rc.off0[i] + q], out[q]);
    }
    if (rc.off1[i]) {
      R s = (R)0;
#pragma unroll
      for (int q = 0; q < NL; ++q) {
        const C x = v[base + rc.off1[i] + q];
        out[q] = rfma(rc.b[i], x, out[q]);
        s = fma(x.x, y[q].x, s);
        s = fma(x.y, y[q].y, s);
      }
      dot[i].add(h * s);
    }
  }
  for (int p = 0; p < g.n_pairs; ++p) {
    const int pd = im.pair_dst[p], ps = im.pair_src[p];
    if (pd != last && ps != last) {
      const int e = p * NL * NL + ((fdig >> (4 * pd)) & 15) * NL + ((fdig >> (4 * ps)) & 15);
      const int off = sm.pair_off[e];
      if (off) {
        const R b = pv[e].x;
#pragma unroll
        for (int q = 0; q < NL; ++q) out[q] = rfma(b, v[base + off + q], out[q]);
      }
    } else if (pd == last) {
      const int xs = (fdig >> (4 * ps)) & 15;
      if (xs % NP < NC) {
        const int off = g.stride[ps];
        const R cb = acs_kp<R>(im)[p] * sqrt_n<R>(xs % NP + 1);
#pragma unroll
        for (int q = 0; q < NL; ++q)
          if (q % NP != 0) out[q] = rfma(cb * sqrt_n<R>(q % NP), v[base + off + q - 1], out[q]);
      }
    } else {
      const int xd = (fdig >> (4 * pd)) & 15;
      if (xd % NP >= 1) {
        const int off = -g.stride[pd];
        const R cb = acs_kp<R>(im)[p] * sqrt_n<R>(xd % NP);
#pragma unroll
        for (int q = 0; q < NL; ++q)
          if (q % NP != NC) out[q] = rfma(cb * sqrt_n<R>(q % NP + 1), v[base + off + q + 1], out[q]);
      }
    }
  }
  // the small terms first, as in the forward series
#pragma unroll
  for (int q = 0; q < NL; ++q) {
    const R hi = h * (Df.hi + acs_kd<R>(im, q).hi);
    const C old = prev[base + q];
    C s = mkc(h * out[q].x, h * out[q].y);
    s = rfma(m, w[q], s);
    s.x += old.x;
    s.y += old.y;
    bk[q] = mkc(fma(-hi, bk[q].y, s.x), fma(hi, bk[q].x, s.y));
  }
}

// Reverse gradient of interval j and the co-state at its start (see above).  One CTA per trajectory, one thread per
// last-node fiber.
template <typename R, int NC, int MAXT>
__global__ void __launch_bounds__(MAXT, MAXT == 96 && sizeof(R) == 4 ? 5 : 1)
    grad_adj_kernel(KtGeom g, int T_layout, int tel, KtGenImage imf, KtGenImage imb, KtOps ops, GradArgs a) {
  typedef typename C2<R>::T C;
  constexpr int NP = NC + 1, NL = 3 * NP;
  extern __shared__ __align__(16) char smem_raw[];
  Smem sm;
  carve(g, sizeof(C), smem_raw, &sm, false);
  C *A = (C *)sm.bufA, *B = (C *)sm.bufB;
  const int k = blockIdx.x, j = a.j;
  const size_t rb = (size_t)k * g.max_jumps;
  if (threadIdx.x < g.n_ctrl) sm.eps[threadIdx.x] = a.eps[threadIdx.x * a.nt + (j - 1)];
  if (threadIdx.x < 8) sm.flag[threadIdx.x] = 0;
  if (threadIdx.x == 0) {
    // records of interval j in ascending time: walk down from the backward cursor, then reverse
    int cur = a.cursor[k], n = 0, idx[12];
    while (cur >= 0 && a.rec_step[rb + cur] == j && n < 12) idx[n++] = cur--;
    if (cur >= 0 && a.rec_step[rb + cur] == j) set_status(a.status, KT_DEV_RECORD_FULL);
    for (int m = 0; m < n; ++m) sm.tin[TI_J0 + m] = idx[n - 1 - m];
    sm.tin[TI_NJ] = n;
    a.cursor[k] = cur;
  }
  __syncthreads();
  const int m = sm.tin[TI_NJ];
  Items<NL, NL> it;
  load_items<NL, NL>(g, ops, it);
  const bool ok = it.ok(0);
  const int base = it.item(0), last = g.n_nodes - 1;
  const uint32_t fdig = it.dig(0);
  const size_t tile = (size_t)(k / T_layout) * tel + (k % T_layout);
  const C *psi = (const C *)a.psi_prev + tile, *chi = (const C *)a.chi_t + tile;
  C *ybuf = (C *)a.scratch + (size_t)k * g.K * NL * blockDim.x + threadIdx.x;   // y_n element q at [n][q][thread]
  const int ys = blockDim.x;
  auto sb = [&](int p) -> double { return p == 0 ? 0.0 : (p > m ? g.dt : a.rec_s[rb + sm.tin[TI_J0 + p - 1]]); };
  const R *cf = (const R *)sm.coef;
  Wide<R> dot[3], dl[2 * NP];
  C w[NL];   // the co-state at the end of the current piece
#pragma unroll
  for (int q = 0; q < NL; ++q) w[q] = ok ? chi[(size_t)(base + q) * T_layout] : mkc((R)0, (R)0);
  for (int q = m; q >= 0; --q) {
    // ---- Z_q: psi(t_{j-1}) taken forward over pieces 0 .. q-1 and their jumps
    if (ok) {
#pragma unroll
      for (int e = 0; e < NL; ++e) A[base + e] = psi[(size_t)(base + e) * T_layout];
    }
    build_tables<R>(g, imf, ops, sm, sm.eps, false);
    __syncthreads();
    for (int p = 0; p < q; ++p) {
      C acc[NL];
      if (threadIdx.x == 0) sm.tsc[TS_X] = sb(p + 1) - sb(p);
      __syncthreads();
      piece_coefs<R, false>(g, imf, sm, g.c_fwd);
      __syncthreads();
      cheb_run_acs<R, NC, 1, true, false>(g, imf, sm, it, g.K, acc);
      if (ok) {
#pragma unroll
        for (int e = 0; e < NL; ++e) A[base + e] = acc[e];
      }
      __syncthreads();
      const size_t ri = rb + sm.tin[TI_J0 + p];
      const R cn = (R)a.rec_c[ri];
      if (ok) {
#pragma unroll 1
        for (int e = 0; e < NL; ++e) {
          const C z = lind_item<R>(g, ops, a.rec_ch[ri], 0, A, base + e, it.dig(e));
          B[base + e] = mkc(cn * z.x, cn * z.y);
        }
      }
      __syncthreads();
      if (ok) {
#pragma unroll
        for (int e = 0; e < NL; ++e) A[base + e] = B[base + e];
      }
      __syncthreads();
    }
    // ---- y_0 .. y_{K-2} of piece q, each thread's fiber to its place in ybuf
    if (m == 0) {
      uniform_coefs<R, false>(g, sm, imf, j);
    } else {
      if (threadIdx.x == 0) sm.tsc[TS_X] = sb(q + 1) - sb(q);
      __syncthreads();
      piece_coefs<R, false>(g, imf, sm, g.c_fwd);
    }
    RowCache<R> rc;
    Diag<R> Df{(R)0, (R)0, (R)0};
    if (ok) {
      load_rows<R, NL>(g, sm, fdig, rc);
      for (int i = 0; i < last; ++i) Df = add_diag(Df, load_diag<R>(sm, i * NL + ((fdig >> (4 * i)) & 15)));
    }
    {
      C vk[NL], t[NL];
      C *P = B, *Q = A;
      if (ok) {
#pragma unroll
        for (int e = 0; e < NL; ++e) {
          vk[e] = A[base + e];
          ybuf[(size_t)e * ys] = vk[e];
        }
      }
      for (int n = 1; n < g.K - 1; ++n) {
        if (ok) {
          if (n == 1) {
            apply_acs<R, NC, 1, true, true, false, false>(g, imf, sm, Q, Q, base, fdig, Df, vk, t, rc);
#pragma unroll
            for (int e = 0; e < NL; ++e) t[e] = mkc((R)0.5 * t[e].x, (R)0.5 * t[e].y);
          } else {
            apply_acs<R, NC, 1, true, true, true, false>(g, imf, sm, Q, P, base, fdig, Df, vk, t, rc);
          }
#pragma unroll
          for (int e = 0; e < NL; ++e) {
            vk[e] = t[e];
            P[base + e] = t[e];
            ybuf[((size_t)n * NL + e) * ys] = t[e];
          }
        }
        __syncthreads();
        C *tmp = P; P = Q; Q = tmp;
      }
      __syncthreads();   // every read of the forward tables and of the coefficients' phase is done
    }
    // ---- the reverse series under B^dag (the backward direction's B), its phase the forward one's conjugate
    if (threadIdx.x == 0) {
      C *ph = (C *)sm.phase;
      ph[0].y = -ph[0].y;
      if (sizeof(R) == 4) ph[1].y = -ph[1].y;
    }
    build_tables<R>(g, imb, ops, sm, sm.eps, false);
    __syncthreads();
    if (ok) {
      load_rows<R, NL>(g, sm, fdig, rc);
      Df = Diag<R>{(R)0, (R)0, (R)0};
      for (int i = 0; i < last; ++i) Df = add_diag(Df, load_diag<R>(sm, i * NL + ((fdig >> (4 * i)) & 15)));
    }
    apply_phase<R, NL>(g, sm, 0, w, [&](int e) { return Df.lo + acs_kd<R>(imb, e).lo; });
    {
      C bk[NL];
      const R mk = cf[g.K - 1];
      C *P = B, *Q = A;
      if (ok) {
#pragma unroll
        for (int e = 0; e < NL; ++e) {
          bk[e] = mkc(mk * w[e].x, mk * w[e].y);
          Q[base + e] = bk[e];
          P[base + e] = mkc((R)0, (R)0);
        }
      }
      __syncthreads();
      for (int n = g.K - 2; n >= 0; --n) {
        if (ok) {
          adj_step<R, NC>(g, imb, sm, Q, P, base, fdig, Df, rc, n == 0 ? (R)0.5 : (R)1, cf[n], w, bk,
                          ybuf + (size_t)n * NL * ys, ys, dot, dl);
#pragma unroll
          for (int e = 0; e < NL; ++e) P[base + e] = bk[e];
        }
        __syncthreads();
        C *tmp = P; P = Q; Q = tmp;
      }
      if (q > 0) {
        // the jump that starts piece q: c L^dag (b_0 is in Q)
        const size_t ri = rb + sm.tin[TI_J0 + q - 1];
        const R cn = (R)a.rec_c[ri];
        if (ok) {
#pragma unroll 1
          for (int e = 0; e < NL; ++e) {
            const C z = lind_item<R>(g, ops, a.rec_ch[ri], 1, Q, base + e, it.dig(e));
            P[base + e] = mkc(cn * z.x, cn * z.y);
          }
        }
#pragma unroll
        for (int e = 0; e < NL; ++e) w[e] = ok ? P[base + e] : mkc((R)0, (R)0);
        __syncthreads();
      } else {
#pragma unroll
        for (int e = 0; e < NL; ++e) w[e] = ok ? bk[e] : mkc((R)0, (R)0);
      }
    }
  }
  if (ok) {
    C *out = (C *)a.chi_out + tile;
#pragma unroll
    for (int e = 0; e < NL; ++e) out[(size_t)(base + e) * T_layout] = w[e];
  }
  // the bilinear forms weighted with the control terms' entries (per unit eps, real: slot 1 of their node's rows)
  double part[KT_MAX_CTRL];
  const int nls = NL * g.S;
#pragma unroll
  for (int c = 0; c < KT_MAX_CTRL; ++c) {
    part[c] = 0.0;
    if (c >= g.n_ctrl || !ok) continue;
    const int node = g.ctrl_node[c];
    const KtCplx *slot = imb.ctrl_slot + (size_t)c * nls;
    if (node == last) {
#pragma unroll
      for (int e = 0; e < 2 * NP; ++e) part[c] += (double)(R)slot[(NP + e) * g.S + 1].re * dl[e].value();
    } else {
      double d = dot[0].value();
      if (node == 1) d = dot[1].value();
      if (node == 2) d = dot[2].value();
      part[c] = (double)(R)slot[((fdig >> (4 * node)) & 15) * g.S + 1].re * d;
    }
  }
  grad_finish(g, sm, a, part);
}

// Strided items (EPT per thread): any model.
template <typename R, int EPT>
__global__ void __launch_bounds__(EPT == 4 ? 256 : 1024)
    grad_kernel(KtGeom g, int T_layout, int tel, KtGenImage imf, KtGenImage imb, KtOps ops, GradArgs a) {
  typedef typename C2<R>::T C;
  extern __shared__ __align__(16) char smem_raw[];
  Smem sm;
  void *Dv = nullptr;
  grad_carve(g, sizeof(C), smem_raw, &sm, &Dv);
  C *D = (C *)Dv;
  C *A = (C *)sm.bufA, *B = (C *)sm.bufB;
  const int k = blockIdx.x;
  const int j = a.j;
  const size_t rb = (size_t)k * g.max_jumps;
  if (threadIdx.x < g.n_ctrl) sm.eps[threadIdx.x] = a.eps[threadIdx.x * a.nt + (j - 1)];
  if (threadIdx.x < 8) sm.flag[threadIdx.x] = 0;
  if (threadIdx.x == 0) {
    // records of interval j in ascending time: walk down from the backward cursor, then reverse
    int cur = a.cursor[k], n = 0, idx[12];
    while (cur >= 0 && a.rec_step[rb + cur] == j && n < 12) idx[n++] = cur--;
    if (cur >= 0 && a.rec_step[rb + cur] == j) set_status(a.status, KT_DEV_RECORD_FULL);
    for (int m = 0; m < n; ++m) sm.tin[TI_J0 + m] = idx[n - 1 - m];
    sm.tin[TI_NJ] = n;
  }
  __syncthreads();
  const int m = sm.tin[TI_NJ];
  Items<EPT, 0> it;
  load_items<EPT, 0>(g, ops, it);
  const C *psi_t = (const C *)a.psi_prev;
  const C *chi_t = (const C *)a.chi_t;
  // piece boundaries s_0 = 0 < s_1 < ... < s_m < s_{m+1} = dt
  auto sb = [&](int p) -> double { return p == 0 ? 0.0 : (p > m ? g.dt : a.rec_s[rb + sm.tin[TI_J0 + p - 1]]); };
  double part[KT_MAX_CTRL];
  for (int c = 0; c < KT_MAX_CTRL; ++c) part[c] = 0.0;
  C acc[EPT], wq[EPT], zq[EPT];
  for (int q = 0; q <= m; ++q) {
    // phase 0: W_q = chi~ taken back over pieces m..q+1 (adjoint generator, jumps c L^dag);
    // phase 1: Z_q = psi(t_{j-1}) taken forward over pieces 0..q-1 (jumps c L)
    for (int ph = 0; ph < 2; ++ph) {
      const bool adj = ph == 0;
      const KtGenImage &imd = adj ? imb : imf;
      const int np = adj ? m - q : q;
      gather_traj<R, EPT>(it, adj ? chi_t : psi_t, k, T_layout, tel, A);
      if (np > 0 || !adj) build_tables<R>(g, imd, ops, sm, sm.eps, !adj);
      __syncthreads();
      for (int step = 0; step < np; ++step) {
        const int p = adj ? m - step : step;
        if (threadIdx.x == 0) sm.tsc[TS_X] = sb(p + 1) - sb(p);
        __syncthreads();
        piece_coefs<R, false>(g, imd, sm, adj ? g.c_bwd : g.c_fwd);
        __syncthreads();
        cheb_run<R, EPT>(g, imd, sm, it, g.K, acc);
#pragma unroll
        for (int qq = 0; qq < EPT; ++qq)
          if (it.ok(qq)) A[it.item(qq)] = acc[qq];
        __syncthreads();
        const size_t ri = rb + sm.tin[TI_J0 + (adj ? p - 1 : p)];
        const R cn = (R)a.rec_c[ri];
#pragma unroll
        for (int qq = 0; qq < EPT; ++qq)
          if (it.ok(qq)) {
            const C z = lind_item<R>(g, ops, a.rec_ch[ri], adj ? 1 : 0, A, it.item(qq), it.dig(qq));
            B[it.item(qq)] = mkc(cn * z.x, cn * z.y);
          }
        __syncthreads();
#pragma unroll
        for (int qq = 0; qq < EPT; ++qq)
          if (it.ok(qq)) A[it.item(qq)] = B[it.item(qq)];
        __syncthreads();
      }
#pragma unroll
      for (int qq = 0; qq < EPT; ++qq) {
        const C v = it.ok(qq) ? A[it.item(qq)] : mkc((R)0, (R)0);
        if (adj) wq[qq] = v;
        else zq[qq] = v;
      }
      __syncthreads();
    }
    // ---- derivative of piece q along every control: <W_q| dP(tau_q)/deps_c |Z_q>
    if (m == 0) {
      uniform_coefs<R, false>(g, sm, imf, j);
    } else {
      if (threadIdx.x == 0) sm.tsc[TS_X] = sb(q + 1) - sb(q);
      __syncthreads();
      piece_coefs<R, false>(g, imf, sm, g.c_fwd);
    }
    for (int c = 0; c < g.n_ctrl; ++c) {
#pragma unroll
      for (int qq = 0; qq < EPT; ++qq)
        if (it.ok(qq)) A[it.item(qq)] = zq[qq];
      __syncthreads();
      aug_run<R, EPT>(g, imf, sm, it, g.K, c, D, acc);
      double sacc = 0.0;
#pragma unroll
      for (int qq = 0; qq < EPT; ++qq)
        if (it.ok(qq)) sacc += (double)(wq[qq].x * acc[qq].x + wq[qq].y * acc[qq].y);   // Re(conj(W) y)
      part[c] += sacc;
    }
  }
  grad_finish(g, sm, a, part);
}

template <typename R, int EPT>
static cudaError_t launch_grad_t(const KtGeom &g1, int T_layout, int tel, const KtGenImage &imf,
                                 const KtGenImage &imb, const KtOps &ops, const GradArgs &a, cudaStream_t st) {
  const cudaError_t attr = kt_allow_large_smem((const void *)grad_kernel<R, EPT>);
  if (attr != cudaSuccess) return attr;
  const size_t smem = grad_carve(g1, sizeof(typename C2<R>::T), nullptr, nullptr, nullptr);
  grad_kernel<R, EPT><<<g1.M, g1.nthreads, smem, st>>>(g1, T_layout, tel, imf, imb, ops, a);
  return cudaGetLastError();
}

template <typename R, int NC, int MAXT>
static cudaError_t launch_adj_t(const KtGeom &g1, int T_layout, int tel, const KtGenImage &imf,
                                const KtGenImage &imb, const KtOps &ops, const GradArgs &a, cudaStream_t st) {
  const cudaError_t attr = kt_allow_large_smem((const void *)grad_adj_kernel<R, NC, MAXT>);
  if (attr != cudaSuccess) return attr;
  const size_t smem = carve(g1, sizeof(typename C2<R>::T), nullptr, nullptr, false);
  grad_adj_kernel<R, NC, MAXT><<<g1.M, g1.nthreads, smem, st>>>(g1, T_layout, tel, imf, imb, ops, a);
  return cudaGetLastError();
}

}  // namespace kt

size_t kt_grad_smem_bytes(const KtGeom &g1, int elem_bytes, bool reverse) {
  return reverse ? kt::carve(g1, elem_bytes, nullptr, nullptr, false)
                 : kt::grad_carve(g1, elem_bytes, nullptr, nullptr, nullptr);
}

// ept 4, 8: strided; -6, -9: the reverse kernel for that local dimension
cudaError_t kt_launch_grad(int fp64, int ept, const KtGeom &g1, int T_layout, int tel, const KtGenImage &imf,
                           const KtGenImage &imb, const KtOps &ops, const GradArgs &a, cudaStream_t st) {
  const bool small = g1.nthreads <= 96;
#define ADJ(R, NC) (small ? kt::launch_adj_t<R, NC, 96>(g1, T_layout, tel, imf, imb, ops, a, st) \
                          : kt::launch_adj_t<R, NC, 736>(g1, T_layout, tel, imf, imb, ops, a, st))
  switch (ept) {
    case 4: return fp64 ? kt::launch_grad_t<double, 4>(g1, T_layout, tel, imf, imb, ops, a, st)
                        : kt::launch_grad_t<float, 4>(g1, T_layout, tel, imf, imb, ops, a, st);
    case 8: return fp64 ? kt::launch_grad_t<double, 8>(g1, T_layout, tel, imf, imb, ops, a, st)
                        : kt::launch_grad_t<float, 8>(g1, T_layout, tel, imf, imb, ops, a, st);
    case -6: return fp64 ? ADJ(double, 1) : ADJ(float, 1);
    case -9: return fp64 ? ADJ(double, 2) : ADJ(float, 2);
  }
#undef ADJ
  return cudaErrorInvalidValue;
}
