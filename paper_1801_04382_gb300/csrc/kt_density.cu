// Density-matrix sweeps: the one Liouville-space state of a two-node model spread over a thread-block cluster.
//
// vec(rho) of two nodes is one state of a four-node network (d^2 = 1296 ... 6561 elements).  In the trajectory kernels it is
// one tile, i.e. one CTA on one SM: at d^2 = 6561 a term waits 8.4 us for 729 threads' walks through the
// tables.  Here every element has its own thread on one of up to eight CTAs, its row of B in registers as in the row
// mapping (real / imaginary classes: 4 x 2 node entries, six pair terms), and reads its neighbours wherever they
// are through distributed shared memory; a term then costs about 14 loads in flight together and one cluster
// barrier.  Nothing couples clusters, so a sweep is one launch of one cluster, the update's sum an exchange of one value
// per CTA and control.  Eight CTAs because that is the portable cluster size; fewer where a CTA would hold less than
// 416 elements and the barrier outweigh them.
// Per interval, forward with update / backward, against one CTA: d^2 = 6561 FP32 260 / 277 -> 60 / 54 us, FP64 3945 / 4057 -> 399 /
// 382 us; d^2 = 1296 FP32 129 / 97 -> 29 / 25 us.
#include "kt_device.cuh"

namespace kt {

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// barrier of all threads of the cluster; writes before it are visible to every thread after it
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(rank));
  return a;
}
// the value at a cluster shared address, 0 where the address is 0
__device__ __forceinline__ float2 ld_cluster(uint32_t addr, uint32_t shift, float2 *) {
  float2 v;
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\tmov.f32 %0, 0f00000000;\n\tmov.f32 %1, 0f00000000;\n\t"
               "@p ld.shared::cluster.v2.f32 {%0, %1}, [%2];\n\t}"
               : "=&f"(v.x), "=&f"(v.y) : "r"(addr + shift), "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ double2 ld_cluster(uint32_t addr, uint32_t shift, double2 *) {
  double2 v;
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\tmov.f64 %0, 0d0000000000000000;\n\t"
               "mov.f64 %1, 0d0000000000000000;\n\t@p ld.shared::cluster.v2.f64 {%0, %1}, [%2];\n\t}"
               : "=&d"(v.x), "=&d"(v.y) : "r"(addr + shift), "r"(addr) : "memory");
  return v;
}

constexpr int DNN = 4, DNP = 6, DSLOTS = 2 * DNN + DNP;

// Intervals a.j .. a.j_last upwards (forward) or downwards (backward) of the state vec(rho) or vec(P).
template <typename R, bool BWD>
__global__ void __launch_bounds__(832) density_kernel(KtGeom g, KtGenImage im, KtOps ops, DensArgs a) {
  typedef typename C2<R>::T C;
  extern __shared__ __align__(16) char smem_raw[];
  Smem sm;
  const size_t used = carve(g, sizeof(C), smem_raw, &sm, false);
  double *xch = (double *)(smem_raw + used);                  // [8 ranks][KT_MAX_CTRL]
  const int E = g.tile_elems;
  const uint32_t rank = cluster_rank();
  const int x = (int)rank * E + (int)threadIdx.x;
  const bool ok = (int)threadIdx.x < E && x < g.d;
  const uint32_t dig = ok ? ops.digits[x] : 0u;
  C *A = (C *)sm.bufA, *B = (C *)sm.bufB;
  const uint32_t sA = smem_u32(A), shift = smem_u32(B) - sA;
  if (threadIdx.x < g.n_ctrl) {
    const int c = threadIdx.x;
    double e = 0.0;
    if (a.j >= 1) {
      e = a.eps_old[c * a.nt + (a.j - 1)];
      if (a.update) e += a.deps[c * a.nt + (a.j - 1)];
    }
    sm.eps[c] = e;
  }
  __syncthreads();
  build_tables<R>(g, im, ops, sm, sm.eps, a.update != 0);
  __syncthreads();
  auto place = [&](int off) -> uint32_t {                     // cluster address of element x + off in buffer A
    const int y = x + off, r = y / E;
    return map_rank(sA + (uint32_t)(y - r * E) * (uint32_t)sizeof(C), (uint32_t)r);
  };
  RowRegs<R, DNN, DNP> row;
  uint32_t adr[DSLOTS];
#pragma unroll
  for (int e = 0; e < DSLOTS; ++e) adr[e] = 0;
  if (ok) {
    load_row<R, DNN, DNP>(g, im, sm, dig, row);
#pragma unroll
    for (int e = 0; e < DSLOTS; ++e) adr[e] = row.off[e] ? place(row.off[e]) : 0u;
  } else {
#pragma unroll
    for (int e = 0; e < DSLOTS; ++e) row.w[e] = (R)0;
  }
  unsigned any = 0;
#pragma unroll
  for (int e = 0; e < DSLOTS; ++e) any |= (__any_sync(0xffffffffu, adr[e] != 0) ? 1u : 0u) << e;
  C cur = ok ? ((const C *)a.in)[x] : mkc((R)0, (R)0);
  if (ok) A[threadIdx.x] = cur;
  const R *cf = (const R *)sm.coef;
  const int step = BWD ? -1 : 1;
  for (int j = a.j;; j += step) {
    if (j != a.j) {
      // the next interval's pulse (an updating sweep: in sm.eps since the exchange)
      if ((BWD || !a.update) && threadIdx.x < g.n_ctrl) sm.eps[threadIdx.x] = a.eps_old[threadIdx.x * a.nt + (j - 1)];
      __syncthreads();
      build_tables<R>(g, im, ops, sm, sm.eps, false, true);
      __syncthreads();
      if (ok) {
        const C *lv = (const C *)sm.loc_val;
#pragma unroll
        for (int i = 0; i < DNN; ++i) {
          const int e0 = (i * g.n_loc + ((dig >> (4 * i)) & 15)) * 2;
          row.w[2 * i] = lv[e0].y;
          row.w[2 * i + 1] = lv[e0 + 1].x;
        }
      }
    }
    const bool need_chi = !BWD && a.update && j < a.nt;
    C chi = mkc((R)0, (R)0);
    if (need_chi && ok) chi = ((const C *)((const char *)a.chi + (size_t)j * a.slot_bytes))[x];
    if (j >= 1) {
      uniform_coefs<R, false>(g, sm, im, j);
      Diag<R> D{(R)0, (R)0, (R)0};
      if (ok) D = diag_of<R>(g, sm, dig);
      __syncthreads();
      cluster_sync();                                        // y_0 of every CTA is in its buffer A
      C prev = mkc((R)0, (R)0), acc = mkc(cf[0] * cur.x, cf[0] * cur.y);
      uint32_t src = 0;
      C *dst = B;
      C s = diag_init(D, cur, prev);   // of the next term, formed before the barrier
      for (int k = 1; k < g.K; ++k) {
        if (ok) {
          C v[DSLOTS];
#pragma unroll
          for (int e = 0; e < DSLOTS; ++e) v[e] = ld_cluster(adr[e], src, (C *)nullptr);
          C z = mkc((R)0, (R)0);
#pragma unroll
          for (int e = 0; e < DSLOTS; ++e) {
            if (sizeof(R) == 8 && !(any >> e & 1)) continue;   // FP64: an FMA that no lane of the warp needs
            C &t = sizeof(R) == 4 && (e >= 2 * DNN || e % 2) ? z : s;
            t = (e < 2 * DNN && e % 2 == 0) ? ifma(row.w[e], v[e], t) : rfma(row.w[e], v[e], t);
          }
          if (sizeof(R) == 4) {
            s.x += z.x;
            s.y += z.y;
          }
          s = diag_done(D, cur, prev, s);
          if (k == 1) s = mkc((R)0.5 * s.x, (R)0.5 * s.y);
          dst[threadIdx.x] = s;
          prev = cur;
          cur = s;
          acc = rfma(cf[k], cur, acc);
          s = diag_init(D, cur, prev);
        }
        cluster_sync();
        src = shift - src;
        dst = src ? A : B;
      }
      C res[1] = {acc};
      apply_phase<R, 1>(g, sm, 0, res, [&](int) { return D.lo; });
      cur = res[0];
      if (ok) A[threadIdx.x] = cur;
      if (BWD) {
        if (ok) ((C *)((char *)a.out + (size_t)(j - 1) * a.slot_bytes))[x] = cur;
      } else if (ok && j == a.j_last) {
        ((C *)a.out)[x] = cur;
      }
    }
    if (!BWD && j == a.nt) {
      // <<P_tgt|rho(T)>> (linear, not normalised) and the norm, over all CTAs in rank order
      double v[4] = {0.0, 0.0, 0.0, 0.0};
      if (ok) {
        const KtCplx t = ops.tgt[x];
        const double xr = (double)cur.x, xi = (double)cur.y;
        v[0] = t.re * xr + t.im * xi;
        v[1] = t.re * xi - t.im * xr;
        v[2] = xr * xr + xi * xi;
      }
      reduce_tau<4>(v, g, sm.red, sm.tsc + TS_V0);
      if (threadIdx.x < 3) {
        const uint32_t slot = map_rank(smem_u32(xch + rank * KT_MAX_CTRL + threadIdx.x), 0u);
        asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(slot), "d"(sm.tsc[TS_V0 + threadIdx.x]) : "memory");
      }
      cluster_sync();
      if (rank == 0 && threadIdx.x == 0) {
        double o[3] = {0.0, 0.0, 0.0};
        for (int r = 0; r < a.ctas; ++r)
          for (int q = 0; q < 3; ++q) o[q] += xch[r * KT_MAX_CTRL + q];
        a.tau[0].re = o[0];
        a.tau[0].im = o[1];
        a.norm2[0] = o[2];
        if (!isfinite(o[2]) || !isfinite(o[0]) || !isfinite(o[1])) set_status(a.status, KT_DEV_NONFINITE);
      }
    }
    if (need_chi) {
      // Delta eps of interval j+1: Im <<P|dG/deps_c rho>> at t_j, neighbours of the state just written to A
      cluster_sync();
      const C *hv = (const C *)sm.hc_val;
      R sc[KT_MAX_CTRL];
#pragma unroll
      for (int c = 0; c < KT_MAX_CTRL; ++c) sc[c] = (R)0;
      for (int t = 0; t < g.n_cterms && ok; ++t) {
        R s = 0;
        for (int e = 0; e < g.SH; ++e) {
          const int b = (t * g.n_loc + ((dig >> (4 * g.cterm_node[t])) & 15)) * g.SH + e;
          const C h = cmul(hv[b], ld_cluster(place(sm.hc_off[b]), 0u, (C *)nullptr));
          s += chi.x * h.y - chi.y * h.x;
        }
        const int ct = g.cterm_ctrl[t];
#pragma unroll
        for (int c = 0; c < KT_MAX_CTRL; ++c)
          if (c == ct) sc[c] += s;
      }
      double v[KT_MAX_CTRL];
#pragma unroll
      for (int c = 0; c < KT_MAX_CTRL; ++c) v[c] = (double)sc[c];
      reduce_tau<KT_MAX_CTRL>(v, g, sm.red, sm.tsc + TS_V0);
      // this CTA's sums to every CTA of the cluster, then each forms the same sum in rank order
      for (int q = threadIdx.x; q < a.ctas * g.n_ctrl; q += blockDim.x) {
        const int c = q % g.n_ctrl, r = q / g.n_ctrl;
        const uint32_t slot = map_rank(smem_u32(xch + rank * KT_MAX_CTRL + c), (uint32_t)r);
        asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(slot), "d"(sm.tsc[TS_V0 + c]) : "memory");
      }
      cluster_sync();
      if (threadIdx.x < g.n_ctrl) {
        const int c = threadIdx.x;
        double s = 0.0;
        for (int r = 0; r < a.ctas; ++r) s += xch[r * KT_MAX_CTRL + c];
        const size_t idx = (size_t)c * a.nt + j;   // interval j+1 (0-based index j)
        const double de = a.shape[idx] / (g.lam[c] * g.M_norm) * s, en = a.eps_old[idx] + de;
        if (rank == 0) {
          a.deps[idx] = de;
          a.eps_new[idx] = en;
          if (!isfinite(de)) set_status(a.status, KT_DEV_NONFINITE);
          if (fabs(en) > g.eps_bound) set_status(a.status, KT_DEV_RANGE);
        }
        sm.eps[c] = en;
      }
    }
    if (j == a.j_last) break;
  }
  cluster_sync();   // no CTA leaves while another may still read its shared memory
}

template <typename R, bool BWD>
static cudaError_t launch_density_t(const KtGeom &g, const KtGenImage &im, const KtOps &ops, const DensArgs &a,
                                    cudaStream_t st) {
  const cudaError_t attr = kt_allow_large_smem((const void *)density_kernel<R, BWD>);
  if (attr != cudaSuccess) return attr;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)a.ctas);
  cfg.blockDim = dim3((unsigned)g.nthreads);
  cfg.dynamicSmemBytes = carve(g, sizeof(typename C2<R>::T), nullptr, nullptr, false) + 8 * KT_MAX_CTRL * sizeof(double);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)a.ctas;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, density_kernel<R, BWD>, g, im, ops, a);
}

}  // namespace kt

cudaError_t kt_launch_density(int fp64, int backward, const KtGeom &g, const KtGenImage &im, const KtOps &ops,
                              const DensArgs &a, cudaStream_t st) {
  if (fp64) return backward ? kt::launch_density_t<double, true>(g, im, ops, a, st)
                            : kt::launch_density_t<double, false>(g, im, ops, a, st);
  return backward ? kt::launch_density_t<float, true>(g, im, ops, a, st)
                  : kt::launch_density_t<float, false>(g, im, ops, a, st);
}
