// Backward interval kernel instantiations, FP32-mixed (one translation unit per
// kernel family and precision so that the build compiles them in parallel).
#include "kt_device.cuh"

namespace kt {
// a whole sweep (strided and row mapping, those of the small problems) runs one tile per CTA
template <typename R, int EPT, int NL, int ACS, int MAXT>
static cudaError_t launch_bwd_t(const KtGeom &g, const KtGenImage &im, const KtOps &ops, const BwdArgs &a, size_t smem,
                                cudaStream_t st) {
  if constexpr (NL > 0 && ACS >= 3 && ACS <= 5) {
    if (a.y_form) return launch_bwd_t<R, EPT, NL, ACS + 8, MAXT>(g, im, ops, a, smem, st);
  }
  if (a.sweep) {
    if constexpr (NL == 0) {
      const cudaError_t attr = kt_allow_large_smem((const void *)bwd_kernel<R, EPT, 0, ACS, true, MAXT>);
      if (attr != cudaSuccess) return attr;
      bwd_kernel<R, EPT, 0, ACS, true, MAXT><<<g.n_tiles, g.nthreads, smem, st>>>(g, im, ops, a);
      return cudaGetLastError();
    } else {
      return cudaErrorInvalidValue;
    }
  }
  const cudaError_t attr = kt_allow_large_smem((const void *)bwd_kernel<R, EPT, NL, ACS, false, MAXT>);
  if (attr != cudaSuccess) return attr;
  bwd_kernel<R, EPT, NL, ACS, false, MAXT><<<g.bwd_grid > 0 ? g.bwd_grid : g.n_tiles, g.nthreads, smem, st>>>(g, im, ops, a);
  return cudaGetLastError();
}
}  // namespace kt

cudaError_t kt_launch_bwd_f32(int ept, const KtGeom &g, const KtGenImage &im, const KtOps &ops, const BwdArgs &a,
                             size_t smem, cudaStream_t st) {
  switch (ept) {
    case 1: return kt::launch_bwd_t<float, 1, 0, 0, 1024>(g, im, ops, a, smem, st);   // strided, small problems
    case 2: return kt::launch_bwd_t<float, 2, 0, 0, 1024>(g, im, ops, a, smem, st);
    case 4: return kt::launch_bwd_t<float, 4, 0, 0, 1024>(g, im, ops, a, smem, st);
    case 8: return kt::launch_bwd_t<float, 8, 0, 0, 1024>(g, im, ops, a, smem, st);
    case 16: return kt::launch_bwd_t<float, 16, 0, 0, 1024>(g, im, ops, a, smem, st);
    case 21:   // row mapping, up to two nodes and one pair
      return g.nthreads <= 256 ? kt::launch_bwd_t<float, 1, 0, 6, 256>(g, im, ops, a, smem, st)
                               : kt::launch_bwd_t<float, 1, 0, 6, 1024>(g, im, ops, a, smem, st);
    case 33:   // row mapping, up to three nodes and three pairs
      return g.nthreads <= 256 ? kt::launch_bwd_t<float, 1, 0, 7, 256>(g, im, ops, a, smem, st)
                               : kt::launch_bwd_t<float, 1, 0, 7, 768>(g, im, ops, a, smem, st);
    case -6: return kt::launch_bwd_t<float, 6, 6, 0, 736>(g, im, ops, a, smem, st);   // fiber mapping, n_loc = 6
    case -9: return kt::launch_bwd_t<float, 9, 9, 0, 736>(g, im, ops, a, smem, st);   // fiber mapping, n_loc = 9
    case -106: return kt::launch_bwd_t<float, 6, 6, 1, 736>(g, im, ops, a, smem, st);  // cavity structure, cutoff 1
    case -109: return kt::launch_bwd_t<float, 9, 9, 1, 736>(g, im, ops, a, smem, st);  // cavity structure, cutoff 2
    case -209: return kt::launch_bwd_t<float, 9, 9, 2, 736>(g, im, ops, a, smem, st);  // cavity structure, cutoff 2, T = 1
    case -306:  // real / imaginary couplings, cutoff 1
      return g.nthreads <= 256 ? kt::launch_bwd_t<float, 6, 6, 3, 256>(g, im, ops, a, smem, st)
                               : kt::launch_bwd_t<float, 6, 6, 3, 736>(g, im, ops, a, smem, st);
    case -309:  // real / imaginary couplings, cutoff 2
      return g.nthreads <= 256 ? kt::launch_bwd_t<float, 9, 9, 3, 256>(g, im, ops, a, smem, st)
                               : kt::launch_bwd_t<float, 9, 9, 3, 736>(g, im, ops, a, smem, st);
    case -409:  // the same with T = 1
      return g.nthreads <= 256 ? kt::launch_bwd_t<float, 9, 9, 4, 256>(g, im, ops, a, smem, st)
                               : kt::launch_bwd_t<float, 9, 9, 4, 736>(g, im, ops, a, smem, st);
    case -506: return kt::launch_bwd_t<float, 12, 6, 5, 256>(g, im, ops, a, smem, st);  // block mapping, cutoff 1
    case -509: return kt::launch_bwd_t<float, 27, 9, 5, 256>(g, im, ops, a, smem, st);  // block mapping, cutoff 2
  }
  return cudaErrorInvalidValue;
}
