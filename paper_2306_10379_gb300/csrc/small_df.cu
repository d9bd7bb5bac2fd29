// Launches of the p x p step without the float64 pipe (pp_dev.cuh): the
// eigenbasis B = D^T D = V diag(beta) V^T of Eq. (Gdec), the line-search
// coefficients of Eqs. (diags)/(CG_linesearch_D), Alg. 3, and the polar
// normaliser M = S^{-1/2} of the measured Gram S of X + tD (Eq. (Ynew)),
// taken in the eigenbasis, where S is diagonal up to rounding-level terms F,
// by the first-order expansion
//   S^{-1/2} = V [diag(s^{-1/2}) + F o Df] V^T,  Df_ij = -1/(r_i r_j (r_i + r_j)),
// r = sqrt(s) (the divided differences of x^{-1/2}).
#include "small_df.cuh"

namespace gsi {
namespace {

template <class P>
__global__ void __launch_bounds__(P::NT, 1) pp_kernel(PpArgs a) {
  PpCtx<P> c = pp_ctx<P>(a.p, a.gws);
  pp_body<P>(a, c);
}

template <class P>
gsi_status launch(const PpArgs& a, cudaStream_t st) {
  const size_t sm = pp_smem(a.p, P::NC);
  GSI_CUDA_TRY(ensure_dyn_smem((const void*)pp_kernel<P>, (int)sm));
  if (P::NC == 1) {
    pp_kernel<P><<<1, P::NT, sm, st>>>(a);
  } else {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(P::NC);
    cfg.blockDim = dim3(P::NT);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = P::NC;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    GSI_CUDA_TRY(cudaLaunchKernelEx(&cfg, pp_kernel<P>, a));
  }
  GSI_LAUNCH_CHECK();
  return GSI_OK;
}

}  // namespace

size_t small_df_scratch_bytes(int p) { return pp_gws_bytes(p); }

gsi_status small_step_df(const PpArgs& a, bool cluster, cudaStream_t st) {
  if (a.p < 1 || a.p > 128 || ((a.mode == 3 || a.mode == 4) && !a.eig)) return GSI_ERR_ARG;
  // one CTA while a product takes fewer cycles than a cluster barrier and the
  // trip through L2 (p <= 32); a cluster of 8 past p = 64, where the matrices
  // leave shared memory. Between the two a cluster is the faster one but
  // holds 8 SMs, which large Grams beside it would miss: the caller decides.
  if (a.p <= 16) return launch<PpCfg<128, 16, 2, 1, 1, 8, 1, 1, 1>>(a, st);
  if (a.p <= 32) return launch<PpCfg<256, 32, 4, 1, 1, 16, 4, 1, 1>>(a, st);
  if (a.p > 64) return launch<PpCfg<512, 32, 2, 2, 2, 64, 16, 4, 8>>(a, st);
  if (cluster) return launch<PpCfg<512, 32, 1, 1, 2, 32, 16, 1, 8>>(a, st);
  return launch<PpCfg<512, 32, 4, 2, 1, 32, 8, 2, 1>>(a, st);
}

}  // namespace gsi
