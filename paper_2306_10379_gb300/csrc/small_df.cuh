// Internal interface of the df64 p x p step (small_df.cu).
#pragma once
#include "blas_f64.cuh"
#include "pp_dev.cuh"

namespace gsi {

// One p x p step (PpArgs, pp_dev.cuh). a.gws: small_df_scratch_bytes(p) of
// device memory. cluster: for 32 < p <= 64, a cluster of 8 CTAs instead of
// one CTA (p > 64 always takes the cluster, p <= 32 never).
size_t small_df_scratch_bytes(int p);
gsi_status small_step_df(const PpArgs& a, bool cluster, cudaStream_t st);

}  // namespace gsi
