// The p x p part of one iteration, run by a single thread block in float64:
// the symmetric eigendecomposition D^T D = V diag(beta) V^T (Eq. (Gdec)), the
// line-search coefficients (Eqs. (diags), (CG_linesearch_D)), the exact step
// of Alg. 3 (bracket of Eqs. (derv1)/(derv2), Brent on phi'(t) of Eq.
// (deriv_P)), and the polar normaliser M = S^{-1/2} of Eq. (Ynew).
//
// The eigensolver is a block-parallel cyclic Jacobi method with round-robin
// (circle) ordering: each round applies p/2 disjoint rotations at once. For
// p <= 128 it starts from the df64 eigenbasis of the same matrix (pp_dev.cuh),
// made orthonormal in float64: V^T B V is then diagonal to about 1e-14 and one
// or two sweeps reach the stopping test, instead of eight from scratch on the
// slow float64 pipe (four barriers and four float64 divisions and roots a
// round): one step p = 8 337 -> 158 us, p = 64 10.2 -> 3.0 ms, p = 128
// 118 -> 21 ms. A and V sit in shared memory up to p = SMALL_SMEM_P.
#include "alg3.cuh"
#include "blas_f64.cuh"
#include "small_dev.cuh"
#include "small_df.cuh"

#include <math.h>

#include <algorithm>

namespace gsi {

constexpr int SMALL_THREADS = 512;
constexpr int SMALL_EIG_MAX = 192;

constexpr int SMALL_SMEM_P = 96;

// the step's own workspace, then the df64 eigenbasis (p x p values and the
// diagonal), 16 diagnostics and the df64 step's scratch
static size_t small_own_doubles(int p) { return (size_t)5 * p * p + 5 * (size_t)p + 64; }
size_t small_scratch_doubles(int p) {
  size_t d = small_own_doubles(p);
  if (p <= 128) d += (size_t)p * p + p + 16 + small_df_scratch_bytes(p) / sizeof(double) + 8;
  return d;
}

// threads of the step: a barrier costs a small p most
static int small_threads(int p) { return p <= 16 ? 128 : p <= 32 ? 256 : SMALL_THREADS; }
static size_t small_smem(int p) { return p <= SMALL_SMEM_P ? (size_t)2 * p * p * sizeof(double) : 0; }

// the df64 eigenbasis of (B + B^T) / 2 into the scratch behind the workspace
static gsi_status small_warm(int p, const double* B, double* scratch, double** eig, cudaStream_t st) {
  *eig = nullptr;
  if (p > 128) return GSI_OK;
  double* e = scratch + ((small_own_doubles(p) + 1) & ~(size_t)1);
  double* out = e + (size_t)p * p + p;
  PpArgs a{};
  a.mode = 3;
  a.p = p;
  a.B = {nullptr, B, 1};
  a.scale_b = 1;
  a.eig = reinterpret_cast<float2*>(e);
  a.out = out;
  a.gws = reinterpret_cast<float2*>(out + 16 + ((p * p + p) & 1));
  *eig = e;
  return small_step_df(a, true, st);
}

// A = (G + G^T) / 2 and V = I, or with a df64 eigenbasis: V from it, one
// Newton-Schulz step in float64, and A = V^T G V. w.T and w.U are scratch.
static __device__ void block_start(int p, const double* G, const float2* eig, SmallWs& w) {
  const int q = p * p;
  if (!eig) {
    for (int e = threadIdx.x; e < q; e += blockDim.x) {
      int i = e / p, j = e - i * p;
      w.A[e] = 0.5 * (G[i * p + j] + G[j * p + i]);
      w.V[e] = (i == j) ? 1.0 : 0.0;
    }
    __syncthreads();
    return;
  }
  for (int e = threadIdx.x; e < q; e += blockDim.x) {
    int i = e / p, j = e - i * p;
    w.V[e] = df_to_double(eig[e]);
    w.A[e] = 0.5 * (G[i * p + j] + G[j * p + i]);
  }
  __syncthreads();
  block_matmul(p, w.V, true, w.V, w.T);
  for (int e = threadIdx.x; e < q; e += blockDim.x) {
    int i = e / p, j = e - i * p;
    w.T[e] = (i == j ? 1.5 : 0.0) - 0.5 * w.T[e];
  }
  __syncthreads();
  block_matmul(p, w.V, false, w.T, w.U);
  for (int e = threadIdx.x; e < q; e += blockDim.x) w.V[e] = w.U[e];
  __syncthreads();
  block_matmul(p, w.A, false, w.V, w.T);
  block_matmul(p, w.V, true, w.T, w.U);
  for (int e = threadIdx.x; e < q; e += blockDim.x) {
    int i = e / p, j = e - i * p;
    w.A[e] = 0.5 * (w.U[i * p + j] + w.U[j * p + i]);
  }
  __syncthreads();
}

static __device__ SmallWs small_carve(double* ws, int p, int in_smem) {
  extern __shared__ __align__(16) unsigned char pp_sm[];
  SmallWs w = carve(ws, p);
  if (in_smem) {
    w.A = reinterpret_cast<double*>(pp_sm);
    w.V = w.A + p * p;
  }
  return w;
}

__global__ void __launch_bounds__(SMALL_THREADS)
small_step_kernel(int mode, int p, const double* C, const double* B, const double* Gam,
                  const double* Z, const double* XX, const double* XD, double* M, double* out,
                  double* ws, const float2* eig, int in_smem) {
  __shared__ double rc[64], rs[64];
  __shared__ int ri[64], rj[64];
  __shared__ double red[64];
  __shared__ int flag;
  __shared__ double sh_t;
  SmallWs w = small_carve(ws, p, in_smem);
  const int q = p * p;
  // 1. eigendecomposition of B (symmetrised)
  block_start(p, B, eig, w);
  block_jacobi(p, w.A, w.V, 60, rc, rs, ri, rj, red);
  if (mode == 1) {
    int st = block_inv_sqrt(p, w.A, w.V, w.sv, M, &flag);
    if (threadIdx.x == 0) {
      out[0] = 0.0;
      out[1] = 0.0;
      out[2] = 0.0;
      out[3] = (double)st;
    }
    return;
  }
  for (int i = threadIdx.x; i < p; i += blockDim.x) w.beta[i] = fmax(w.A[i * p + i], 0.0);
  __syncthreads();
  // 2. alpha, gamma, zeta = diag(V^T {C, Gam, Z} V)
  block_diag_quad(p, C, w.V, w.T, w.alpha);
  block_diag_quad(p, Gam, w.V, w.T, w.gamma);
  block_diag_quad(p, Z, w.V, w.T, w.zeta);
  // 3. the exact step (one warp, the branches over its lanes)
  if (threadIdx.x < 32) {
    int ev = 0;
    const double t = get_mu_warp(p, w.alpha, w.beta, w.gamma, w.zeta, &ev);
    const double ph = phi_model_warp(t, p, w.alpha, w.beta, w.gamma, w.zeta);
    if (threadIdx.x == 0) {
      double bmax = 0.0;
      for (int i = 0; i < p; ++i) bmax = fmax(bmax, w.beta[i]);
      sh_t = t;
      out[0] = t;
      out[1] = ph;
      out[2] = (double)ev;
      out[4] = bmax;
    }
  }
  __syncthreads();
  const double t = sh_t;
  // 4. S = XX + t (XD + XD^T) + t^2 B, rotated into the eigenbasis of B
  for (int e = threadIdx.x; e < q; e += blockDim.x) {
    int i = e / p, j = e - i * p;
    double sij = 0.5 * (XX[i * p + j] + XX[j * p + i]) + t * (XD[i * p + j] + XD[j * p + i]) +
                 t * t * 0.5 * (B[i * p + j] + B[j * p + i]);
    w.S[e] = sij;
  }
  __syncthreads();
  block_matmul(p, w.S, false, w.V, w.T);  // T = S V
  block_matmul(p, w.V, true, w.T, w.U);   // V^T S V (nearly diagonal)
  // exactly symmetric: the rotations look at one half only, and the rounding
  // by which the other half differs kept the sweeps from ever reaching the
  // test (60 of them)
  for (int e = threadIdx.x; e < q; e += blockDim.x) {
    int i = e / p, j = e - i * p;
    w.A[e] = 0.5 * (w.U[i * p + j] + w.U[j * p + i]);
  }
  __syncthreads();
  // the eigenvectors of S: V times the rotations
  block_jacobi(p, w.A, w.V, 60, rc, rs, ri, rj, red);
  int st = block_inv_sqrt(p, w.A, w.V, w.sv, M, &flag);
  if (threadIdx.x == 0) out[3] = (double)st;
}

gsi_status small_step(int mode, int p, const double* C, const double* B, const double* Gam,
                      const double* Z, const double* XX, const double* XD, double* M,
                      double* out, double* scratch, cudaStream_t st) {
  if (p < 1 || p > 128) return GSI_ERR_ARG;
  double* eig = nullptr;
  GSI_TRY(small_warm(p, B, scratch, &eig, st));
  const size_t sm = small_smem(p);
  if (sm) GSI_CUDA_TRY(ensure_dyn_smem((const void*)small_step_kernel, (int)sm));
  small_step_kernel<<<1, small_threads(p), sm, st>>>(mode, p, C, B, Gam, Z, XX, XD, M, out, scratch,
                                                  reinterpret_cast<const float2*>(eig), sm ? 1 : 0);
  GSI_LAUNCH_CHECK();
  return GSI_OK;
}

// Rayleigh-Ritz (Eq. (rr1)): theta descending and U (columns) with
// (C + C^T)/2 = U diag(theta) U^T; p <= SMALL_EIG_MAX (the 3p x 3p
// Rayleigh-Ritz matrix of LOBCG at p <= 64).
__global__ void __launch_bounds__(SMALL_THREADS)
small_eig_kernel(int p, const double* C, double* theta, double* Uout, double* ws, const float2* eig, int in_smem) {
  __shared__ double rc[SMALL_EIG_MAX / 2], rs[SMALL_EIG_MAX / 2];
  __shared__ int ri[SMALL_EIG_MAX / 2], rj[SMALL_EIG_MAX / 2];
  __shared__ double red[64];
  __shared__ int order[SMALL_EIG_MAX];
  SmallWs w = small_carve(ws, p, in_smem);
  const int q = p * p;
  block_start(p, C, eig, w);
  block_jacobi(p, w.A, w.V, 60, rc, rs, ri, rj, red);
  if (threadIdx.x == 0) {
    for (int i = 0; i < p; ++i) order[i] = i;
    for (int i = 0; i < p; ++i) {  // selection sort, descending
      int best = i;
      for (int j = i + 1; j < p; ++j)
        if (w.A[order[j] * p + order[j]] > w.A[order[best] * p + order[best]]) best = j;
      int tmp = order[i];
      order[i] = order[best];
      order[best] = tmp;
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < p; i += blockDim.x) theta[i] = w.A[order[i] * p + order[i]];
  for (int e = threadIdx.x; e < q; e += blockDim.x) {
    int r = e / p, c = e - r * p;
    Uout[e] = w.V[r * p + order[c]];
  }
}

gsi_status small_eig(int p, const double* C, double* theta, double* U, double* scratch,
                     cudaStream_t st) {
  if (p < 1 || p > SMALL_EIG_MAX) return GSI_ERR_ARG;
  double* eig = nullptr;
  GSI_TRY(small_warm(p, C, scratch, &eig, st));
  const size_t sm = small_smem(p);
  if (sm) GSI_CUDA_TRY(ensure_dyn_smem((const void*)small_eig_kernel, (int)sm));
  small_eig_kernel<<<1, small_threads(p), sm, st>>>(p, C, theta, U, scratch, reinterpret_cast<const float2*>(eig),
                                                 sm ? 1 : 0);
  GSI_LAUNCH_CHECK();
  return GSI_OK;
}

}  // namespace gsi
