// Learned warm start: a multilayer perceptron maps the 16 coefficients of a
// diffusion operator to a coarse basis C (m = nc^2 rows, p columns); the
// start block is its bilinear prolongation P C to the fine grid. Training
// minimises the subspace loss L = p - tr(N^{-1} Q), N = C^T S C, S = P^T P,
// Q = C^T Bt Bt^T C, Bt = P^T U against the plain method's converged bases U.
// The paper motivates starting subspace iterations from related problems but
// gives no network; everything here is the project's own.
//
// Kernels: a bfloat16 tensor-core GEMM (mma.sync m16n8k16, float32
// accumulation) with bias / ReLU / ReLU-mask epilogues for the three layers
// forward and backward; column sums for the bias gradients; the per-sample
// loss and its analytic gradient; Adam; prolongation and restriction.
#include <cuda_bf16.h>
#include <math.h>

#include <algorithm>
#include <vector>

#include "common.cuh"
#include "df.cuh"

namespace gsi {
namespace {

__device__ __forceinline__ void mma_bf16_16816(float c[4], const uint32_t a[4], const uint32_t b[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ void cp_bytes16(float* smem, const float* gmem, int bytes) {
  const uint32_t sa = (uint32_t)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(sa), "l"(gmem), "r"(bytes));
}
__device__ __forceinline__ void cp_float(float* smem, const float* gmem, bool valid) {
  const uint32_t sa = (uint32_t)__cvta_generic_to_shared(smem);
  const int sz = valid ? 4 : 0;
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(sa), "l"(gmem), "r"(sz));
}

// How an operand X(i, k) = X[i si + k sk] is staged: along k (sk == 1) or along
// i (si == 1) in 16-byte pieces where base and rows are 16-byte aligned,
// element by element otherwise.
enum : int { G_K16 = 0, G_I16 = 1, G_ANY = 2 };

constexpr int GBK = 32;  // columns of a stage

// A stage of T rows x GBK: [i][k] (row stride GBK + 4), or for G_I16 [k][i]
// (row stride T + 8); both leave the fragment reads free of bank conflicts.
template <int T>
struct GStage {
  static constexpr int KS = GBK + 4, IS = T + 8;
  static constexpr int FLOATS = T * KS > GBK * IS ? T * KS : GBK * IS;
};

template <int T, int NTH>
__device__ __forceinline__ void g_stage(float* dst, const float* __restrict__ X, int64_t si, int64_t sk, int mode,
                                        int i0, int imax, int k0, int kmax) {
  if (mode == G_K16) {
#pragma unroll
    for (int e = threadIdx.x; e < T * (GBK / 4); e += NTH) {
      const int i = e / (GBK / 4), k = 4 * (e % (GBK / 4));
      const int left = i0 + i < imax ? min(4, kmax - (k0 + k)) : 0;
      cp_bytes16(dst + i * GStage<T>::KS + k, left > 0 ? X + (i0 + i) * si + k0 + k : X, left > 0 ? 4 * left : 0);
    }
  } else if (mode == G_I16) {
#pragma unroll
    for (int e = threadIdx.x; e < GBK * (T / 4); e += NTH) {
      const int k = e / (T / 4), i = 4 * (e % (T / 4));
      const int left = k0 + k < kmax ? min(4, imax - (i0 + i)) : 0;
      cp_bytes16(dst + k * GStage<T>::IS + i, left > 0 ? X + (k0 + k) * sk + i0 + i : X, left > 0 ? 4 * left : 0);
    }
  } else {
    for (int e = threadIdx.x; e < T * GBK; e += NTH) {
      // consecutive threads walk the operand's contiguous index
      const int i = si == 1 ? e % T : e / GBK, k = si == 1 ? e / T : e % GBK;
      const bool ok = i0 + i < imax && k0 + k < kmax;
      cp_float(dst + i * GStage<T>::KS + k, ok ? X + (i0 + i) * si + (k0 + k) * sk : X, ok);
    }
  }
}

// the bfloat16 pair (k, k + 1) of row i of a stage
template <int T>
__device__ __forceinline__ uint32_t g_pair(const float* st, int mode, int i, int k) {
  float x, y;
  if (mode == G_I16) {
    x = st[k * GStage<T>::IS + i];
    y = st[(k + 1) * GStage<T>::IS + i];
  } else {
    const float2 v = *reinterpret_cast<const float2*>(st + i * GStage<T>::KS + k);
    x = v.x;
    y = v.y;
  }
  const __nv_bfloat162 b = __floats2bfloat162_rn(x, y);
  return *reinterpret_cast<const uint32_t*>(&b);
}

// C[i][j] = alpha sum_k A(i,k) B(k,j) + beta C[i][j] (+ bias[j]); then, if
// mask: C = 0 where mask[i][j] <= 0; if relu: C = max(C, 0). A(i,k) =
// A[i*sai + k*sak], B(k,j) = B[k*sbk + j*sbj]; operands rounded to
// bfloat16 (nearest even), products summed in float32, k ascending by 16 as
// one accumulation per output whatever the tile.
// Block T x T, 4 warps of T/2 x T/2. The products are few (batch 64): what
// bounds them is the operands' way from memory, so float32 stages of 32
// columns come through NST cp.async buffers, NST - 1 ahead, and are rounded
// when a fragment is read. With one synchronous stage at a time a step of K
// cost a memory latency: 64 x 256 x 256 33 us (now 5 us), 64 x 32768 x 512
// (67 MB of weights) 255 us (now 48 us). T = 32 where T = 64 leaves SMs idle.
template <int T>
__global__ void __launch_bounds__(128) gemm_bf16_kernel(int M, int N, int K, const float* __restrict__ A,
                                                        int64_t sai, int64_t sak, int modeA,
                                                        const float* __restrict__ B, int64_t sbk, int64_t sbj,
                                                        int modeB, float* __restrict__ C, int64_t ldc, float alpha,
                                                        float beta, const float* __restrict__ bias,
                                                        const float* __restrict__ mask, int relu) {
  constexpr int NST = 4, W = T / 2, MI = W / 16, NI = W / 8, SF = GStage<T>::FLOATS;
  extern __shared__ __align__(16) float g_sm[];  // NST stages of A, then of B
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wm = warp >> 1, wn = warp & 1, g = lane >> 2, t = lane & 3;
  const int m0 = blockIdx.y * T, n0 = blockIdx.x * T;
  float acc[MI][NI][4];
#pragma unroll
  for (int a = 0; a < MI; ++a)
#pragma unroll
    for (int b = 0; b < NI; ++b)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[a][b][c] = 0.f;
  const int ns = (K + GBK - 1) / GBK;
  auto stage = [&](int s) {
    if (s < ns) {
      g_stage<T, 128>(g_sm + (s % NST) * SF, A, sai, sak, modeA, m0, M, s * GBK, K);
      g_stage<T, 128>(g_sm + (NST + s % NST) * SF, B, sbj, sbk, modeB, n0, N, s * GBK, K);
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
#pragma unroll
  for (int s = 0; s < NST - 1; ++s) stage(s);
  for (int s = 0; s < ns; ++s) {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(NST - 2) : "memory");
    __syncthreads();  // stage s has landed; stage s - 1 is free
    stage(s + NST - 1);
    const float* as = g_sm + (s % NST) * SF;
    const float* bs = g_sm + (NST + s % NST) * SF;
#pragma unroll
    for (int kk = 0; kk < GBK; kk += 16) {
      uint32_t af[MI][4], bfr[NI][2];
#pragma unroll
      for (int mi = 0; mi < MI; ++mi) {
        const int r = wm * W + mi * 16 + g;
        af[mi][0] = g_pair<T>(as, modeA, r, kk + 2 * t);
        af[mi][1] = g_pair<T>(as, modeA, r + 8, kk + 2 * t);
        af[mi][2] = g_pair<T>(as, modeA, r, kk + 2 * t + 8);
        af[mi][3] = g_pair<T>(as, modeA, r + 8, kk + 2 * t + 8);
      }
#pragma unroll
      for (int ni = 0; ni < NI; ++ni) {
        const int c = wn * W + ni * 8 + g;
        bfr[ni][0] = g_pair<T>(bs, modeB, c, kk + 2 * t);
        bfr[ni][1] = g_pair<T>(bs, modeB, c, kk + 2 * t + 8);
      }
#pragma unroll
      for (int mi = 0; mi < MI; ++mi)
#pragma unroll
        for (int ni = 0; ni < NI; ++ni) mma_bf16_16816(acc[mi][ni], af[mi], bfr[ni]);
    }
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");
#pragma unroll
  for (int mi = 0; mi < MI; ++mi) {
#pragma unroll
    for (int ni = 0; ni < NI; ++ni) {
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int i = m0 + wm * W + mi * 16 + g + (r >= 2 ? 8 : 0);
        const int j = n0 + wn * W + ni * 8 + 2 * t + (r & 1);
        if (i >= M || j >= N) continue;
        const int64_t o = (int64_t)i * ldc + j;
        float v = alpha * acc[mi][ni][r];
        if (beta != 0.f) v += beta * C[o];
        if (bias) v += bias[j];
        if (mask && !(mask[o] > 0.f)) v = 0.f;
        if (relu) v = fmaxf(v, 0.f);
        C[o] = v;
      }
    }
  }
}

// out[j] = sum_i G[i][j] (rows in order)
__global__ void colsum_kernel(int rows, int cols, const float* __restrict__ G, float* __restrict__ out) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= cols) return;
  float s = 0.f;
  for (int i = 0; i < rows; ++i) s += G[(int64_t)i * cols + j];
  out[j] = s;
}

// Adam (Kingma & Ba 2015): c1 = 1 / (1 - b1^t), c2 = 1 / (1 - b2^t)
__global__ void adam_kernel(int64_t count, float* __restrict__ w, const float* __restrict__ g,
                            float* __restrict__ m, float* __restrict__ v, float lr, float b1, float b2,
                            float eps, float c1, float c2) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  w[i] -= lr * (mi * c1) / (sqrtf(vi * c2) + eps);
}

// hat-function weights of fine node f (0-based) against coarse nodes: the
// two neighbours a0, a0 + 1 with weights w0, w1 (absent ones get weight 0)
__device__ __forceinline__ void hat(int f, int nc, int nf, int& a0, double& w0, double& w1) {
  const double tx = (double)(f + 1) * (nc + 1) / (nf + 1) - 1.0;
  a0 = (int)floor(tx);
  w1 = tx - a0;
  w0 = 1.0 - w1;
}

// X[s] (nf^2 x p, float64) = P C[s] (C: nc^2 x p, float32), P = P1 (x) P1
__global__ void prolong_kernel(int nc, int nf, int p, int batch, const float* __restrict__ C,
                               double* __restrict__ X) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t per = (int64_t)nf * nf * p;
  if (idx >= per * batch) return;
  const int s = (int)(idx / per);
  const int64_t e = idx - s * per;
  const int r = (int)(e / p), c = (int)(e - (int64_t)r * p);
  const int i = r % nf, j = r / nf;
  int ax, ay;
  double wx[2], wy[2];
  hat(i, nc, nf, ax, wx[0], wx[1]);
  hat(j, nc, nf, ay, wy[0], wy[1]);
  const float* Cs = C + (int64_t)s * nc * nc * p;
  double v = 0.0;
  for (int db = 0; db < 2; ++db) {
    const int b = ay + db;
    if (b < 0 || b >= nc) continue;
    for (int da = 0; da < 2; ++da) {
      const int a = ax + da;
      if (a < 0 || a >= nc) continue;
      v += wy[db] * wx[da] * (double)Cs[(a + nc * b) * p + c];
    }
  }
  X[idx] = v;
}

// Bt[s] (nc^2 x p, float32) = P^T U[s] (U: nf^2 x p, float64): coarse node
// a gathers the fine nodes inside its hat's support
__global__ void restrict_kernel(int nc, int nf, int p, int batch, const double* __restrict__ U,
                                float* __restrict__ Bt) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t per = (int64_t)nc * nc * p;
  if (idx >= per * batch) return;
  const int s = (int)(idx / per);
  const int64_t e = idx - s * per;
  const int rc = (int)(e / p), c = (int)(e - (int64_t)rc * p);
  const int a = rc % nc, b = rc / nc;
  // fine nodes with |x_f - x_c| < 1/(nc+1): (i+1)/(nf+1) in (a/(nc+1), (a+2)/(nc+1))
  const int lo_a = max(0, (int)floor((double)a * (nf + 1) / (nc + 1)) - 1);
  const int hi_a = min(nf - 1, (int)ceil((double)(a + 2) * (nf + 1) / (nc + 1)));
  const int lo_b = max(0, (int)floor((double)b * (nf + 1) / (nc + 1)) - 1);
  const int hi_b = min(nf - 1, (int)ceil((double)(b + 2) * (nf + 1) / (nc + 1)));
  const double* Us = U + (int64_t)s * nf * nf * p;
  double v = 0.0;
  for (int j = lo_b; j <= hi_b; ++j) {
    const double wy = fmax(0.0, 1.0 - fabs((double)(j + 1) * (nc + 1) / (nf + 1) - (b + 1)));
    if (wy == 0.0) continue;
    for (int i = lo_a; i <= hi_a; ++i) {
      const double wx = fmax(0.0, 1.0 - fabs((double)(i + 1) * (nc + 1) / (nf + 1) - (a + 1)));
      if (wx == 0.0) continue;
      v += wx * wy * Us[(int64_t)(i + nf * j) * p + c];
    }
  }
  Bt[idx] = (float)v;
}

// The loss and its gradient, per sample s with C = C[s], Bt = Bt[s] (m x p):
//   SC = S C; N = C^T SC (symmetrised); G = Bt^T C; Q = G^T G;
//   loss[s] = p - tr(N^{-1} Q);
//   dC[s] = gscale * (-2) [Bt (G N^{-1}) - SC (N^{-1} Q N^{-1})].
// Long sums in float32 over 32-row chunks, chunk sums and the p x p algebra
// in float64 (N^{-1} from its Cholesky factor). A non-positive pivot gives
// loss = NaN and dC = 0.
// Three launches: the row work (SC, N, G; then dC) goes over blocks of WR rows
// of every sample, only the algebra takes one block per sample. One block
// per sample for everything left half of the SMs idle and read every operand
// of the Grams from memory twice per multiply-add: 64 samples, m = 1024,
// p = 32 1,207 us (now 82 + 113 + 28 us; the algebra, a chain on the
// float64 pipe, is what is left).
constexpr int WT = 256;
constexpr int WR = 128;  // rows of a block, a multiple of 32
constexpr int WNZ = 1536;  // entries of S staged per block (bilinear elements: 9 a row)

// acc += a x with a split in two floats: 2^-46 of the terms in float32
// arithmetic, for a sum that is rounded to float32 (C's range decides its
// overflow and underflow as long as |a| lies in [2^-100, 2^60))
__device__ __forceinline__ void w_mac(float& h, float& e, float2 a, float x) {
  const float p = __fmul_rn(a.x, x);
  const float pe = __fmaf_rn(a.x, x, -p);
  const float2 t = two_sum(h, p);
  h = t.x;
  e = __fadd_rn(e, __fadd_rn(t.y, __fmaf_rn(a.y, x, pe)));
}

__global__ void __launch_bounds__(WT) warm_gram_kernel(int m, int p, const int64_t* __restrict__ Srp,
                                                       const int32_t* __restrict__ Sci,
                                                       const double* __restrict__ Sv,
                                                       const float* __restrict__ Call,
                                                       const float* __restrict__ Btall, float* __restrict__ SCall,
                                                       double* __restrict__ part) {
  extern __shared__ __align__(16) float w_rows[];  // WR rows of C, SC and Bt, row stride pp
  // the block's rows of S, its values split in two floats once (a float64
  // conversion for every value and column took half of the kernel's time);
  // rows beyond WNZ entries are read from memory
  __shared__ float2 sval[WNZ];
  __shared__ int32_t scol[WNZ];
  const int tid = threadIdx.x, pp = (p + 3) & ~3, q = p * p;
  float *cs = w_rows, *ss = cs + WR * pp, *bs = ss + WR * pp;
  const int64_t off = (int64_t)blockIdx.y * m * p;
  const float* C = Call + off;
  const int r0 = blockIdx.x * WR, nr = min(WR, m - r0);
  const int64_t k0 = Srp[r0], kn = min((int64_t)WNZ, Srp[r0 + nr] - k0);
  // float64 compares are slow: the exponent field decides
  auto in_range = [](double v) {
    const uint32_t hi = (uint32_t)__double2hiint(v) & 0x7fffffffu;
    return (hi | (uint32_t)__double2loint(v)) == 0u || hi - ((1023u - 100u) << 20) < (160u << 20);
  };
  bool range = true;
  for (int k = tid; k < kn; k += WT) {
    const double v = Sv[k0 + k];
    range = range && in_range(v);
    sval[k] = df_from_double(v);
    scol[k] = Sci[k0 + k];
  }
  for (int64_t k = kn + tid; k < Srp[r0 + nr] - k0; k += WT) range = range && in_range(Sv[k0 + k]);
  const bool pairs = __syncthreads_and(range);
  for (int e = tid; e < WR * pp; e += WT) {
    const int r = e / pp, c = e - r * pp;
    const bool ok = r < nr && c < p;
    float h = 0.f, l = 0.f;
    if (ok) {
      const int64_t kb = Srp[r0 + r] - k0, ke = Srp[r0 + r + 1] - k0;
      int64_t k = kb;
#pragma unroll 3
      for (; k < min(ke, kn); ++k) w_mac(h, l, sval[k], C[(int64_t)scol[k] * p + c]);
      for (; k < ke; ++k) w_mac(h, l, df_from_double(Sv[k0 + k]), C[(int64_t)Sci[k0 + k] * p + c]);
    }
    const float sc = h + l;
    cs[e] = ok ? C[(int64_t)(r0 + r) * p + c] : 0.f;
    bs[e] = ok ? Btall[off + (int64_t)(r0 + r) * p + c] : 0.f;
    ss[e] = sc;
    if (ok) SCall[off + (int64_t)(r0 + r) * p + c] = sc;
  }
  if (!pairs)  // some value beyond a pair's range: S C again, in float64
    for (int e = tid; e < WR * pp; e += WT) {
      const int r = e / pp, c = e - r * pp;
      if (r >= nr || c >= p) continue;
      double a = 0.0;
      for (int64_t k = Srp[r0 + r]; k < Srp[r0 + r + 1]; ++k) a += Sv[k] * (double)C[(int64_t)Sci[k] * p + c];
      ss[e] = (float)a;
      SCall[off + (int64_t)(r0 + r) * p + c] = (float)a;
    }
  __syncthreads();
  // N = C^T SC and G = Bt^T C: a thread forms 4 x 2 entries
  const int ti = pp / 4, tj = (p + 1) / 2;
  double* out = part + ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * 2 * q;
  for (int w = tid; w < 2 * ti * tj; w += WT) {
    const int which = w / (ti * tj), rem = w - which * ti * tj, i = 4 * (rem / tj), j = 2 * (rem % tj);
    const float* U = (which == 0 ? cs : bs) + i;
    const float* V = (which == 0 ? ss : cs) + j;
    double tot[4][2] = {};
    for (int b0 = 0; b0 < nr; b0 += 32) {
      float a[4][2] = {};
      const int b1 = min(nr, b0 + 32);
#pragma unroll 4
      for (int r = b0; r < b1; ++r) {
        const float4 u = *reinterpret_cast<const float4*>(U + r * pp);
        const float2 v = *reinterpret_cast<const float2*>(V + r * pp);
        a[0][0] = fmaf(u.x, v.x, a[0][0]);
        a[0][1] = fmaf(u.x, v.y, a[0][1]);
        a[1][0] = fmaf(u.y, v.x, a[1][0]);
        a[1][1] = fmaf(u.y, v.y, a[1][1]);
        a[2][0] = fmaf(u.z, v.x, a[2][0]);
        a[2][1] = fmaf(u.z, v.y, a[2][1]);
        a[3][0] = fmaf(u.w, v.x, a[3][0]);
        a[3][1] = fmaf(u.w, v.y, a[3][1]);
      }
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 2; ++y) tot[x][y] += (double)a[x][y];
    }
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
      for (int y = 0; y < 2; ++y)
        if (i + x < p && j + y < p) out[which * q + (i + x) * p + j + y] = tot[x][y];
  }
}

// 1/sqrt(d) in float64 from a float32 seed: the pipe's own root and division
// are serial chains of many slow operations
__device__ __forceinline__ double w_rsqrt(double d) {
  const int ex = ((__double2hiint(d) >> 20) & 0x7ff) - 1023;
  if (ex == -1023) return 1.0 / sqrt(d);  // subnormal
  const int h = ex >= 0 ? ex / 2 : -((1 - ex) / 2);              // floor(ex / 2)
  const double sc = __hiloint2double((1023 - 2 * h) << 20, 0);   // d sc in [1, 4)
  const double x = d * sc;
  double y = (double)rsqrtf((float)x);
  y = y * fma(-0.5 * x, y * y, 1.5);
  y = y * fma(-0.5 * x, y * y, 1.5);
  return y * __hiloint2double((1023 - h) << 20, 0);
}

// Dynamic shared memory: 5 p^2 + p doubles. A1 = G N^{-1} and A2 = N^{-1} Q
// N^{-1}: float32, 2 p^2 per sample. status: 1 where N is not positive
// definite (a loss can be NaN for other reasons), else 0.
__global__ void __launch_bounds__(WT) warm_alg_kernel(int p, int nblk, const double* __restrict__ part,
                                                      double* __restrict__ loss, float* __restrict__ Aall,
                                                      int32_t* __restrict__ status) {
  extern __shared__ __align__(16) double wsm[];
  __shared__ int bad;
  __shared__ double trw[WT / 32];
  const int s = blockIdx.x, tid = threadIdx.x, q = p * p;
  double* Nm = wsm;       // N, then its Cholesky factor L (lower)
  double* Gm = Nm + q;    // G
  double* Qm = Gm + q;    // Q
  double* Ni = Qm + q;    // L^{-1}, then N^{-1}
  double* Tm = Ni + q;    // scratch
  double* dinv = Tm + q;  // 1 / L_kk
  float* A1 = Aall + (size_t)s * 2 * q;
  float* A2 = A1 + q;
  if (tid == 0) bad = 0;
  for (int e = tid; e < 2 * q; e += WT) {
    double t = 0.0;
    for (int b = 0; b < nblk; ++b) t += part[((size_t)s * nblk + b) * 2 * q + e];
    (e < q ? Tm : Gm - q)[e] = t;
  }
  __syncthreads();
  for (int e = tid; e < q; e += WT) {  // symmetrise N; Q = G^T G
    const int i = e / p, j = e - i * p;
    Nm[e] = 0.5 * (Tm[e] + Tm[j * p + i]);
    if (j >= i) {
      double a = 0.0;
      for (int k = 0; k < p; ++k) a = fma(Gm[k * p + i], Gm[k * p + j], a);
      Qm[e] = a;
      Qm[j * p + i] = a;
    }
  }
  __syncthreads();
  // Cholesky N = L L^T (right-looking, column k by the block)
  for (int k = 0; k < p; ++k) {
    const double d = Nm[k * p + k];
    const bool ok = d > 0.0 && isfinite(d);
    const double inv = ok ? w_rsqrt(d) : 1.0;
    __syncthreads();
    if (tid == 0) {
      if (!ok) bad = 1;
      dinv[k] = inv;
    }
    for (int i = k + 1 + tid; i < p; i += WT) Nm[i * p + k] *= inv;
    __syncthreads();
    const int w = p - k - 1;
    for (int e = tid; e < w * w; e += WT) {
      const int i = k + 1 + e / w, j = k + 1 + e % w;
      if (j <= i) Nm[i * p + j] -= Nm[i * p + k] * Nm[j * p + k];
    }
    __syncthreads();
  }
  // L^{-1} by forward substitution, four lanes per column (their partial sums
  // are folded in a fixed order)
  for (int c = tid >> 2; c < (p + 7) / 8 * 8; c += WT / 4) {
    const int l4 = tid & 3;
    for (int i = 0; i < p; ++i) {
      double v = 0.0;
      if (c < p)
        for (int k = c + l4; k < i; k += 4) v = fma(Nm[i * p + k], Ni[k * p + c], v);
      v += __shfl_xor_sync(0xffffffffu, v, 1);
      v += __shfl_xor_sync(0xffffffffu, v, 2);
      if (l4 == 0 && c < p) Ni[i * p + c] = i < c ? 0.0 : ((i == c ? 1.0 : 0.0) - v) * dinv[i];
      __syncwarp();
    }
  }
  __syncthreads();
  // N^{-1} = L^{-T} L^{-1}
  for (int e = tid; e < q; e += WT) {
    const int i = e / p, j = e - i * p;
    if (j >= i) {
      double a = 0.0;
      for (int k = j; k < p; ++k) a = fma(Ni[k * p + i], Ni[k * p + j], a);
      Tm[e] = a;
      Tm[j * p + i] = a;
    }
  }
  __syncthreads();
  for (int e = tid; e < q; e += WT) Ni[e] = Tm[e];
  __syncthreads();
  const bool ok = !bad;
  // T = N^{-1} Q; A1 = G N^{-1}
  double tr = 0.0;
  for (int e = tid; e < q; e += WT) {
    const int i = e / p, j = e - i * p;
    double a = 0.0, b = 0.0;
    for (int k = 0; k < p; ++k) {
      a = fma(Ni[i * p + k], Qm[k * p + j], a);
      b = fma(Gm[i * p + k], Ni[k * p + j], b);
    }
    Tm[e] = a;
    A1[e] = ok ? (float)b : NAN;
    if (i == j) tr += a;
  }
  for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(0xffffffffu, tr, o);
  if ((tid & 31) == 0) trw[tid >> 5] = tr;
  __syncthreads();
  // A2 = T N^{-1} (symmetric)
  for (int e = tid; e < q; e += WT) {
    const int i = e / p, j = e - i * p;
    if (j >= i) {
      double a = 0.0;
      for (int k = 0; k < p; ++k) a = fma(Tm[i * p + k], Ni[k * p + j], a);
      A2[e] = ok ? (float)a : NAN;
      A2[j * p + i] = ok ? (float)a : NAN;
    }
  }
  if (tid == 0) {
    double t = 0.0;
    for (int w = 0; w < WT / 32; ++w) t += trw[w];
    loss[s] = ok ? (double)p - t : NAN;
    status[s] = bad;
  }
}

__global__ void __launch_bounds__(WT) warm_dc_kernel(int m, int p, const float* __restrict__ Btall,
                                                     const float* __restrict__ SCall,
                                                     const float* __restrict__ Aall,
                                                     const int32_t* __restrict__ status,
                                                     float* __restrict__ dCall, float sc) {
  extern __shared__ __align__(16) float w_sm[];  // A1, A2, then 32 rows of Bt and SC at a time
  const int tid = threadIdx.x, q = p * p;
  float *a1 = w_sm, *a2 = a1 + q, *bt = a2 + q, *st = bt + 32 * p;
  const float* A = Aall + (size_t)blockIdx.y * 2 * q;
  for (int e = tid; e < 2 * q; e += WT) a1[e] = A[e];
  const bool ok = status[blockIdx.y] == 0;
  const int64_t off = (int64_t)blockIdx.y * m * p;
  const int r0 = blockIdx.x * WR, r1 = min(m, r0 + WR);
  for (int b0 = r0; b0 < r1; b0 += 32) {
    const int cnt = min(32, r1 - b0) * p;
    __syncthreads();
    for (int e = tid; e < cnt; e += WT) {
      bt[e] = Btall[off + (int64_t)b0 * p + e];
      st[e] = SCall[off + (int64_t)b0 * p + e];
    }
    __syncthreads();
    // a thread forms 4 rows of one column: each value of A1, A2 read serves four
    const int RG = WT / p, c = tid % p, rows = min(32, r1 - b0);
    if (tid < RG * p)
      for (int r = tid / p; r < rows; r += 4 * RG) {
        int o[4];
        float a[4];
#pragma unroll
        for (int z = 0; z < 4; ++z) {
          o[z] = min(r + z * RG, rows - 1) * p;
          a[z] = 0.f;
        }
        for (int k = 0; k < p; ++k) {
          const float v = a1[k * p + c];
#pragma unroll
          for (int z = 0; z < 4; ++z) a[z] = fmaf(bt[o[z] + k], v, a[z]);
        }
        for (int k = 0; k < p; ++k) {
          const float v = a2[k * p + c];
#pragma unroll
          for (int z = 0; z < 4; ++z) a[z] = fmaf(-st[o[z] + k], v, a[z]);
        }
#pragma unroll
        for (int z = 0; z < 4; ++z)
          if (r + z * RG < rows) dCall[off + (int64_t)b0 * p + o[z] + c] = ok ? sc * a[z] : 0.f;
      }
  }
}

size_t warm_alg_smem(int p) { return ((size_t)5 * p * p + p) * sizeof(double); }
size_t warm_gram_smem(int p) { return (size_t)3 * WR * ((p + 3) & ~3) * sizeof(float); }
size_t warm_dc_smem(int p) { return ((size_t)2 * p * p + 64 * p) * sizeof(float); }
// partial Grams (float64), then A1 and A2 and the status of every sample
size_t warm_ws_bytes(int batch, int m, int p) {
  const size_t nblk = (m + WR - 1) / WR, q = (size_t)p * p;
  return (size_t)batch * (nblk * 2 * q * sizeof(double) + 2 * q * sizeof(float) + sizeof(int32_t));
}

}  // namespace
}  // namespace gsi

using namespace gsi;

// parameters, flat: W1 (hid x din), b1, W2 (hid x hid), b2, W3 (dout x hid), b3
struct gsi_mlp {
  int din = 0, hid = 0, dout = 0, max_batch = 0;
  int64_t np = 0, step = 0;
  cudaStream_t st = nullptr;
  float *w = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;
  float *h1 = nullptr, *h2 = nullptr, *out = nullptr, *d1 = nullptr, *d2 = nullptr, *dout_buf = nullptr;
  float* sc_buf = nullptr;
  void* loss_ws = nullptr;  // scratch of the loss, sized for the largest (batch, m, p) so far
  size_t loss_ws_bytes = 0;
  double* loss = nullptr;
  double* hloss = nullptr;  // pinned
  std::vector<void*> allocs;
  float* W1() const { return w; }
  float* b1() const { return w + (int64_t)hid * din; }
  float* W2() const { return b1() + hid; }
  float* b2() const { return W2() + (int64_t)hid * hid; }
  float* W3() const { return b2() + hid; }
  float* b3() const { return W3() + (int64_t)dout * hid; }
  // the same offsets into the gradient
  float* gof(const float* p) const { return g + (p - w); }
};

namespace {

gsi_status gemm(cudaStream_t st, int M, int N, int K, const float* A, int64_t sai, int64_t sak,
                const float* B, int64_t sbk, int64_t sbj, float* C, int64_t ldc, float alpha, float beta,
                const float* bias, const float* mask, int relu) {
  if (M <= 0 || N <= 0) return GSI_OK;
  auto mode = [](const float* X, int64_t si, int64_t sk) {
    if (((uintptr_t)X & 15) != 0) return (int)G_ANY;
    if (sk == 1 && (si & 3) == 0) return (int)G_K16;
    if (si == 1 && (sk & 3) == 0) return (int)G_I16;
    return (int)G_ANY;
  };
  const int ma = mode(A, sai, sak), mb = mode(B, sbj, sbk);
  // 64 x 64 tiles read each operand least often; with fewer of them than SMs
  // the 32 x 32 ones spread the reads over four times as many
  const bool big = (int64_t)((N + 63) / 64) * ((M + 63) / 64) >= sm_count();
  const int T = big ? 64 : 32;
  const size_t sm = (size_t)8 * (big ? GStage<64>::FLOATS : GStage<32>::FLOATS) * sizeof(float);
  dim3 grid((unsigned)((N + T - 1) / T), (unsigned)((M + T - 1) / T));
  auto kern = big ? gemm_bf16_kernel<64> : gemm_bf16_kernel<32>;
  GSI_CUDA_TRY(ensure_dyn_smem((const void*)kern, (int)sm));
  kern<<<grid, 128, sm, st>>>(M, N, K, A, sai, sak, ma, B, sbk, sbj, mb, C, ldc, alpha, beta, bias, mask, relu);
  GSI_LAUNCH_CHECK();
  return GSI_OK;
}

gsi_status malloc_t(gsi_mlp* n, void** p, size_t bytes) {
  cudaError_t e = cudaMalloc(p, std::max<size_t>(bytes, 256));
  if (e != cudaSuccess) return cuda_status(e);
  n->allocs.push_back(*p);
  return GSI_OK;
}

// forward with the activations kept for backward
gsi_status mlp_forward(gsi_mlp* n, int batch, const float* x, float* out) {
  const int H = n->hid;
  GSI_TRY(gemm(n->st, batch, H, n->din, x, n->din, 1, n->W1(), 1, n->din, n->h1, H, 1.f, 0.f, n->b1(),
               nullptr, 1));
  GSI_TRY(gemm(n->st, batch, H, H, n->h1, H, 1, n->W2(), 1, H, n->h2, H, 1.f, 0.f, n->b2(), nullptr, 1));
  GSI_TRY(gemm(n->st, batch, n->dout, H, n->h2, H, 1, n->W3(), 1, H, out, n->dout, 1.f, 0.f, n->b3(),
               nullptr, 0));
  return GSI_OK;
}

// gradients of sum(out * dout) for the batch of the last forward
gsi_status mlp_backward(gsi_mlp* n, int batch, const float* x, const float* dout) {
  const int H = n->hid, D = n->dout;
  cudaStream_t st = n->st;
  // W3: dout^T h2; b3: column sums of dout
  GSI_TRY(gemm(st, D, H, batch, dout, 1, D, n->h2, H, 1, n->gof(n->W3()), H, 1.f, 0.f, nullptr, nullptr, 0));
  colsum_kernel<<<ceil_div(D, 256), 256, 0, st>>>(batch, D, dout, n->gof(n->b3()));
  GSI_LAUNCH_CHECK();
  // d2 = (dout W3) o [h2 > 0]
  GSI_TRY(gemm(st, batch, H, D, dout, D, 1, n->W3(), H, 1, n->d2, H, 1.f, 0.f, nullptr, n->h2, 0));
  GSI_TRY(gemm(st, H, H, batch, n->d2, 1, H, n->h1, H, 1, n->gof(n->W2()), H, 1.f, 0.f, nullptr, nullptr, 0));
  colsum_kernel<<<ceil_div(H, 256), 256, 0, st>>>(batch, H, n->d2, n->gof(n->b2()));
  GSI_LAUNCH_CHECK();
  // d1 = (d2 W2) o [h1 > 0]
  GSI_TRY(gemm(st, batch, H, H, n->d2, H, 1, n->W2(), H, 1, n->d1, H, 1.f, 0.f, nullptr, n->h1, 0));
  GSI_TRY(gemm(st, H, n->din, batch, n->d1, 1, H, x, n->din, 1, n->gof(n->W1()), n->din, 1.f, 0.f, nullptr,
               nullptr, 0));
  colsum_kernel<<<ceil_div(H, 256), 256, 0, st>>>(batch, H, n->d1, n->gof(n->b1()));
  GSI_LAUNCH_CHECK();
  return GSI_OK;
}

gsi_status mlp_adam(gsi_mlp* n, double lr, double b1, double b2, double eps) {
  n->step++;
  const double c1 = 1.0 / (1.0 - pow(b1, (double)n->step));
  const double c2 = 1.0 / (1.0 - pow(b2, (double)n->step));
  adam_kernel<<<ceil_div(n->np, 256), 256, 0, n->st>>>(n->np, n->w, n->g, n->m, n->v, (float)lr, (float)b1,
                                                       (float)b2, (float)eps, (float)c1, (float)c2);
  GSI_LAUNCH_CHECK();
  return GSI_OK;
}

// ws: warm_ws_bytes(batch, m, p) bytes of device memory
gsi_status loss_grad(int batch, int m, int p, const int64_t* Srp, const int32_t* Sci, const double* Sv,
                     const float* C, const float* Bt, float* SC, double* loss, float* dC, float gscale,
                     void* ws, cudaStream_t st) {
  if (batch <= 0) return GSI_OK;
  const int nblk = (m + WR - 1) / WR;
  double* part = reinterpret_cast<double*>(ws);
  float* A = reinterpret_cast<float*>(part + (size_t)batch * nblk * 2 * p * p);
  int32_t* status = reinterpret_cast<int32_t*>(A + (size_t)batch * 2 * p * p);
  GSI_CUDA_TRY(ensure_dyn_smem((const void*)warm_gram_kernel, (int)warm_gram_smem(p)));
  GSI_CUDA_TRY(ensure_dyn_smem((const void*)warm_alg_kernel, (int)warm_alg_smem(p)));
  GSI_CUDA_TRY(ensure_dyn_smem((const void*)warm_dc_kernel, (int)warm_dc_smem(p)));
  // samples go in the grid's second dimension, at most 65,535 at a time
  for (int b0 = 0; b0 < batch; b0 += 65535) {
    const int nb = std::min(batch - b0, 65535);
    const size_t o = (size_t)b0 * m * p;
    double* pt = part + (size_t)b0 * nblk * 2 * p * p;
    float* Ab = A + (size_t)b0 * 2 * p * p;
    warm_gram_kernel<<<dim3(nblk, nb), WT, warm_gram_smem(p), st>>>(m, p, Srp, Sci, Sv, C + o, Bt + o, SC + o, pt);
    GSI_LAUNCH_CHECK();
    warm_alg_kernel<<<nb, WT, warm_alg_smem(p), st>>>(p, nblk, pt, loss + b0, Ab, status + b0);
    GSI_LAUNCH_CHECK();
    warm_dc_kernel<<<dim3(nblk, nb), WT, warm_dc_smem(p), st>>>(m, p, Bt + o, SC + o, Ab, status + b0, dC + o,
                                                               -2.f * gscale);
    GSI_LAUNCH_CHECK();
  }
  return GSI_OK;
}

}  // namespace

extern "C" {

int64_t gsi_mlp_num_params(int32_t din, int32_t hidden, int32_t dout) {
  return (int64_t)hidden * din + hidden + (int64_t)hidden * hidden + hidden + (int64_t)dout * hidden + dout;
}

gsi_status gsi_mlp_destroy(gsi_mlp* n) {
  if (!n) return GSI_ERR_ARG;
  if (n->st) cudaStreamSynchronize(n->st);
  for (void* p : n->allocs) cudaFree(p);
  if (n->loss_ws) cudaFree(n->loss_ws);
  if (n->hloss) cudaFreeHost(n->hloss);
  delete n;
  return GSI_OK;
}

gsi_status gsi_mlp_create(int32_t din, int32_t hidden, int32_t dout, int32_t max_batch, const float* params,
                          void* stream, gsi_mlp** out) {
  if (!out || !params || din < 1 || hidden < 1 || dout < 1 || max_batch < 1) return GSI_ERR_ARG;
  *out = nullptr;
  gsi_mlp* n = new gsi_mlp();
  n->din = din;
  n->hid = hidden;
  n->dout = dout;
  n->max_batch = max_batch;
  n->st = (cudaStream_t)stream;
  n->np = gsi_mlp_num_params(din, hidden, dout);
  const size_t pb = (size_t)n->np * sizeof(float);
  const size_t hb = (size_t)max_batch * hidden * sizeof(float);
  const size_t ob = (size_t)max_batch * dout * sizeof(float);
  gsi_status s = GSI_OK;
#define CK(expr)                \
  do {                          \
    s = (expr);                 \
    if (s != GSI_OK) goto fail; \
  } while (0)
  CK(malloc_t(n, (void**)&n->w, pb));
  CK(malloc_t(n, (void**)&n->g, pb));
  CK(malloc_t(n, (void**)&n->m, pb));
  CK(malloc_t(n, (void**)&n->v, pb));
  CK(malloc_t(n, (void**)&n->h1, hb));
  CK(malloc_t(n, (void**)&n->h2, hb));
  CK(malloc_t(n, (void**)&n->d1, hb));
  CK(malloc_t(n, (void**)&n->d2, hb));
  CK(malloc_t(n, (void**)&n->out, ob));
  CK(malloc_t(n, (void**)&n->dout_buf, ob));
  CK(malloc_t(n, (void**)&n->sc_buf, ob));
  CK(malloc_t(n, (void**)&n->loss, (size_t)max_batch * sizeof(double)));
  CK(cuda_status_ok(cudaMallocHost((void**)&n->hloss, (size_t)max_batch * sizeof(double))));
  CK(cuda_status_ok(cudaMemcpy(n->w, params, pb, cudaMemcpyHostToDevice)));
  CK(cuda_status_ok(cudaMemset(n->g, 0, pb)));
  CK(cuda_status_ok(cudaMemset(n->m, 0, pb)));
  CK(cuda_status_ok(cudaMemset(n->v, 0, pb)));
#undef CK
  *out = n;
  return GSI_OK;
fail:
  gsi_mlp_destroy(n);
  return s;
}

gsi_status gsi_mlp_get_params(gsi_mlp* n, float* params, float* grads) {
  if (!n) return GSI_ERR_ARG;
  GSI_CUDA_TRY(cudaStreamSynchronize(n->st));
  if (params) GSI_CUDA_TRY(cudaMemcpy(params, n->w, (size_t)n->np * sizeof(float), cudaMemcpyDeviceToHost));
  if (grads) GSI_CUDA_TRY(cudaMemcpy(grads, n->g, (size_t)n->np * sizeof(float), cudaMemcpyDeviceToHost));
  return GSI_OK;
}

gsi_status gsi_mlp_forward(gsi_mlp* n, int32_t batch, const float* x, float* out) {
  if (!n || !x || !out || batch < 1 || batch > n->max_batch) return GSI_ERR_ARG;
  return mlp_forward(n, batch, x, out);
}

gsi_status gsi_mlp_backward(gsi_mlp* n, int32_t batch, const float* x, const float* dout) {
  if (!n || !x || !dout || batch < 1 || batch > n->max_batch) return GSI_ERR_ARG;
  return mlp_backward(n, batch, x, dout);
}

gsi_status gsi_mlp_adam(gsi_mlp* n, double lr, double beta1, double beta2, double eps) {
  if (!n || !(lr > 0.0)) return GSI_ERR_ARG;
  return mlp_adam(n, lr, beta1, beta2, eps);
}

gsi_status gsi_warm_loss_grad(int32_t batch, int32_t m, int32_t p, const int64_t* S_rowptr,
                              const int32_t* S_colidx, const double* S_val, const float* C, const float* Bt,
                              float* SC_scratch, double* loss, float* dC, float gscale, void* stream) {
  if (batch < 1 || m < 1 || p < 1 || p > 64 || !S_rowptr || !S_colidx || !S_val || !C || !Bt ||
      !SC_scratch || !loss || !dC)
    return GSI_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  void* ws = nullptr;
  GSI_CUDA_TRY(cudaMallocAsync(&ws, warm_ws_bytes(batch, m, p), st));
  const gsi_status s = loss_grad(batch, m, p, S_rowptr, S_colidx, S_val, C, Bt, SC_scratch, loss, dC, gscale, ws, st);
  const cudaError_t fe = cudaFreeAsync(ws, st);
  GSI_TRY(s);
  GSI_CUDA_TRY(fe);
  return GSI_OK;
}

gsi_status gsi_warm_train_step(gsi_mlp* n, int32_t batch, const float* x, int32_t m, int32_t p,
                               const int64_t* S_rowptr, const int32_t* S_colidx, const double* S_val,
                               const float* Bt, double lr, double* mean_loss) {
  if (!n || !x || !Bt || batch < 1 || batch > n->max_batch || p < 1 || p > 64 || (int64_t)m * p != n->dout)
    return GSI_ERR_ARG;
  // a captured step gets a buffer of the graph's own: the kept one is
  // replaced by a later, larger step, which a replay would not learn of
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  GSI_CUDA_TRY(cudaStreamIsCapturing(n->st, &cap));
  const size_t need = warm_ws_bytes(batch, m, p);
  void *ws = nullptr, *tmp = nullptr;
  if (cap != cudaStreamCaptureStatusNone) {
    GSI_CUDA_TRY(cudaMallocAsync(&tmp, need, n->st));
    ws = tmp;
  } else {
    if (need > n->loss_ws_bytes) {  // stream-ordered: earlier steps on n->st may still use the old one
      void* old = n->loss_ws;
      n->loss_ws = nullptr;
      n->loss_ws_bytes = 0;
      if (old) GSI_CUDA_TRY(cudaFreeAsync(old, n->st));
      GSI_CUDA_TRY(cudaMallocAsync(&n->loss_ws, need, n->st));
      n->loss_ws_bytes = need;
    }
    ws = n->loss_ws;
  }
  gsi_status ls = mlp_forward(n, batch, x, n->out);
  if (ls == GSI_OK)
    ls = loss_grad(batch, m, p, S_rowptr, S_colidx, S_val, n->out, Bt, n->sc_buf, n->loss, n->dout_buf, 1.f / batch,
                   ws, n->st);
  const cudaError_t fe = tmp ? cudaFreeAsync(tmp, n->st) : cudaSuccess;
  GSI_TRY(ls);
  GSI_CUDA_TRY(fe);
  GSI_TRY(mlp_backward(n, batch, x, n->dout_buf));
  GSI_TRY(mlp_adam(n, lr, 0.9, 0.999, 1e-8));
  if (mean_loss) {
    GSI_CUDA_TRY(cudaMemcpyAsync(n->hloss, n->loss, (size_t)batch * sizeof(double), cudaMemcpyDeviceToHost,
                                 n->st));
    GSI_CUDA_TRY(cudaStreamSynchronize(n->st));
    double s = 0.0;
    for (int i = 0; i < batch; ++i) s += n->hloss[i];
    *mean_loss = s / batch;
  }
  return GSI_OK;
}

gsi_status gsi_prolong(int32_t nc, int32_t nf, int32_t p, int32_t batch, const float* C, double* X,
                       void* stream) {
  if (nc < 1 || nf < 1 || p < 1 || batch < 1 || !C || !X) return GSI_ERR_ARG;
  const int64_t total = (int64_t)batch * nf * nf * p;
  prolong_kernel<<<ceil_div(total, 256), 256, 0, (cudaStream_t)stream>>>(nc, nf, p, batch, C, X);
  GSI_LAUNCH_CHECK();
  return GSI_OK;
}

gsi_status gsi_restrict(int32_t nc, int32_t nf, int32_t p, int32_t batch, const double* U, float* Bt,
                        void* stream) {
  if (nc < 1 || nf < 1 || p < 1 || batch < 1 || !U || !Bt) return GSI_ERR_ARG;
  const int64_t total = (int64_t)batch * nc * nc * p;
  restrict_kernel<<<ceil_div(total, 256), 256, 0, (cudaStream_t)stream>>>(nc, nf, p, batch, U, Bt);
  GSI_LAUNCH_CHECK();
  return GSI_OK;
}

gsi_status gsi_gemm_bf16(int32_t M, int32_t N, int32_t K, const float* A, int64_t sai, int64_t sak,
                         const float* B, int64_t sbk, int64_t sbj, float* C, int64_t ldc, float alpha,
                         float beta, const float* bias, const float* mask, int32_t relu, void* stream) {
  if (M < 0 || N < 0 || K < 0 || !A || !B || !C) return GSI_ERR_ARG;
  return gemm((cudaStream_t)stream, M, N, K, A, sai, sak, B, sbk, sbj, C, ldc, alpha, beta, bias, mask, relu);
}

}  // extern "C"
