// Device code of the p x p step (Alg. 3 and the polar normaliser) for one
// thread block or one thread-block cluster per problem, all matrices df64.
//
// Eigenbasis of a symmetric B: float32 Jacobi sweeps give V0; V is made
// orthonormal in df64; then B' = V^T B V = diag(lambda) + F is formed in df64
// and the small F rotated away by the same float32 Jacobi, which works on F
// and on df64 differences of lambda, so that its float32 rounding is relative
// to F: each such pass gains six to seven digits (F 1e-6 -> 1e-13 of ||B||).
// The rotations of a pass are gathered in one matrix, applied in df64. Against
// df64 Jacobi sweeps this trades the serial rounds of ~400 float operations a
// 2 x 2 block for df64 products, which have no chain between rounds.
//
// Layout of the work. A Jacobi round is one barrier for the angles (one
// thread per rotation), one for the 2 x 2 blocks of J^T A J (one thread per
// unordered pair of rotations: A is symmetric, both halves are stored); the
// update of V by a round's rotations runs beside the next round's angles.
// Products give every thread a TR x TC register tile. With NC > 1 CTAs the
// matrices live in global memory (L2), each CTA forms p / NC rows of every
// product from copies in its shared memory, and rank 0 alone runs the
// sweeps; the CTAs meet at cluster barriers.
#pragma once
#include <math.h>

#include "alg3.cuh"
#include "df.cuh"

namespace gsi {

// Block shape: NT threads; a group of CL lanes covers TC CL columns of a
// product (NCG such column blocks), the groups its rows, TR each. MI: 2 x 2
// blocks a thread holds in a Jacobi round (half (half - 1) / 2 of them).
template <int NT_, int CL_, int TR_, int TC_, int NCG_, int MI_, int NC_>
struct PpCfg {
  static constexpr int NT = NT_, CL = CL_, TR = TR_, TC = TC_, NCG = NCG_, MI = MI_, NC = NC_;
  static constexpr int NG = NT / CL, RG = NG / NCG;
};

struct PpMat {  // a p x p input: df64, or float64 (then symmetrised where sym is set)
  const float2* f;
  const double* d;
  int sym;
};

struct PpArgs {
  int mode, p;
  // B = D^T D (modes 0, 3) or the matrix itself (modes 1, 2); C = X^T A X,
  // Gam = D^T W, Z = D^T R, XX = X^T X; XD = X^T D, or null pointers: formed
  // here as (I - XX)(C + beta K)
  PpMat C, B, Gam, Z, XX, XD, K;
  double beta;
  double* M;      // p x p result (eigenvectors in mode 2)
  double* Kd;     // K_next = M (XD + t B), float64 (or null)
  float2* Kf;     // and df64 (or null)
  double* theta;  // mode 2: eigenvalues
  float2* eig;    // modes 3, 4: V (p x p), then the diagonal of V^T B V
  double* out;    // 16 doubles: t, phi, evaluations, status, max beta, cycle counts and sweeps
  float2* gws;    // NC > 1: 4 p x p matrices and PP_CTL float2 of global scratch
};
constexpr int PP_CTL = 1024 + 64;  // float2: partial dots of up to 8 ranks, then the control words

struct PpSh {  // small tables, shared memory
  double al[128], be[128], ga[128], ze[128], sv[128];
  float2 lam[130];
  float2 cs[2][64];
  float red[32];
  double t;
  int flag, ctl;
};

template <class P>
struct PpCtx {
  int p, ld, tid, cl, g, rank, r0, r1;
  float2 *Bd, *Vd, *Td, *Ud;  // p x p df64, rows ld apart (shared memory; global for NC > 1)
  float *Af, *Vf;             // Jacobi matrices, rows lda apart (shared memory)
  int lda;
  float2 *sX, *sY;            // NC > 1: the strip of X and the whole Y of a product
  float2* ctl;                // NC > 1: control words in global memory
  PpSh* sh;
};

__host__ __device__ inline int pp_lda(int p) { return (p + 31) / 32 * 32; }
__host__ __device__ inline size_t pp_al(size_t b) { return (b + 15) & ~(size_t)15; }
// dynamic shared memory: NC = 1: four df64 matrices and the two Jacobi
// matrices; NC > 1: staged Y (the Jacobi matrices share its space), strip of
// X, float32 copy of E
inline size_t pp_smem(int p, int nc) {
  const size_t ld = p | 1, m = (p + 1) & ~1, lda = pp_lda((int)m);
  const size_t jac = 2 * pp_al(m * lda * sizeof(float));
  if (nc == 1) return 4 * pp_al((size_t)p * ld * sizeof(float2)) + jac;
  const size_t sy = pp_al((size_t)p * ld * sizeof(float2));
  return (sy > jac ? sy : jac) + pp_al((size_t)((p + nc - 1) / nc) * ld * sizeof(float2)) +
         pp_al(m * lda * sizeof(float));
}
inline size_t pp_gws_bytes(int p) { return (4 * (size_t)p * p + PP_CTL) * sizeof(float2); }

template <class P>
__device__ __forceinline__ void pp_sync() {
  if constexpr (P::NC == 1) {
    __syncthreads();
  } else {
    asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
  }
}

template <class P>
__device__ __forceinline__ float2 pp_ld(const float2* p) {
  if constexpr (P::NC == 1) return *p;
  else return __ldcg(p);
}

template <class P>
__device__ PpCtx<P> pp_ctx(unsigned char* sm, PpSh* sh, int p, float2* gws) {
  PpCtx<P> c;
  c.p = p;
  c.tid = threadIdx.x;
  c.cl = c.tid % P::CL;
  c.g = c.tid / P::CL;
  c.sh = sh;
  const int m = (p + 1) & ~1;
  c.lda = pp_lda(m);
  unsigned char* cur = sm;
  auto take = [&](size_t b) {
    unsigned char* r = cur;
    cur += pp_al(b);
    return r;
  };
  if constexpr (P::NC == 1) {
    c.rank = 0;
    c.r0 = 0;
    c.r1 = p;
    c.ld = p | 1;
    const size_t mb = (size_t)p * c.ld * sizeof(float2);
    c.Bd = (float2*)take(mb);
    c.Vd = (float2*)take(mb);
    c.Td = (float2*)take(mb);
    c.Ud = (float2*)take(mb);
    c.Af = (float*)take((size_t)m * c.lda * sizeof(float));
    c.Vf = (float*)take((size_t)m * c.lda * sizeof(float));
    c.sX = c.sY = c.ctl = nullptr;
  } else {
    uint32_t rk;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rk));
    c.rank = (int)rk;
    const int rs = (p + P::NC - 1) / P::NC;
    c.r0 = min(p, c.rank * rs);
    c.r1 = min(p, c.r0 + rs);
    c.ld = p;
    const size_t q = (size_t)p * p;
    c.Bd = gws;
    c.Vd = gws + q;
    c.Td = gws + 2 * q;
    c.Ud = gws + 3 * q;
    c.ctl = gws + 4 * q;
    const size_t jac = pp_al((size_t)m * c.lda * sizeof(float));
    const size_t sy = pp_al((size_t)p * (p | 1) * sizeof(float2));
    unsigned char* y = take(sy > 2 * jac ? sy : 2 * jac);
    c.sY = (float2*)y;
    c.Vf = (float*)(y + jac);
    c.sX = (float2*)take((size_t)rs * (p | 1) * sizeof(float2));
    // the Jacobi matrix of rank 0 and every rank's copy of E share this
    c.Af = (float*)take((size_t)m * c.lda * sizeof(float));
  }
  return c;
}

// f(i, j) over this CTA's rows of a p x p matrix
template <class P, class F>
__device__ __forceinline__ void pp_each(const PpCtx<P>& c, F f) {
  for (int i = c.r0 + c.g; i < c.r1; i += P::NG)
    for (int j = c.cl; j < c.p; j += P::CL) f(i, j);
}

__device__ __forceinline__ float2 pp_neg(float2 a) { return make_float2(-a.x, -a.y); }

// acc += a b (df64): leading product and sum exact, second order in the low word
__device__ __forceinline__ void pp_mac(float& sh, float& se, float2 a, float2 b) {
  const float pr = __fmul_rn(a.x, b.x);
  const float pe = __fmaf_rn(a.x, b.x, -pr);
  const float2 t = two_sum(sh, pr);
  sh = t.x;
  se = __fadd_rn(se, __fadd_rn(t.y, __fmaf_rn(a.x, b.y, __fmaf_rn(a.y, b.x, pe))));
}

// Rows r0..r1 of X' Y', X' = X^T if tx, Y' = Y^T if ty. With dots null:
// Out = (Add +) X' Y' - dsub I. With dots: dots[g p + j] += sum over this
// group's rows i of Vdot[i, j] (X' Y')[i, j] (df64 pairs, one row of dots per
// row group). The caller synchronises before and after. One copy of the code
// serves every product of a step (the instruction cache is cold at each
// launch).
template <class P>
__device__ __noinline__ void pp_mm(const PpCtx<P>& c, const float2* X, bool tx, const float2* Y, bool ty,
                                   float2* Out, const float2* Add, float dsub, const float2* Vdot = nullptr,
                                   float2* dots = nullptr) {
  const int p = c.p, rows = c.r1 - c.r0;
  const float2 *xs, *ys;
  int xi, xk, yk, yj;
  if constexpr (P::NC == 1) {
    xs = X;
    ys = Y;
    xi = tx ? 1 : c.ld;
    xk = tx ? c.ld : 1;
    yk = ty ? 1 : c.ld;
    yj = ty ? c.ld : 1;
  } else {
    const int ls = p | 1;
    for (int k = c.g; k < p; k += P::NG)
      for (int j = c.cl; j < p; j += P::CL) {
        const float2 v = __ldcg(Y + k * p + j);
        c.sY[ty ? j * ls + k : k * ls + j] = v;
      }
    if (tx) {
      for (int e = c.tid; e < rows * p; e += P::NT) {
        const int k = e / rows, i = e - k * rows;
        c.sX[i * ls + k] = __ldcg(X + k * p + c.r0 + i);
      }
    } else {
      for (int i = c.g; i < rows; i += P::NG)
        for (int k = c.cl; k < p; k += P::CL) c.sX[i * ls + k] = __ldcg(X + (c.r0 + i) * p + k);
    }
    __syncthreads();
    xs = c.sX;
    ys = c.sY;
    xi = ls;
    xk = 1;
    yk = ls;
    yj = 1;
  }
  const int rg = P::NCG == 1 ? c.g : c.g / P::NCG;
  const int jb = (P::NCG == 1 ? 0 : c.g % P::NCG) * (P::CL * P::TC) + c.cl;
  const float2* yp[P::TC];
#pragma unroll
  for (int t = 0; t < P::TC; ++t) yp[t] = ys + min(jb + t * P::CL, p - 1) * yj;
  float2 dacc[P::TC];
#pragma unroll
  for (int t = 0; t < P::TC; ++t) dacc[t] = make_float2(0.f, 0.f);
  for (int i0 = rg * P::TR; i0 < rows; i0 += P::RG * P::TR) {
    float h[P::TR][P::TC], e[P::TR][P::TC];
    const float2* xp[P::TR];
#pragma unroll
    for (int s = 0; s < P::TR; ++s) {
      xp[s] = xs + min(i0 + s, rows - 1) * xi;
#pragma unroll
      for (int t = 0; t < P::TC; ++t) h[s][t] = e[s][t] = 0.f;
    }
#pragma unroll 2
    for (int k = 0; k < p; ++k) {
      float2 x[P::TR], y[P::TC];
#pragma unroll
      for (int s = 0; s < P::TR; ++s) x[s] = xp[s][k * xk];
#pragma unroll
      for (int t = 0; t < P::TC; ++t) y[t] = yp[t][k * yk];
#pragma unroll
      for (int s = 0; s < P::TR; ++s)
#pragma unroll
        for (int t = 0; t < P::TC; ++t) pp_mac(h[s][t], e[s][t], x[s], y[t]);
    }
#pragma unroll
    for (int s = 0; s < P::TR; ++s)
#pragma unroll
      for (int t = 0; t < P::TC; ++t) {
        const int i = c.r0 + i0 + s, j = jb + t * P::CL;
        if (i0 + s < rows && j < p) {
          float2 v = fast_two_sum(h[s][t], e[s][t]);
          if (dots) {
            pp_mac(dacc[t].x, dacc[t].y, pp_ld<P>(Vdot + i * c.ld + j), v);
          } else {
            if (i == j && dsub != 0.f) v = df_add_f(v, -dsub);
            if (Add) v = df_add(pp_ld<P>(Add + i * c.ld + j), v);
            Out[i * c.ld + j] = v;
          }
        }
      }
  }
  if (dots) {
#pragma unroll
    for (int t = 0; t < P::TC; ++t) {
      const int j = jb + t * P::CL;
      if (j < p) dots[rg * p + j] = fast_two_sum(dacc[t].x, dacc[t].y);
    }
  }
}

// sum over the block (float32, fixed order), the same in every thread
template <class P>
__device__ float pp_bsum(PpSh* sh, float v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh->red[threadIdx.x >> 5] = v;
  __syncthreads();
  float s = 0.f;
#pragma unroll
  for (int w = 0; w < P::NT / 32; ++w) s += sh->red[w];
  return s;
}

template <class P>
__device__ float pp_bmax(PpSh* sh, float v) {
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh->red[threadIdx.x >> 5] = v;
  __syncthreads();
  float s = 0.f;
#pragma unroll
  for (int w = 0; w < P::NT / 32; ++w) s = fmaxf(s, sh->red[w]);
  return s;
}

// Round-robin ordering of m (even) indices: in round r slot 0 pairs r with
// m - 1, slot k pairs r + k and r - k modulo m - 1.
__device__ __forceinline__ void pp_pair(int r, int k, int m1, int& a, int& b) {
  if (k == 0) {
    a = r;
    b = m1;
  } else {
    a = r + k;
    a -= a >= m1 ? m1 : 0;
    b = r - k;
    b += b < 0 ? m1 : 0;
  }
}

// Jacobi sweeps in float32 by one CTA on the symmetric m x m matrix A (m = p
// rounded up to even; the dummy row and column of an odd p are zero and stay
// so), rotations gathered in V (p rows) on the right, until the squared
// off-diagonal mass is at most `stop`. DELTA: A holds only the off-diagonal
// part (zero diagonal) and lam the df64 diagonal.
template <class P, bool DELTA>
__device__ int pp_jacobi(const PpCtx<P>& c, int max_sweeps, float stop) {
  const int p = c.p, lda = c.lda, tid = c.tid;
  const int m = (p + 1) & ~1, half = m / 2, m1 = m - 1;
  float* const A = c.Af;
  float* const V = c.Vf;
  float2* const lam = c.sh->lam;
  const int items = half * (half - 1) / 2;
  int ik[P::MI], il[P::MI];
#pragma unroll
  for (int z = 0; z < P::MI; ++z) {
    const int e = tid + z * P::NT;
    ik[z] = -1;
    il[z] = 0;
    if (e < items) {
      const int d = e / half;  // partner distance d + 1
      ik[z] = e - d * half;
      il[z] = ik[z] + d + 1;
      il[z] -= il[z] >= half ? half : 0;
    }
  }
  auto update_v = [&](int r, const float2* cs) {
    for (int l = c.cl; l < half; l += P::CL) {
      int a, b;
      pp_pair(r, l, m1, a, b);
      const float2 w = cs[l];
      for (int row = c.g; row < p; row += P::NG) {
        const float x = V[row * lda + a], y = V[row * lda + b];
        V[row * lda + a] = w.x * x - w.y * y;
        V[row * lda + b] = w.y * x + w.x * y;
      }
    }
  };
  int sweep = 0;
  for (; sweep < max_sweeps; ++sweep) {
    float off = 0.f;
    for (int i = c.g; i < p; i += P::NG)
      for (int j = c.cl; j < p; j += P::CL)
        if (i != j) off += A[i * lda + j] * A[i * lda + j];
    off = pp_bsum<P>(c.sh, off);
    if (!(off > stop)) break;
    for (int r = 0; r < m1; ++r) {
      float2* const cs = c.sh->cs[r & 1];
      if (tid < half) {
        int a, b;
        pp_pair(r, tid, m1, a, b);
        const float f = A[a * lda + b];
        float t = 0.f;
        if (DELTA) {
          const float2 la = lam[a], lb = lam[b];
          const float2 dd = df_add(lb, pp_neg(la));
          const float d = __fadd_rn(dd.x, dd.y), b2 = 2.f * f;
          const float q = __fsqrt_rn(__fmaf_rn(d, d, b2 * b2));
          if (q > 0.f) t = __fdiv_rn(d >= 0.f ? b2 : -b2, fabsf(d) + q);
          const float x = t * f;
          lam[a] = df_add_f(la, -x);
          lam[b] = df_add_f(lb, x);
        } else {
          const float aa = A[a * lda + a], ab = A[b * lda + b];
          const float d = ab - aa, b2 = 2.f * f;
          const float q2 = __fmaf_rn(d, d, b2 * b2);
          if (q2 > 0.f) t = __fdividef(d >= 0.f ? b2 : -b2, fabsf(d) + q2 * rsqrtf(q2));
          const float x = t * f;
          A[a * lda + a] = aa - x;
          A[b * lda + b] = ab + x;
        }
        A[a * lda + b] = 0.f;
        A[b * lda + a] = 0.f;
        const float q = __fmaf_rn(t, t, 1.f);
        float cc = rsqrtf(q);
        cc = cc * __fmaf_rn(-0.5f * q, cc * cc, 1.5f);  // one Newton step: c^2 + s^2 = 1 to rounding
        cs[tid] = make_float2(cc, t * cc);
      }
      if (r > 0) update_v(r - 1, c.sh->cs[(r - 1) & 1]);
      __syncthreads();
#pragma unroll
      for (int z = 0; z < P::MI; ++z) {
        if (ik[z] >= 0) {
          int ak, bk, al, bl;
          pp_pair(r, ik[z], m1, ak, bk);
          pp_pair(r, il[z], m1, al, bl);
          const float2 wk = cs[ik[z]], wl = cs[il[z]];
          const float x00 = A[ak * lda + al], x01 = A[ak * lda + bl];
          const float x10 = A[bk * lda + al], x11 = A[bk * lda + bl];
          const float y00 = wl.x * x00 - wl.y * x01, y01 = wl.y * x00 + wl.x * x01;
          const float y10 = wl.x * x10 - wl.y * x11, y11 = wl.y * x10 + wl.x * x11;
          const float z00 = wk.x * y00 - wk.y * y10, z10 = wk.y * y00 + wk.x * y10;
          const float z01 = wk.x * y01 - wk.y * y11, z11 = wk.y * y01 + wk.x * y11;
          A[ak * lda + al] = z00;
          A[ak * lda + bl] = z01;
          A[bk * lda + al] = z10;
          A[bk * lda + bl] = z11;
          A[al * lda + ak] = z00;
          A[bl * lda + ak] = z01;
          A[al * lda + bk] = z10;
          A[bl * lda + bk] = z11;
        }
      }
      __syncthreads();
    }
    update_v(m1 - 1, c.sh->cs[(m1 - 1) & 1]);
    __syncthreads();
  }
  return sweep;
}

// Out = V (V^T V)^{-1/2} to third order in E = V^T V - I (E of about 1e-6:
// V comes from float32 rotations): Out = V + V G, G = -E/2 + 3/8 E^2, E^2 in
// float32. T is scratch; V is not changed. Synchronised on entry and exit.
template <class P>
__device__ void pp_orth(const PpCtx<P>& c, const float2* V, float2* T, float2* Out) {
  pp_mm(c, V, true, V, false, T, (const float2*)nullptr, 1.f);  // E
  pp_sync<P>();
  for (int i = c.g; i < c.p; i += P::NG)
    for (int j = c.cl; j < c.p; j += P::CL) c.Af[i * c.lda + j] = pp_ld<P>(T + i * c.ld + j).x;
  __syncthreads();
  pp_each(c, [&](int i, int j) {
    float s = 0.f;
    for (int k = 0; k < c.p; ++k) s = fmaf(c.Af[i * c.lda + k], c.Af[k * c.lda + j], s);
    const float2 e = T[i * c.ld + j];
    T[i * c.ld + j] = df_add_f(make_float2(-0.5f * e.x, -0.5f * e.y), 0.375f * s);
  });
  pp_sync<P>();
  pp_mm(c, V, false, T, false, Out, V, 0.f);
  pp_sync<P>();
}

// Eigenbasis of the symmetric c.Bd into c.Vd; c.Ud = V^T B V, diagonal up to
// rounding (`first_order` set: to first order in V -- the last correction of
// V is not put into Ud, whose off-diagonal part is then the corrected one's
// and whose diagonal is exact to second order). B is synchronised on entry.
template <class P>
__device__ void pp_eig(const PpCtx<P>& c, bool first_order, double* diag) {
  const int p = c.p, lda = c.lda, m = (p + 1) & ~1;
  PpSh* sh = c.sh;
  const long long c0 = clock64();
  float sc = 1.f;  // a power of two that brings max |B| near 1 (rank 0)
  int s32 = 0, s_delta = 0;
  auto identity_v = [&]() {
    for (int i = c.g; i < p; i += P::NG)
      for (int j = c.cl; j < m; j += P::CL) c.Vf[i * lda + j] = i == j ? 1.f : 0.f;
  };
  // V of the sweeps into a df64 matrix, and a control word for the other ranks
  auto publish = [&](float2* V, int word) {
    if (c.rank == 0) {
      for (int i = c.g; i < p; i += P::NG)
        for (int j = c.cl; j < p; j += P::CL) V[i * c.ld + j] = make_float2(c.Vf[i * lda + j], 0.f);
      if (c.tid == 0) {
        sh->ctl = word;
        if (P::NC > 1) c.ctl[0] = make_float2(__int_as_float(word), 0.f);
      }
    }
    pp_sync<P>();
    return P::NC == 1 ? sh->ctl : __float_as_int(__ldcg(&c.ctl[0].x));
  };
  if (c.rank == 0) {
    float mx = 0.f, tot = 0.f;
    for (int i = c.g; i < p; i += P::NG)
      for (int j = c.cl; j < p; j += P::CL) mx = fmaxf(mx, fabsf(pp_ld<P>(c.Bd + i * c.ld + j).x));
    mx = pp_bmax<P>(sh, mx);
    const int ex = ((__float_as_int(mx) >> 23) & 255) - 127;
    if (mx > 0.f && ex <= 127) sc = exp2i(max(-126, min(126, -ex)));
    for (int i = c.g; i < m; i += P::NG)
      for (int j = c.cl; j < m; j += P::CL) {
        const float v = i < p && j < p ? pp_ld<P>(c.Bd + i * c.ld + j).x * sc : 0.f;
        c.Af[i * lda + j] = v;
        tot += v * v;
      }
    identity_v();
    tot = pp_bsum<P>(sh, tot);  // (its barriers also publish A and V)
    __syncthreads();
    // down to ~1e-5 relative off-diagonal mass, above float32's rounding floor
    s32 = pp_jacobi<P, false>(c, 12, 1e-10f * tot);
  }
  const bool rotated = publish(c.Td, s32 > 0) != 0;
  const long long c1 = clock64();
  if (rotated) {
    pp_orth(c, c.Td, c.Ud, c.Vd);
    pp_mm(c, c.Bd, false, c.Vd, false, c.Td, (const float2*)nullptr, 0.f);
    pp_sync<P>();
    pp_mm(c, c.Vd, true, c.Td, false, c.Ud, (const float2*)nullptr, 0.f);
  } else {
    pp_each(c, [&](int i, int j) {
      c.Vd[i * c.ld + j] = make_float2(i == j ? 1.f : 0.f, 0.f);
      c.Ud[i * c.ld + j] = c.Bd[i * c.ld + j];
    });
  }
  pp_sync<P>();
  const long long c2 = clock64();
  for (int pass = 0; pass < 3; ++pass) {
    int word = 0;  // 0: done, 1: rotations in Td, 2: first-order correction in Td
    if (c.rank == 0) {
      // F scaled by 2^30 so that squares of entries at 1e-15 stay in range
      constexpr float UP = 1073741824.f;
      float off = 0.f, tot = 0.f;
      for (int i = c.g; i < m; i += P::NG)
        for (int j = c.cl; j < m; j += P::CL) {
          float2 u = i < p && j < p ? pp_ld<P>(c.Ud + i * c.ld + j) : make_float2(0.f, 0.f);
          u = make_float2(u.x * sc, u.y * sc);
          tot += u.x * u.x;
          if (i == j) {
            sh->lam[i] = make_float2(u.x * UP, u.y * UP);
            c.Af[i * lda + j] = 0.f;
          } else {
            off += u.x * u.x;
            c.Af[i * lda + j] = u.x * UP;
          }
        }
      tot = pp_bsum<P>(sh, tot);
      off = pp_bsum<P>(sh, off);
      identity_v();
      __syncthreads();
      if (off > 1e-27f * tot) {
        float kmax = 1.f;
        if (first_order && pass > 0) {
          // largest rotation angle F_ij / (lambda_j - lambda_i): below 1e-8
          // the rotations are I + K to working accuracy. K is made exactly
          // skew from the upper half of F: the halves differ by rounding,
          // which over a small gap would leave V off orthogonal
          kmax = 0.f;
          for (int i = c.g; i < p; i += P::NG)
            for (int j = c.cl; j < p; j += P::CL)
              if (i < j) {
                const float2 d = df_add(sh->lam[j], pp_neg(sh->lam[i]));
                const float f = c.Af[i * lda + j];
                const float k = f == 0.f ? 0.f : f / d.x;
                c.Vf[i * lda + j] = k;
                c.Vf[j * lda + i] = -k;
                kmax = fmaxf(kmax, fabsf(k) <= 1.f ? fabsf(k) : 1.f);
              }
          kmax = pp_bmax<P>(sh, kmax);
        }
        if (kmax <= 1e-8f) {
          for (int i = c.g; i < p; i += P::NG)
            if (c.cl == 0) c.Vf[i * lda + i] = 0.f;
          __syncthreads();
          word = 2;
        } else {
          if (first_order && pass > 0) {
            identity_v();
            __syncthreads();
          }
          s_delta += pp_jacobi<P, true>(c, 8, 1e-30f * tot * UP * UP);
          word = 1;
        }
      }
    }
    word = publish(c.Td, word);
    if (word == 0) break;
    if (word == 2) {  // V += V K
      pp_mm(c, c.Vd, false, c.Td, false, c.Bd, c.Vd, 0.f);
      pp_sync<P>();
      pp_each(c, [&](int i, int j) { c.Vd[i * c.ld + j] = c.Bd[i * c.ld + j]; });
      pp_sync<P>();
      break;
    }
    // V <- orth(V W), U = V^T B V
    pp_mm(c, c.Vd, false, c.Td, false, c.Ud, (const float2*)nullptr, 0.f);
    pp_sync<P>();
    pp_orth(c, c.Ud, c.Td, c.Vd);
    pp_mm(c, c.Bd, false, c.Vd, false, c.Td, (const float2*)nullptr, 0.f);
    pp_sync<P>();
    pp_mm(c, c.Vd, true, c.Td, false, c.Ud, (const float2*)nullptr, 0.f);
    pp_sync<P>();
  }
  if (c.rank == 0 && c.tid == 0 && diag) {
    diag[0] = (double)(c1 - c0);
    diag[1] = (double)(c2 - c1);
    diag[2] = (double)(clock64() - c2);
    diag[3] = s32;
    diag[4] = s_delta;
  }
}

// M = V [diag(s^-1/2) + F o Df] V^T for S' = diag(s) + F in c.Ud, df64 into
// c.Ud and float64 into M; status (0, or 5 if some s_i is not positive) in
// sh->flag of every CTA. F is rounding-level, so its divided differences are
// taken in float32.
template <class P>
__device__ void pp_inv_sqrt(const PpCtx<P>& c, double* M) {
  PpSh* sh = c.sh;
  const int p = c.p;
  if (c.tid < 32) {
    double mx = 0.0;
    for (int i = c.tid; i < p; i += 32) {
      const double s = df_to_double(pp_ld<P>(c.Ud + i * c.ld + i));
      sh->be[i] = s;
      mx = fmax(mx, s);
    }
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    bool bad = false;
    for (int i = c.tid; i < p; i += 32) {
      const double s = sh->be[i];
      // numerically singular: below the df64 rounding level of the largest
      bad = bad || !(s > 1e-13 * mx) || !isfinite(s);
      sh->sv[i] = s > 0.0 ? sqrt(s) : 1.0;
    }
    bad = __any_sync(0xffffffffu, bad);
    if (c.tid == 0) sh->flag = bad ? 5 : 0;
  }
  __syncthreads();
  pp_sync<P>();  // every rank has read the diagonal
  pp_each(c, [&](int i, int j) {
    float2 v;
    if (i == j) {
      v = df_from_double(1.0 / sh->sv[i]);
    } else {
      const float ri = (float)sh->sv[i], rj = (float)sh->sv[j];
      const float2 f = c.Ud[i * c.ld + j];
      v = make_float2(-((__fadd_rn(f.x, f.y) / ri) / rj) / (ri + rj), 0.f);
    }
    c.Ud[i * c.ld + j] = v;
  });
  pp_sync<P>();
  pp_mm(c, c.Vd, false, c.Ud, false, c.Td, (const float2*)nullptr, 0.f);  // V N
  pp_sync<P>();
  pp_mm(c, c.Td, false, c.Vd, true, c.Ud, (const float2*)nullptr, 0.f);   // (V N) V^T
  pp_sync<P>();
  pp_each(c, [&](int i, int j) { M[i * p + j] = df_to_double(c.Ud[i * c.ld + j]); });
}

// this CTA's rows of an input into a df64 matrix
template <class P, class F>
__device__ __forceinline__ void pp_load(const PpCtx<P>& c, const PpMat& a, float2* dst, F f) {
  const int p = c.p;
  pp_each(c, [&](int i, int j) {
    float2 v;
    if (a.f) v = a.f[i * p + j];
    else if (a.sym) v = df_from_double(0.5 * (a.d[i * p + j] + a.d[j * p + i]));
    else v = df_from_double(a.d[i * p + j]);
    dst[i * c.ld + j] = f(i, j, v);
  });
}

// ---- the exact step of Alg. 3 ------------------------------------------------

__device__ __forceinline__ float2 df_div(float2 a, float2 b) {
  const float q1 = __fdiv_rn(a.x, b.x);
  const float p = __fmul_rn(q1, b.x);
  const float e = __fmaf_rn(q1, b.y, __fmaf_rn(q1, b.x, -p));
  const float2 r = df_add(a, make_float2(-p, -e));
  return fast_two_sum(q1, __fdiv_rn(__fadd_rn(r.x, r.y), b.x));
}

__device__ __forceinline__ bool df_less(float2 a, float2 b) { return a.x < b.x || (a.x == b.x && a.y < b.y); }

// The scaled line-search model of one warp: lane l holds the branches l,
// l + 32, .. (t = T tau, phi'(t) = Sz phi'_s(tau), T and Sz powers of two).
template <int MC>
struct PpModel {
  int cnt;  // branches of this lane
  float2 z[MC], dl[MC], bz[MC], b[MC];
};

template <int MC>
__device__ __forceinline__ float2 pp_dphi(const PpModel<MC>& md, float2 tau) {
  float2 s = make_float2(0.f, 0.f);
  const float2 t2 = df_mul(tau, tau);
#pragma unroll
  for (int u = 0; u < MC; ++u)
    if (u < md.cnt) {
      const float2 num = df_add(df_add(md.z[u], df_mul(md.dl[u], tau)), pp_neg(df_mul(md.bz[u], t2)));
      const float2 den = df_add(make_float2(1.f, 0.f), df_mul(md.b[u], t2));
      s = df_add(s, df_div(num, df_mul(den, den)));
    }
  for (int o = 16; o > 0; o >>= 1) {
    const float2 w = make_float2(__shfl_xor_sync(0xffffffffu, s.x, o), __shfl_xor_sync(0xffffffffu, s.y, o));
    s = (threadIdx.x & o) ? df_add(w, s) : df_add(s, w);
  }
  return make_float2(-__shfl_sync(0xffffffffu, s.x, 0), -__shfl_sync(0xffffffffu, s.y, 0));
}

// Brent-Dekker on phi' (as brent_warp of alg3.cuh) in df64 on [a, b]
template <int MC>
__device__ __forceinline__ float2 pp_brent(const PpModel<MC>& md, float2 a, float2 b, float2 fa, float2 fb, int* ev) {
  auto half_of = [](float2 v) { return make_float2(0.5f * v.x, 0.5f * v.y); };
  auto sub = [](float2 x, float2 y) { return df_add(x, pp_neg(y)); };
  auto mag = [](float2 v) { return v.x < 0.f ? pp_neg(v) : v; };
  if (fa.x == 0.f) return a;
  if (fb.x == 0.f) return b;
  float2 c = a, fc = fa, d = sub(b, a), e = d;
  for (int it = 0; it < 100; ++it) {
    if ((fb.x > 0.f && fc.x > 0.f) || (fb.x < 0.f && fc.x < 0.f)) {
      c = a;
      fc = fa;
      d = e = sub(b, a);
    }
    if (df_less(mag(fc), mag(fb))) {
      a = b; b = c; c = a;
      fa = fb; fb = fc; fc = fa;
    }
    const float tol = 5.7e-14f * fabsf(b.x) + 1e-37f;  // 2 units of the df64 significand
    const float2 m = half_of(sub(c, b));
    if (fabsf(m.x) <= tol || fb.x == 0.f) break;
    if (fabsf(e.x) >= tol && df_less(mag(fb), mag(fa))) {
      // the interpolated point only has to be good to float32 relative to
      // the correction d: it is added to b in df64
      const float s = fb.x / fa.x, mm = m.x;
      float P, Q;
      if (a.x == c.x && a.y == c.y) {
        P = 2.f * mm * s;
        Q = 1.f - s;
      } else {
        const float q = fa.x / fc.x, r = fb.x / fc.x;
        P = s * (2.f * mm * q * (q - r) - sub(b, a).x * (r - 1.f));
        Q = (q - 1.f) * (r - 1.f) * (s - 1.f);
      }
      if (P > 0.f) Q = -Q; else P = -P;
      if (2.f * P < fminf(3.f * mm * Q - fabsf(tol * Q), fabsf(e.x * Q))) {
        e = d;
        d = make_float2(P / Q, 0.f);
      } else {
        d = m;
        e = m;
      }
    } else {
      d = m;
      e = m;
    }
    a = b;
    fa = fb;
    b = df_add(b, fabsf(d.x) > tol ? d : make_float2(copysignf(tol, m.x), 0.f));
    fb = pp_dphi(md, b);
    ++*ev;
  }
  return b;
}

// The step of get_mu_warp (alg3.cuh: bracket from the branch roots xi_i, the
// right end doubled from xi_min, Brent on phi'), one warp. The bracket ends
// come in float64; the evaluations of the search run in df64 on a scaled
// model (a float64 evaluation is a chain of ~25 operations on a pipe with
// 1/64 of the float32 rate, ~5,000 cycles an evaluation); the root is then
// corrected by one Newton step from a float64 evaluation of phi', which
// leaves it as accurate as a search in float64. Where the scaled model
// leaves float32's range or the Newton step is not small, the float64
// search runs instead.
template <int MC>
__device__ __noinline__ double pp_step_length(int p, const double* al, const double* be, const double* ga,
                                              const double* ze, int* ev) {
  const int lane = threadIdx.x & 31;
  double sb = 0.0, bmax = 0.0, zmax = 0.0, dmax = 0.0;
  for (int i = lane; i < p; i += 32) {
    sb += be[i];
    bmax = fmax(bmax, be[i]);
    zmax = fmax(zmax, fabs(ze[i]));
    dmax = fmax(dmax, fabs(ga[i] - al[i] * be[i]));
  }
  sb = warp_sum(sb);
  double xmin = INFINITY, xmax = -INFINITY;
  int cnt = 0;
  for (int i = lane; i < p; i += 32) {
    const double b = be[i], z = ze[i];
    if (!(b > ALG3_EPS * sb) || !(z > 0.0)) continue;
    const double d = ga[i] - al[i] * b;
    const double disc = sqrt(d * d + 4.0 * b * z * z);
    const double xi = (d < 0.0) ? 2.0 * z / (-d + disc) : (d + disc) / (2.0 * b * z);
    xmin = fmin(xmin, xi);
    xmax = fmax(xmax, xi);
    ++cnt;
  }
  for (int o = 16; o > 0; o >>= 1) {
    xmin = fmin(xmin, __shfl_xor_sync(0xffffffffu, xmin, o));
    xmax = fmax(xmax, __shfl_xor_sync(0xffffffffu, xmax, o));
    bmax = fmax(bmax, __shfl_xor_sync(0xffffffffu, bmax, o));
    zmax = fmax(zmax, __shfl_xor_sync(0xffffffffu, zmax, o));
    dmax = fmax(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
    cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
  }
  *ev = 0;
  if (cnt == 0) return 0.0;
  // t = T tau with T = min(1/sqrt(max beta), max|zeta| / max|delta|), values
  // over Sz = max|zeta|, each rounded down to a power of two
  double T = 1.0 / sqrt(bmax);
  if (dmax > 0.0) T = fmin(T, zmax / dmax);
  const int eT = T > 0.0 && isfinite(T) ? ilogb(T) : 1 << 20, eZ = zmax > 0.0 && isfinite(zmax) ? ilogb(zmax) : 1 << 20;
  const double lo_s = abs(eT) < 900 ? scalbn(xmin, -eT) : 0.0;
  const bool scaled = abs(eT) < 900 && abs(eZ) < 900 && lo_s > 1e-9 && lo_s < 1e9;
  if (!scaled) return get_mu_warp(p, al, be, ga, ze, ev);
  PpModel<MC> md;
  md.cnt = 0;
#pragma unroll
  for (int u = 0; u < MC; ++u) {
    const int i = lane + 32 * u;
    if (i < p) {
      const double b = scalbn(be[i], 2 * eT), z = scalbn(ze[i], -eZ);
      md.z[u] = df_from_double(z);
      md.b[u] = df_from_double(b);
      md.bz[u] = df_from_double(b * z);
      md.dl[u] = df_from_double(scalbn(ga[i] - al[i] * be[i], eT - eZ));
      md.cnt = u + 1;
    }
  }
  const double hmax = scalbn(xmax, -eT);
  const float2 xmn = df_from_double(lo_s);
  const float2 xmx = hmax < 1e30 ? df_from_double(hmax) : make_float2(1e30f, 0.f);
  const float2 fa = pp_dphi(md, xmn);
  ++*ev;
  float2 lo, flo, hi, fhi;
  if (fa.x > 0.f) {
    lo = make_float2(0.f, 0.f);
    flo = pp_dphi(md, lo);
    ++*ev;
    if (flo.x >= 0.f) return 0.0;
    hi = xmn;
    fhi = fa;
  } else {
    lo = hi = xmn;
    flo = fhi = fa;
    int k = 0;
    while (fhi.x < 0.f) {
      if (k >= 64 || hi.x > 1e18f) return get_mu_warp(p, al, be, ga, ze, ev);
      float2 nxt = make_float2(2.f * hi.x, 2.f * hi.y);
      if (df_less(hi, xmx) && df_less(xmx, nxt)) nxt = xmx;
      lo = hi;
      flo = fhi;
      hi = nxt;
      fhi = pp_dphi(md, hi);
      ++*ev;
      ++k;
    }
  }
  const float2 tau = pp_brent(md, lo, hi, flo, fhi, ev);
  const double t = scalbn(df_to_double(tau), eT);
  // d phi'_s / d tau in float32
  float sl = 0.f;
#pragma unroll
  for (int u = 0; u < MC; ++u)
    if (u < md.cnt) {
      const float x = tau.x, b = md.b[u].x;
      const float num = md.z[u].x + md.dl[u].x * x - md.bz[u].x * x * x, den = 1.f + b * x * x;
      sl += ((md.dl[u].x - 2.f * md.bz[u].x * x) * den - 4.f * b * x * num) / (den * den * den);
    }
  for (int o = 16; o > 0; o >>= 1) sl += __shfl_xor_sync(0xffffffffu, sl, o);
  sl = -__shfl_sync(0xffffffffu, sl, 0);
  const double f = dphi_warp(t, p, al, be, ga, ze);
  ++*ev;
  const double corr = scalbn(f / (double)sl, eT - eZ);
  if (!(fabs(corr) <= 1e-9 * t)) return get_mu_warp(p, al, be, ga, ze, ev);
  return t - corr;
}

// The diagonal of V^T G V (G in c.Ud, V in c.Vd) into d (shared memory of
// every CTA). The row groups' sums pass through c.Af, the ranks' through the
// control words. Synchronised on exit.
template <class P>
__device__ void pp_diag(const PpCtx<P>& c, double* d) {
  const int p = c.p;
  float2* part = reinterpret_cast<float2*>(c.Af);
  pp_mm(c, c.Ud, false, c.Vd, false, (float2*)nullptr, (const float2*)nullptr, 0.f, c.Vd, part);
  __syncthreads();
  for (int j = c.tid; j < p; j += P::NT) {
    float2 s = part[j];
    for (int g = 1; g < P::RG; ++g) s = df_add(s, part[g * p + j]);
    if constexpr (P::NC == 1) d[j] = df_to_double(s);
    else c.ctl[64 + c.rank * 128 + j] = s;
  }
  pp_sync<P>();
  if constexpr (P::NC > 1) {
    for (int j = c.tid; j < p; j += P::NT) {
      float2 s = __ldcg(c.ctl + 64 + j);
      for (int g = 1; g < P::NC; ++g) s = df_add(s, __ldcg(c.ctl + 64 + g * 128 + j));
      d[j] = df_to_double(s);
    }
    pp_sync<P>();
  }
}

// One p x p step by the whole CTA (or cluster). mode 0: eigenbasis of B,
// line-search coefficients, the step t of Alg. 3 and M = S^{-1/2}; mode 1:
// M = B^{-1/2}; mode 2: eigenvectors of B into M, eigenvalues into theta,
// unsorted. Mode 0 in two launches: mode 3 leaves the eigenbasis in eig,
// mode 4 takes it from there.
template <class P>
__device__ void pp_body(const PpArgs& a, PpCtx<P>& c) {
  const int p = c.p;
  PpSh* sh = c.sh;
  double* out = a.out;
  const bool lead = c.rank == 0 && c.tid == 0;
  const long long t0 = clock64();
  auto same = [](int, int, float2 v) { return v; };
  if (a.mode == 4) {
    pp_each(c, [&](int i, int j) { c.Vd[i * c.ld + j] = a.eig[i * p + j]; });
    for (int i = c.tid; i < p; i += P::NT) sh->be[i] = fmax(df_to_double(a.eig[p * p + i]), 0.0);
    __syncthreads();
  } else {
    pp_load(c, a.B, c.Bd, same);
    pp_sync<P>();
    pp_eig(c, a.mode != 1, out + 8);
    if (a.mode == 0) {
      for (int i = c.tid; i < p; i += P::NT)
        sh->be[i] = fmax(df_to_double(pp_ld<P>(c.Ud + i * c.ld + i)), 0.0);
      __syncthreads();
    }
  }
  const long long t1 = clock64();
  if (a.mode == 3) {
    pp_each(c, [&](int i, int j) {
      a.eig[i * p + j] = c.Vd[i * c.ld + j];
      if (i == j) a.eig[p * p + i] = c.Ud[i * c.ld + i];
    });
    if (lead) out[5] = (double)(t1 - t0);
    return;
  }
  if (a.mode == 2) {
    pp_each(c, [&](int i, int j) {
      a.M[i * p + j] = df_to_double(c.Vd[i * c.ld + j]);
      if (i == j) a.theta[i] = df_to_double(c.Ud[i * c.ld + i]);
    });
    if (lead) out[3] = 0.0;
    return;
  }
  if (a.mode == 1) {
    pp_inv_sqrt(c, a.M);
    if (lead) {
      out[0] = out[1] = out[2] = 0.0;
      out[3] = (double)sh->flag;
    }
    return;
  }
  // alpha, gamma, zeta = diag(V^T {C, Gam, Z} V)
  pp_sync<P>();  // every rank has read the diagonal from Ud
  pp_load(c, a.C, c.Ud, same);
  pp_sync<P>();
  pp_diag(c, sh->al);
  pp_load(c, a.Gam, c.Ud, same);
  pp_sync<P>();
  pp_diag(c, sh->ga);
  pp_load(c, a.Z, c.Ud, same);
  pp_sync<P>();
  pp_diag(c, sh->ze);
  // X^T D = (I - X^T X)(C + beta K) into Bd
  if (a.XD.f || a.XD.d) {
    pp_load(c, a.XD, c.Bd, same);
  } else {
    pp_load(c, a.XX, c.Ud, [](int i, int j, float2 v) {
      v = pp_neg(v);
      return i == j ? df_add(make_float2(1.f, 0.f), v) : v;
    });
    const float2 bt = df_from_double(a.beta);
    const bool use_k = a.beta != 0.0;
    pp_load(c, a.C, c.Td, [&](int i, int j, float2 v) {
      if (!use_k) return v;
      const float2 k = a.K.f ? a.K.f[i * p + j] : df_from_double(a.K.d[i * p + j]);
      return df_add(v, df_mul(bt, k));
    });
    pp_sync<P>();
    pp_mm(c, c.Ud, false, c.Td, false, c.Bd, (const float2*)nullptr, 0.f);
  }
  pp_sync<P>();
  const long long t2 = clock64();
  if (c.tid < 32) {
    if (c.rank == 0) {
      int ev = 0;
      const double t = pp_step_length<(P::CL * P::TC * P::NCG + 31) / 32>(p, sh->al, sh->be, sh->ga, sh->ze, &ev);
      double bmax = 0.0;
      for (int i = c.tid; i < p; i += 32) bmax = fmax(bmax, sh->be[i]);
      for (int o = 16; o > 0; o >>= 1) bmax = fmax(bmax, __shfl_xor_sync(0xffffffffu, bmax, o));
      const double ph = phi_model_warp(t, p, sh->al, sh->be, sh->ga, sh->ze);
      if (c.tid == 0) {
        sh->t = t;
        if (P::NC > 1) *reinterpret_cast<double*>(c.ctl + 2) = t;
        out[0] = t;
        out[1] = ph;
        out[2] = (double)ev;
        out[4] = bmax;
      }
    }
  }
  pp_sync<P>();
  const double t = P::NC == 1 ? sh->t : __ldcg(reinterpret_cast<const double*>(c.ctl + 2));
  const long long t3 = clock64();
  // S' = V^T S V with S = XX + t (XD + XD^T) + t^2 B
  const float2 td = df_from_double(t), tt = df_from_double(t * t);
  auto elem = [&](const PpMat& g, int i, int j) {
    return g.f ? g.f[i * p + j]
               : df_from_double(g.sym ? 0.5 * (g.d[i * p + j] + g.d[j * p + i]) : g.d[i * p + j]);
  };
  pp_load(c, a.XX, c.Ud, [&](int i, int j, float2 v) {
    const float2 xd = df_add(pp_ld<P>(c.Bd + i * c.ld + j), pp_ld<P>(c.Bd + j * c.ld + i));
    return df_add(df_add(v, df_mul(td, xd)), df_mul(tt, elem(a.B, i, j)));
  });
  pp_sync<P>();
  pp_mm(c, c.Ud, false, c.Vd, false, c.Td, (const float2*)nullptr, 0.f);
  pp_sync<P>();
  pp_mm(c, c.Vd, true, c.Td, false, c.Ud, (const float2*)nullptr, 0.f);
  pp_sync<P>();
  pp_inv_sqrt(c, a.M);
  if (lead) out[3] = (double)sh->flag;
  if (a.Kd) {  // K_next = X_new^T D = M (X^T D + t D^T D)
    pp_each(c, [&](int i, int j) {
      c.Td[i * c.ld + j] = df_add(c.Bd[i * c.ld + j], df_mul(td, elem(a.B, i, j)));
    });
    pp_sync<P>();
    pp_mm(c, c.Ud, false, c.Td, false, c.Bd, (const float2*)nullptr, 0.f);
    pp_sync<P>();
    pp_each(c, [&](int i, int j) {
      const float2 v = c.Bd[i * c.ld + j];
      a.Kd[i * p + j] = df_to_double(v);
      if (a.Kf) a.Kf[i * p + j] = v;
    });
  }
  if (lead) {
    // cycles: eigenbasis (mode 3 wrote it), coefficients and X^T D, line
    // search (index 13), polar normaliser and K
    if (a.mode != 4) out[5] = (double)(t1 - t0);
    out[6] = (double)(t2 - t1);
    out[13] = (double)(t3 - t2);
    out[7] = (double)(clock64() - t3);
  }
}

}  // namespace gsi
