// Device code of the p x p step (Alg. 3 and the polar normaliser) for one
// thread block or one thread-block cluster per problem. Matrices and products
// are df64; S = Gram of X + tD and K_next are formed in float64, and the root
// of the line search is corrected with a float64 evaluation.
//
// Eigenbasis of a symmetric B: float32 Jacobi sweeps give V0; V is made
// orthonormal in df64; then B' = V^T B V = diag(lambda) + F is formed in df64
// and the small F taken out by V <- V exp(K), K_ij = F_ij / (lambda_j -
// lambda_i), which squares the relative size of F without a sweep's dependent
// rounds. Where eigenvalues cluster (|K| > 0.07), F is rotated away by the same
// float32 Jacobi, which works on F and on df64 differences of lambda, so that
// its float32 rounding is relative to F: each such pass gains six to seven
// digits. Either way the correction is one matrix, applied in df64. One step
// of a random B in one launch, p = 8 / 32 / 64 / 128: 66 / 177 / 351 / 1540 us;
// as one CTA of 1024 threads with df64 sweeps and a float64 line search 159 /
// 515 / 1432 / 10660. In the solver's two launches and with K: 71 / 194 / 382 /
// 1610. (Sweeps instead of the corrections cost 10% at p = 8 and 30% at 128.)
//
// Layout of the work. The sweeps are a chain of p - 1 rounds each, so a
// round is kept short: AW warps (1, 4, 8 or 16) work on A alone, every lane
// computes the angle of its own rotation, 2 x 2 blocks take their partner's
// by shuffle, and A is double-buffered, which leaves one barrier among those
// warps per round. The rotations go to a log; V is a chain per row only, and
// is formed from a sweep's log by the other warps (ranks, for NC > 1) while
// the next sweep runs. For p > 64 the angles pass through shared memory (two
// barriers a round).
// Products give every thread a TR x TC register tile. With NC > 1 CTAs the
// matrices live in global memory (L2), each CTA forms p / NC rows of every
// product from copies in its shared memory, rank 0 runs the sweeps and the
// other ranks form V; the CTAs meet at cluster barriers.
#pragma once
#include <math.h>

#include "alg3.cuh"
#include "df.cuh"

namespace gsi {

// Block shape: NT threads; a group of CL lanes covers TC CL columns of a
// product (NCG such column blocks), the groups its rows, TR each. Jacobi:
// AW warps work on A (p = 64: 687 cycles a round with 16 warps of one block
// a lane, 934 with 8 of two; p = 32: 689 with 4, 779 with 2; 453 at p = 32
// with unpadded rows); a segment of SEG lanes holds one rotation per lane
// (SEG = 64: p > 64), IL 2 x 2 blocks a lane: the blocks of rotations k and
// k + d, 1 <= d <= half / 2, half <= SEG rotations a round.
template <int NT_, int CL_, int TR_, int TC_, int NCG_, int SEG_, int AW_, int IL_, int NC_>
struct PpCfg {
  static constexpr int NT = NT_, CL = CL_, TR = TR_, TC = TC_, NCG = NCG_, NC = NC_;
  static constexpr int NG = NT / CL, RG = NG / NCG;
  static_assert(RG <= 16, "pp_jac_bytes");
  static constexpr int SEG = SEG_, AW = AW_, IL = IL_;
  static_assert(SEG == 64 || (32 / SEG) * AW * IL * 2 >= SEG, "every pair of rotations has a lane");
  static_assert(NC > 1 ? NT / 32 >= AW : NT / 32 > AW, "V needs warps (or ranks) of its own");
};

// a p x p input: float64 (symmetrised where sym is set), and where f is set
// the same in df64, which the df64 products then take
struct PpMat {
  const float2* f;
  const double* d;
  int sym;
};

struct PpArgs {
  int mode, p;
  int want_phi;  // mode 0: out[1] = phi(t)
  int scale_b;  // mode 3, float64 B: divided by a power of two near max |B| (B may leave float32's range)
  // B = D^T D (modes 0, 3) or the matrix itself (modes 1, 2); C = X^T A X,
  // Gam = D^T W, Z = D^T R, XX = X^T X; XD = X^T D, or null pointers: formed
  // here as (I - XX)(C + beta K)
  PpMat C, B, Gam, Z, XX, XD, K;
  double beta;
  double* M;      // p x p result (eigenvectors in mode 2)
  double* Kd;     // K_next = M (XD + t B), float64 (or null; one CTA only)
  double* Tn;     // XD + t B alone, for a product on more SMs (or null)
  double* theta;  // mode 2: eigenvalues
  float2* eig;    // modes 3, 4: V (p x p), then the diagonal of V^T B V
  double* out;    // 16 doubles: t, phi, evaluations, status, max beta, cycle counts and sweeps
  float2* gws;    // NC > 1: pp_gws_bytes(p) of global scratch
};
constexpr int PP_K_INSIDE = 16;  // widest block whose K_next the step forms itself in a solve
constexpr int PP_CTL = 1024 + 64;  // float2: control words, then the partial dots of up to 8 ranks

struct PpSh {  // small tables, shared memory
  double al[128], be[128], ga[128], ze[128], sv[128];
  float2 alf[128], bef[128], gaf[128], zef[128], svf[128];  // the same in df64
  float2 lam[2][130];
  float2 cs[64];
  float red[32];
  double t;
  int flag, ctl;
};

// All dynamic shared memory of a kernel that runs this code: PpSh first, then
// the matrices. Everything is addressed as pp_sm + offset, so that the
// compiler sees shared accesses: pointers kept in a context struct became
// generic ones, and the loads of a Jacobi round's chain took twice as long.
extern __shared__ __align__(16) unsigned char pp_sm[];
__device__ __forceinline__ PpSh* pp_sh() { return reinterpret_cast<PpSh*>(pp_sm); }

template <class P>
struct PpCtx {
  int p, ld, tid, cl, g, rank, r0, r1, lda;
  // offsets: df64 matrices (rows ld apart) and the two logs of a sweep's
  // rotations in float2 units of pp_sm (NC = 1) or gws (NC > 1); the Jacobi
  // matrices (rows lda apart) in floats of pp_sm; for NC > 1 the staged Y and
  // strip of X of a product in float2 of pp_sm, the control words in gws
  int Bd, Vd, Td, Ud, log0, log1, Af, A2, Vf, sX, sY, ctl;
  float2* gws;
  __device__ __forceinline__ float2* mat(int o) const {
    if constexpr (P::NC == 1) return reinterpret_cast<float2*>(pp_sm) + o;
    else return gws + o;
  }
  __device__ __forceinline__ float2 ldm(int o) const {
    if constexpr (P::NC == 1) return reinterpret_cast<float2*>(pp_sm)[o];
    else return __ldcg(gws + o);
  }
};
__device__ __forceinline__ float* pp_sf(int o) { return reinterpret_cast<float*>(pp_sm) + o; }
__device__ __forceinline__ float2* pp_s2(int o) { return reinterpret_cast<float2*>(pp_sm) + o; }

// Row stride of the Jacobi matrices for m (even) columns. Over the lanes a row
// index grows by one and a column index grows or falls by one, so the banks
// of a round's accesses step by lda + 1 or lda - 1: both are odd for the even
// m itself, and no two lanes of a segment meet.
__host__ __device__ inline int pp_lda(int m) { return m; }
// bytes of a Jacobi matrix; the first also holds the dot products' partial
// sums (up to 16 row groups of p df64 values, pp_diag)
__host__ __device__ inline int pp_jac_bytes(int p) {
  const int m = (p + 1) & ~1, a = m * pp_lda(m) * (int)sizeof(float), b = 16 * p * (int)sizeof(float2);
  return ((a > b ? a : b) + 15) & ~15;
}
__host__ __device__ inline size_t pp_al(size_t b) { return (b + 15) & ~(size_t)15; }
__host__ __device__ inline size_t pp_log_len(int p) {  // rotations of a sweep
  const size_t m = (p + 1) & ~1;
  return (m - 1) * (m / 2);
}
// dynamic shared memory: NC = 1: four df64 matrices, the Jacobi matrices A
// (two buffers) and V, two logs; NC > 1: staged Y (V or a log share its
// space), strip of X, A or a float32 copy of E, A's second buffer (p <= 64)
inline size_t pp_smem(int p, int nc) {
  const size_t ld = p | 1, jac = pp_jac_bytes(p);
  const size_t sh = pp_al(sizeof(PpSh));
  if (nc == 1)
    return sh + 4 * pp_al((size_t)p * ld * sizeof(float2)) + 3 * jac + 2 * pp_al(pp_log_len(p) * sizeof(float2));
  const size_t sy = pp_al((size_t)p * ld * sizeof(float2));
  return sh + (sy > jac ? sy : jac) + pp_al((size_t)((p + nc - 1) / nc) * ld * sizeof(float2)) + (p > 64 ? 1 : 2) * jac;
}
inline size_t pp_gws_bytes(int p) { return (4 * (size_t)p * p + PP_CTL + 2 * pp_log_len(p)) * sizeof(float2); }

template <class P>
__device__ __forceinline__ void pp_sync() {
  if constexpr (P::NC == 1) {
    __syncthreads();
  } else {
    asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
  }
}

template <class P>
__device__ __forceinline__ PpCtx<P> pp_ctx(int p, float2* gws) {
  PpCtx<P> c;
  c.p = p;
  c.gws = gws;
  c.tid = threadIdx.x;
  c.cl = c.tid % P::CL;
  c.g = c.tid / P::CL;
  const int m = (p + 1) & ~1;
  c.lda = pp_lda(m);
  int cur = (int)pp_al(sizeof(PpSh));
  auto take = [&](int bytes) {
    const int r = cur;
    cur += (bytes + 15) & ~15;
    return r;
  };
  const int jac = pp_jac_bytes(p), len = (m - 1) * (m / 2);
  if constexpr (P::NC == 1) {
    c.rank = 0;
    c.r0 = 0;
    c.r1 = p;
    c.ld = p | 1;
    const int mb = p * c.ld * 8;
    c.Bd = take(mb) / 8;
    c.Vd = take(mb) / 8;
    c.Td = take(mb) / 8;
    c.Ud = take(mb) / 8;
    c.Af = take(jac) / 4;
    c.A2 = take(jac) / 4;
    c.Vf = take(jac) / 4;
    c.log0 = take(len * 8) / 8;
    c.log1 = take(len * 8) / 8;
    c.sX = c.sY = c.ctl = 0;
  } else {
    uint32_t rk;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rk));
    c.rank = (int)rk;
    const int rs = (p + P::NC - 1) / P::NC, q = p * p;
    c.r0 = min(p, c.rank * rs);
    c.r1 = min(p, c.r0 + rs);
    c.ld = p;
    c.Bd = 0;
    c.Vd = q;
    c.Td = 2 * q;
    c.Ud = 3 * q;
    c.ctl = 4 * q;
    c.log0 = c.ctl + PP_CTL;
    c.log1 = c.log0 + len;
    const int y = take(max(p * (p | 1) * 8, jac));
    c.sY = y / 8;
    c.Vf = y / 4;  // rank 0: the first-order correction K
    c.sX = take(rs * (p | 1) * 8) / 8;
    // the Jacobi matrix of rank 0 and every rank's copy of E share this
    c.Af = take(jac) / 4;
    c.A2 = P::SEG == 64 ? 0 : take(jac) / 4;
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

// Rows r0..r1 of X' Y', X' = X^T if tx, Y' = Y^T if ty (matrices by offset,
// -1: none). Without dots: Out = (Add +) X' Y' - dsub I. With dots (in
// shared memory): dots[g p + j] += sum over this
// group's rows i of Vdot[i, j] (X' Y')[i, j] (df64 pairs, one row of dots per
// row group). The caller synchronises before and after. One copy of the code
// serves every product of a step (the instruction cache is cold at each
// launch).
template <class P>
__device__ __noinline__ void pp_mm_fn(int p, float2* gws, int X, bool tx, int Y, bool ty, int Out, int Add, float dsub,
                                      int Vdot, int dots) {
  const PpCtx<P> c = pp_ctx<P>(p, gws);
  const int rows = c.r1 - c.r0;
  const float2 *xs, *ys;
  int xi, xk, yk, yj;
  if constexpr (P::NC == 1) {
    xs = pp_s2(X);
    ys = pp_s2(Y);
    xi = tx ? 1 : c.ld;
    xk = tx ? c.ld : 1;
    yk = ty ? 1 : c.ld;
    yj = ty ? c.ld : 1;
  } else {
    const int ls = p | 1;
    float2 *const sY = pp_s2(c.sY), *const sX = pp_s2(c.sX);
    for (int k = c.g; k < p; k += P::NG)
      for (int j = c.cl; j < p; j += P::CL) sY[ty ? j * ls + k : k * ls + j] = c.ldm(Y + k * p + j);
    if (tx) {
      for (int e = c.tid; e < rows * p; e += P::NT) {
        const int k = e / rows, i = e - k * rows;
        sX[i * ls + k] = c.ldm(X + k * p + c.r0 + i);
      }
    } else {
      for (int i = c.g; i < rows; i += P::NG)
        for (int k = c.cl; k < p; k += P::CL) sX[i * ls + k] = c.ldm(X + (c.r0 + i) * p + k);
    }
    __syncthreads();
    xs = sX;
    ys = sY;
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
          if (dots >= 0) {
            pp_mac(dacc[t].x, dacc[t].y, c.ldm(Vdot + i * c.ld + j), v);
          } else {
            if (i == j && dsub != 0.f) v = df_add_f(v, -dsub);
            if (Add >= 0) v = df_add(c.ldm(Add + i * c.ld + j), v);
            c.mat(Out)[i * c.ld + j] = v;
          }
        }
      }
  }
  if (dots >= 0) {
#pragma unroll
    for (int t = 0; t < P::TC; ++t) {
      const int j = jb + t * P::CL;
      if (j < p) pp_s2(dots)[rg * p + j] = fast_two_sum(dacc[t].x, dacc[t].y);
    }
  }
}

template <class P>
__device__ __forceinline__ void pp_mm(const PpCtx<P>& c, int X, bool tx, int Y, bool ty, int Out, int Add = -1,
                                      float dsub = 0.f, int Vdot = -1, int dots = -1) {
  pp_mm_fn<P>(c.p, c.gws, X, tx, Y, ty, Out, Add, dsub, Vdot, dots);
}

// sum over the block (float32, fixed order), the same in every thread
template <class P>
__device__ float pp_bsum(float v) {
  PpSh* const sh = pp_sh();
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
__device__ float pp_bmax(float v) {
  PpSh* const sh = pp_sh();
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh->red[threadIdx.x >> 5] = v;
  __syncthreads();
  float s = 0.f;
#pragma unroll
  for (int w = 0; w < P::NT / 32; ++w) s = fmaxf(s, sh->red[w]);
  return s;
}

__device__ __forceinline__ float pp_rsqrt(float x) {  // 1/sqrt(x), one Newton step on the approximation
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y * __fmaf_rn(-0.5f * x, y * y, 1.5f);
}

// The rotation of a pivot f with diagonal entries la, lb (DELTA: df64;
// otherwise la.x, lb.x): returns (c, s), t = s / c. From cos 2 theta =
// |d| / sqrt(d^2 + 4 f^2), d = lb - la: c^2 = (1 + cos 2 theta) / 2 and
// s = f / (sqrt(d^2 + 4 f^2) c), a chain of two reciprocal roots (a division,
// a root and a reciprocal root took half of a round).
template <bool DELTA>
__device__ __forceinline__ float2 pp_angle(float f, float2 la, float2 lb, float& t) {
  float d;
  if (DELTA) {
    const float2 dd = df_add(lb, pp_neg(la));
    d = __fadd_rn(dd.x, dd.y);
  } else {
    d = lb.x - la.x;
  }
  const float b2 = 2.f * f, q2 = __fmaf_rn(d, d, b2 * b2);
  const bool rot = q2 >= 1.17549435e-38f;  // else d and f are zero, or far below the matrix's rounding
  const float h = pp_rsqrt(rot ? q2 : 1.f);
  const float c2 = __fmaf_rn(0.5f * fabsf(d), h, 0.5f);
  const float rc = pp_rsqrt(c2);
  const float sn = (d >= 0.f ? f : -f) * h * rc;
  t = rot ? sn * rc : 0.f;
  return rot ? make_float2(c2 * rc, sn) : make_float2(1.f, 0.f);
}

// 2 x 2 block z = J_k^T x J_l
__device__ __forceinline__ void pp_rot2(float2 wk, float2 wl, const float x[4], float z[4]) {
  const float y00 = wl.x * x[0] - wl.y * x[1], y01 = wl.y * x[0] + wl.x * x[1];
  const float y10 = wl.x * x[2] - wl.y * x[3], y11 = wl.y * x[2] + wl.x * x[3];
  z[0] = wk.x * y00 - wk.y * y10;
  z[2] = wk.y * y00 + wk.x * y10;
  z[1] = wk.x * y01 - wk.y * y11;
  z[3] = wk.y * y01 + wk.x * y11;
}

// Round-robin ordering of m (even) indices: in round r slot 0 pairs r with
// m - 1, slot k pairs r + k and r - k modulo m - 1.
// One sweep over A (symmetric m x m, m even; the dummy row and column of an
// odd p are zero and stay so) by the first AW warps of the CTA, p <= 64; the
// result is in `An` after an odd number of rounds. DELTA: A holds only the
// off-diagonal part and lam[lp] the df64 diagonal (lam[lp ^ 1] on return).
// A, An: offsets of the two buffers.
template <class P, bool DELTA>
__device__ void pp_sweep(const PpCtx<P>& c, int Ao, int Ano, int lp, int log) {
  constexpr int SEG = P::SEG, NSEG = 32 / SEG;
  const int lda = c.lda, m = (c.p + 1) & ~1, half = m / 2, m1 = m - 1;
  const int lane = c.tid & 31, w = c.tid >> 5, seg = lane / SEG, k = lane % SEG;
  const bool own = k < half, lead = own && w == 0 && seg == 0;
  int a = own ? k : 0, b = own ? (k == 0 ? m1 : m1 - k) : 0;  // round 0's pair
  int src[P::IL], al[P::IL], bl[P::IL];  // the partner's lane and pair
  bool live[P::IL], l0[P::IL];
#pragma unroll
  for (int z = 0; z < P::IL; ++z) {
    const int d = 1 + ((z * P::AW + w) * NSEG + seg);
    live[z] = own && 2 * d <= half && !(2 * d == half && k >= d);
    int l = k + d;
    l -= l >= half ? half : 0;
    src[z] = live[z] ? seg * SEG + l : lane;
    al[z] = live[z] ? l : 0;
    l0[z] = l == 0;
    bl[z] = live[z] ? (l == 0 ? m1 : m1 - l) : 0;
  }
  for (int r = 0; r < m1; ++r) {
    float *const A = pp_sf(Ao), *const An = pp_sf(Ano);
    float2 *const lam = pp_sh()->lam[lp], *const lamn = pp_sh()->lam[lp ^ 1];
    const int ra = a * lda, rb = b * lda;
    const float f = own ? A[ra + b] : 0.f;
    float2 la = make_float2(0.f, 0.f), lb = la;
    if (DELTA) {
      la = lam[a];
      lb = lam[b];
    } else if (own) {
      la.x = A[ra + a];
      lb.x = A[rb + b];
    }
    float x[P::IL][4];
#pragma unroll
    for (int z = 0; z < P::IL; ++z) {
      if (live[z]) {
        x[z][0] = A[ra + al[z]];
        x[z][1] = A[ra + bl[z]];
        x[z][2] = A[rb + al[z]];
        x[z][3] = A[rb + bl[z]];
      } else {
        x[z][0] = x[z][1] = x[z][2] = x[z][3] = 0.f;
      }
    }
    float t;
    const float2 cs = pp_angle<DELTA>(f, la, lb, t);
    if (lead) {
      c.mat(log)[r * half + k] = cs;
      const float d = t * f;
      if (DELTA) {
        lamn[a] = df_add_f(la, -d);
        lamn[b] = df_add_f(lb, d);
      } else {
        An[ra + a] = la.x - d;
        An[rb + b] = lb.x + d;
      }
      An[ra + b] = 0.f;
      An[rb + a] = 0.f;
    }
#pragma unroll
    for (int z = 0; z < P::IL; ++z) {
      const float2 wl = make_float2(__shfl_sync(0xffffffffu, cs.x, src[z]), __shfl_sync(0xffffffffu, cs.y, src[z]));
      float y[4];
      pp_rot2(cs, wl, x[z], y);
      if (live[z]) {
        const int rl = al[z] * lda, sl = bl[z] * lda;
        An[ra + al[z]] = y[0];
        An[ra + bl[z]] = y[1];
        An[rb + al[z]] = y[2];
        An[rb + bl[z]] = y[3];
        An[rl + a] = y[0];
        An[sl + a] = y[1];
        An[rl + b] = y[2];
        An[sl + b] = y[3];
      }
    }
    // both indices of a pair advance by one modulo m - 1 (slot 0 keeps m - 1)
    a = a + 1 == m1 ? 0 : a + 1;
    if (k != 0) b = b + 1 == m1 ? 0 : b + 1;
#pragma unroll
    for (int z = 0; z < P::IL; ++z) {
      al[z] = al[z] + 1 == m1 ? 0 : al[z] + 1;
      if (!l0[z]) bl[z] = bl[z] + 1 == m1 ? 0 : bl[z] + 1;
    }
    const int u = Ao;
    Ao = Ano;
    Ano = u;
    lp ^= 1;
    if constexpr (P::AW == 1) __syncwarp();
    else asm volatile("bar.sync 1, %0;" ::"n"(P::AW * 32) : "memory");
  }
}

// The same for p > 64 by the whole CTA, A in place: half threads form the
// angles, then every unordered pair of rotations is one thread's block. A
// thread's pairs advance by one index a round, as in pp_sweep (recomputing
// them took 2080 cycles a round at p = 128, this takes 1890; loading all of a
// thread's blocks before the first store 2080 again).
template <class P, bool DELTA>
__device__ void pp_sweep_wide(const PpCtx<P>& c, int log) {
  float2* const lam = pp_sh()->lam[0];
  const int lda = c.lda, tid = c.tid, m = (c.p + 1) & ~1, half = m / 2, m1 = m - 1;
  const int items = half * (half - 1) / 2;
  auto next = [&](int x) { return x + 1 == m1 ? 0 : x + 1; };
  int ta = tid < half ? tid : 0, tb = ta == 0 ? m1 : m1 - ta;  // round 0's pair
  int ik[P::IL], il[P::IL], ak[P::IL], bk[P::IL], al[P::IL], bl[P::IL];
#pragma unroll
  for (int z = 0; z < P::IL; ++z) {
    const int e = tid + z * P::NT;
    ik[z] = -1;
    il[z] = 0;
    if (e < items) {
      const int d = e / half;  // partner distance d + 1
      ik[z] = e - d * half;
      il[z] = ik[z] + d + 1;
      il[z] -= il[z] >= half ? half : 0;
    }
    ak[z] = max(ik[z], 0);
    bk[z] = ak[z] == 0 ? m1 : m1 - ak[z];
    al[z] = il[z];
    bl[z] = il[z] == 0 ? m1 : m1 - il[z];
  }
  for (int r = 0; r < m1; ++r) {
    float* const A = pp_sf(c.Af);
    if (tid < half) {
      const int ra = ta * lda, rb = tb * lda;
      const float f = A[ra + tb];
      float2 la, lb;
      if (DELTA) {
        la = lam[ta];
        lb = lam[tb];
      } else {
        la = make_float2(A[ra + ta], 0.f);
        lb = make_float2(A[rb + tb], 0.f);
      }
      float t;
      const float2 cs = pp_angle<DELTA>(f, la, lb, t);
      pp_sh()->cs[tid] = cs;
      c.mat(log)[r * half + tid] = cs;
      const float d = t * f;
      if (DELTA) {
        lam[ta] = df_add_f(la, -d);
        lam[tb] = df_add_f(lb, d);
      } else {
        A[ra + ta] = la.x - d;
        A[rb + tb] = lb.x + d;
      }
      A[ra + tb] = 0.f;
      A[rb + ta] = 0.f;
      ta = next(ta);
      if (tid != 0) tb = next(tb);
    }
    __syncthreads();
#pragma unroll
    for (int z = 0; z < P::IL; ++z) {
      if (ik[z] >= 0) {
        const int ra = ak[z] * lda, rb = bk[z] * lda, rl = al[z] * lda, sl = bl[z] * lda;
        const float x[4] = {A[ra + al[z]], A[ra + bl[z]], A[rb + al[z]], A[rb + bl[z]]};
        float y[4];
        pp_rot2(pp_sh()->cs[ik[z]], pp_sh()->cs[il[z]], x, y);
        A[ra + al[z]] = y[0];
        A[ra + bl[z]] = y[1];
        A[rb + al[z]] = y[2];
        A[rb + bl[z]] = y[3];
        A[rl + ak[z]] = y[0];
        A[sl + ak[z]] = y[1];
        A[rl + bk[z]] = y[2];
        A[sl + bk[z]] = y[3];
        ak[z] = next(ak[z]);
        if (ik[z] != 0) bk[z] = next(bk[z]);
        al[z] = next(al[z]);
        if (il[z] != 0) bl[z] = next(bl[z]);
      }
    }
    __syncthreads();
  }
}

// rows [0, rows) of V (ldv apart; offsets of V and of the log in shared
// memory) times the rotations of a sweep's log, by nw
// warps (this one is w of them): a row belongs to one segment of lanes
template <class P>
__device__ void pp_apply_log(int p, int Vo, int ldv, int rows, int logo, int w, int nw) {
  float* const V = pp_sf(Vo);
  const float2* const log = pp_s2(logo);
  constexpr int SEG = P::SEG > 32 ? 32 : P::SEG, NSEG = 32 / SEG, LL = P::SEG / SEG;  // rotations a lane
  const int m = (p + 1) & ~1, half = m / 2, m1 = m - 1;
  const int lane = threadIdx.x & 31, seg = lane / SEG;
  int a[LL], b[LL];
#pragma unroll
  for (int z = 0; z < LL; ++z) {
    const int l = lane % SEG + z * SEG;
    a[z] = l;
    b[z] = l == 0 ? m1 : m1 - l;
  }
  for (int r = 0; r < m1; ++r) {
#pragma unroll
    for (int z = 0; z < LL; ++z) {
      const int l = lane % SEG + z * SEG;
      if (l < half) {
        const float2 cs = log[r * half + l];
        // four rows in flight: their loads before any of their stores
        for (int row = w * NSEG + seg; row < rows; row += 4 * nw * NSEG) {
          float x[4], y[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int rr = row + u * nw * NSEG;  // other rows belong to other segments
            x[u] = rr < rows ? V[rr * ldv + a[z]] : 0.f;
            y[u] = rr < rows ? V[rr * ldv + b[z]] : 0.f;
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int rr = row + u * nw * NSEG;
            if (rr < rows) {
              V[rr * ldv + a[z]] = cs.x * x[u] - cs.y * y[u];
              V[rr * ldv + b[z]] = cs.y * x[u] + cs.x * y[u];
            }
          }
        }
        a[z] = a[z] + 1 == m1 ? 0 : a[z] + 1;
        if (l != 0) b[z] = b[z] + 1 == m1 ? 0 : b[z] + 1;
      }
    }
    __syncwarp();
  }
}

// rows of V of this rank for NC > 1 (rank 0 runs the sweeps and has none)
template <class P>
__device__ __forceinline__ void pp_vrows(const PpCtx<P>& c, int& v0, int& v1) {
  constexpr int VR = P::NC > 1 ? P::NC - 1 : 1;
  const int per = (c.p + VR - 1) / VR;
  v0 = c.rank == 0 ? 0 : min(c.p, (c.rank - 1) * per);
  v1 = c.rank == 0 ? 0 : min(c.p, v0 + per);
}

// Float32 Jacobi sweeps on c.Af until the squared off-diagonal mass is at most
// `stop` (rank 0's value), and for one sweep more if it is then above `stop2`;
// the rotations gathered in V: c.Vf (NC = 1) or the
// ranks' rows in c.sX. A and lam[0] are synchronised on entry, V on exit.
// Returns the sweeps (rank 0; the others 0 or not 0).
template <class P, bool DELTA>
__device__ int pp_jacobi(const PpCtx<P>& c, int max_sweeps, float stop, float stop2) {
  const int p = c.p, lda = c.lda, m = (p + 1) & ~1;
  int A = c.Af, An = c.A2, lp = 0;
  const int w = c.tid >> 5;
  int v0 = 0, v1 = p, V = c.Vf, ldv = lda;
  if constexpr (P::NC > 1) {
    pp_vrows(c, v0, v1);
    V = 2 * c.sX;
    ldv = m;
  }
  for (int e = c.tid; e < (v1 - v0) * ldv; e += P::NT) {
    const int i = e / ldv, j = e - i * ldv;
    pp_sf(V)[e] = v0 + i == j ? 1.f : 0.f;
  }
  __syncthreads();
  int sweep = 0;
  bool reached = false;
  for (;; ++sweep) {
    bool go = true;
    const int log = sweep & 1 ? c.log1 : c.log0, prev = sweep & 1 ? c.log0 : c.log1;
    if (c.rank == 0) {
      const float* const a = pp_sf(A);
      float off = 0.f;
      for (int i = c.g; i < p; i += P::NG)
        for (int j = c.cl; j < p; j += P::CL)
          if (i != j) off += a[i * lda + j] * a[i * lda + j];
      off = pp_bsum<P>(off);
      go = sweep < max_sweeps && (off > stop || (!reached && off > stop2));
      reached = off <= stop;
      if constexpr (P::SEG == 64) {
        if (go) pp_sweep_wide<P, DELTA>(c, log);
      } else {
        if (w < P::AW) {
          if (go) pp_sweep<P, DELTA>(c, A, An, lp, log);
        } else if (P::NC == 1 && sweep > 0) {
          pp_apply_log<P>(p, V, ldv, p, prev, w - P::AW, P::NT / 32 - P::AW);
        }
        const int u = A;  // m - 1 rounds: odd
        A = An;
        An = u;
        lp ^= 1;
      }
    }
    if constexpr (P::NC == 1) {
      __syncthreads();
      if (!go) break;
    } else {
      float2* const word = c.gws + c.ctl + 4 + (sweep & 1);
      if (c.rank == 0 && c.tid == 0) *word = make_float2(go ? 1.f : 0.f, 0.f);
      pp_sync<P>();
      if (c.rank == 0) {
        if (!go) break;
      } else {
        if (__ldcg(&word->x) == 0.f) break;
        const int len = (int)pp_log_len(p);
        for (int e = c.tid; e < len; e += P::NT) pp_s2(c.sY)[e] = c.ldm(log + e);
        __syncthreads();
        pp_apply_log<P>(p, V, ldv, v1 - v0, c.sY, w, P::NT / 32);
        __syncthreads();
      }
    }
  }
  return sweep;
}

// Out = V (V^T V)^{-1/2} to third order in E = V^T V - I (E of about 1e-6:
// V comes from float32 rotations): Out = V + V G, G = -E/2 + 3/8 E^2, E^2 in
// float32. T is scratch; V is not changed. Synchronised on entry and exit.
template <class P>
__device__ void pp_orth(const PpCtx<P>& c, int V, int T, int Out) {
  pp_mm(c, V, true, V, false, T, -1, 1.f);  // E
  pp_sync<P>();
  for (int i = c.g; i < c.p; i += P::NG)
    for (int j = c.cl; j < c.p; j += P::CL) pp_sf(c.Af)[i * c.lda + j] = c.ldm(T + i * c.ld + j).x;
  pp_sync<P>();  // every rank has read T before its rows are replaced
  pp_each(c, [&](int i, int j) {
    float s = 0.f;
    for (int k = 0; k < c.p; ++k) s = fmaf(pp_sf(c.Af)[i * c.lda + k], pp_sf(c.Af)[k * c.lda + j], s);
    const float2 e = c.mat(T)[i * c.ld + j];
    c.mat(T)[i * c.ld + j] = df_add_f(make_float2(-0.5f * e.x, -0.5f * e.y), 0.375f * s);
  });
  pp_sync<P>();
  pp_mm(c, V, false, T, false, Out, V);
  pp_sync<P>();
}

// Eigenbasis of the symmetric c.Bd into c.Vd; c.Ud = V^T B V, diagonal up to
// rounding (`first_order` set: to first order in V -- the last correction of
// V is not put into Ud, whose off-diagonal part is then the corrected one's
// and whose diagonal is exact to second order). B is synchronised on entry.
template <class P>
__device__ void pp_eig(const PpCtx<P>& c, bool first_order, double* diag) {
  const int p = c.p, lda = c.lda, m = (p + 1) & ~1;
  PpSh* const sh = pp_sh();
  const long long c0 = clock64();
  float sc = 1.f;  // a power of two that brings max |B| near 1 (rank 0)
  int s32 = 0, s_delta = 0;  // sweeps
  // a control word of rank 0 to all ranks, and into a df64 matrix: nothing
  // (what = 0), the gathered rotations (1) or rank 0's c.Vf (2)
  auto publish = [&](int Vo, int word, int what) {
    float2* const V = c.mat(Vo);
    if (what == 0) {
    } else if (P::NC == 1 || what == 2) {
      if (c.rank == 0)
        for (int i = c.g; i < p; i += P::NG)
          for (int j = c.cl; j < p; j += P::CL) V[i * c.ld + j] = make_float2(pp_sf(c.Vf)[i * lda + j], 0.f);
    } else {
      int v0, v1;
      pp_vrows(c, v0, v1);
      const float* const sv = pp_sf(2 * c.sX);
      for (int i = v0 + c.g; i < v1; i += P::NG)
        for (int j = c.cl; j < p; j += P::CL) V[i * c.ld + j] = make_float2(sv[(i - v0) * m + j], 0.f);
    }
    if (c.rank == 0 && c.tid == 0) {
      sh->ctl = word;
      if (P::NC > 1) c.gws[c.ctl] = make_float2(__int_as_float(word), 0.f);
    }
    pp_sync<P>();
    return P::NC == 1 ? sh->ctl : __float_as_int(__ldcg(&c.gws[c.ctl].x));
  };
  float tot0 = 0.f;
  if (c.rank == 0) {
    float mx = 0.f;
    for (int i = c.g; i < p; i += P::NG)
      for (int j = c.cl; j < p; j += P::CL) mx = fmaxf(mx, fabsf(c.ldm(c.Bd + i * c.ld + j).x));
    mx = pp_bmax<P>(mx);
    const int ex = ((__float_as_int(mx) >> 23) & 255) - 127;
    if (mx > 0.f && ex <= 127) sc = exp2i(max(-126, min(126, -ex)));
    for (int i = c.g; i < m; i += P::NG)
      for (int j = c.cl; j < m; j += P::CL) {
        const float v = i < p && j < p ? c.ldm(c.Bd + i * c.ld + j).x * sc : 0.f;
        pp_sf(c.Af)[i * lda + j] = v;
        tot0 += v * v;
      }
    tot0 = pp_bsum<P>(tot0);  // (its barriers also publish A)
  }
  // down to ~1e-5 relative off-diagonal mass, above float32's rounding floor;
  // past p = 16 one sweep more brings the off-diagonal part to that floor,
  // where the gaps of most spectra leave the rest to the corrections below (at
  // p = 64 an extra sweep and three corrections take less than two sweeps
  // there, the orthogonalisation after them and one correction)
  s32 = pp_jacobi<P, false>(c, 12, 1e-10f * tot0, p > 16 ? 3e-13f * tot0 : tot0);
  const bool rotated = publish(c.Td, s32 > 0, 1) != 0;
  const long long c1 = clock64();
  if (rotated) {
    pp_orth(c, c.Td, c.Ud, c.Vd);
    pp_mm(c, c.Bd, false, c.Vd, false, c.Td);
    pp_sync<P>();
    pp_mm(c, c.Vd, true, c.Td, false, c.Ud);
  } else {
    pp_each(c, [&](int i, int j) {
      c.mat(c.Vd)[i * c.ld + j] = make_float2(i == j ? 1.f : 0.f, 0.f);
      c.mat(c.Ud)[i * c.ld + j] = c.mat(c.Bd)[i * c.ld + j];
    });
  }
  pp_sync<P>();
  const long long c2 = clock64();
  for (int pass = 0; pass < 4; ++pass) {
    // 0: done, 1: rotations in Td, 2: the last, first-order correction K in Td,
    // 3: a skew K in Td, V <- V exp(K), 4: the same, then orthogonalised
    int word = 0;
    float stop = 0.f;
    if (c.rank == 0) {
      // F scaled by 2^30 so that squares of entries at 1e-15 stay in range
      constexpr float UP = 1073741824.f;
      float off = 0.f, tot = 0.f;
      float2* const lam = sh->lam[0];
      for (int i = c.g; i < m; i += P::NG)
        for (int j = c.cl; j < m; j += P::CL) {
          float2 u = i < p && j < p ? c.ldm(c.Ud + i * c.ld + j) : make_float2(0.f, 0.f);
          u = make_float2(u.x * sc, u.y * sc);
          tot += u.x * u.x;
          if (i == j) {
            lam[i] = make_float2(u.x * UP, u.y * UP);
            pp_sf(c.Af)[i * lda + j] = 0.f;
          } else {
            off += u.x * u.x;
            pp_sf(c.Af)[i * lda + j] = u.x * UP;
          }
        }
      tot = pp_bsum<P>(tot);
      off = pp_bsum<P>(off);
      stop = 1e-30f * tot * UP * UP;
      if (off > 1e-27f * tot) {
        // K_ij = F_ij / (lambda_j - lambda_i) leaves F of the order |F| |K|,
        // without a sweep of its m - 1 dependent rounds. Up to |K| = 2e-4,
        // I + K + K^2 / 2 with K^2 in df64 is orthogonal to |K|^4 / 4 = 4e-16.
        // Up to |K| = 0.07 (single small gaps) the pairs' exact angles and an
        // orthogonalisation of the result (which leaves |K|^12 / 200) still
        // replace the sweeps.
        // Angles below 1e-8 are I + K to working accuracy. K is made exactly
        // skew from the upper half of F: the halves differ by rounding,
        // which over a small gap would leave V off orthogonal. Small gaps
        // (clusters, tiny eigenvalues) take the rotations instead.
        float kmax = 0.f, kf = 0.f;
        for (int i = c.g; i < p; i += P::NG)
          for (int j = c.cl; j < p; j += P::CL)
            if (i < j) {
              const float2 d = df_add(lam[j], pp_neg(lam[i]));
              const float f = pp_sf(c.Af)[i * lda + j];
              float k = f == 0.f ? 0.f : f / d.x;
              if (fabsf(k) > 1e-4f) k = 0.5f * atanf(2.f * k);
              pp_sf(c.Vf)[i * lda + j] = k;
              pp_sf(c.Vf)[j * lda + i] = -k;
              kmax = fmaxf(kmax, fabsf(k));
              kf += k * k;
            } else if (i == j) {
              pp_sf(c.Vf)[i * lda + i] = 0.f;
            }
        kmax = pp_bmax<P>(kmax);
        kf = pp_bsum<P>(kf);
        word = first_order && pass > 0 && kmax <= 1e-8f ? 2 : kf <= 4e-8f ? 3 : kf <= 5e-3f ? 4 : 1;
      }
    }
    word = publish(c.Td, word, word >= 2 ? 2 : 0);
    if (word == 1) {
      s_delta += pp_jacobi<P, true>(c, 8, stop, stop);
      publish(c.Td, 1, 1);
    }
    if (word == 0) break;
    if (word == 2) {  // V += V K
      pp_mm(c, c.Vd, false, c.Td, false, c.Bd, c.Vd);
      pp_sync<P>();
      pp_each(c, [&](int i, int j) { c.mat(c.Vd)[i * c.ld + j] = c.mat(c.Bd)[i * c.ld + j]; });
      pp_sync<P>();
      break;
    }
    if (word >= 3) {  // V += V (K + K^2 / 2)
      for (int i = c.g; i < p; i += P::NG)
        for (int j = c.cl; j < p; j += P::CL) pp_sf(c.Af)[i * lda + j] = c.ldm(c.Td + i * c.ld + j).x;
      pp_sync<P>();  // every rank has read Td before its rows are replaced
      pp_each(c, [&](int i, int j) {
        float h = 0.f, e = 0.f;
        for (int k = 0; k < p; ++k) {
          const float x = pp_sf(c.Af)[i * lda + k], y = pp_sf(c.Af)[k * lda + j], pr = __fmul_rn(x, y);
          const float2 t = two_sum(h, pr);
          h = t.x;
          e = __fadd_rn(e, __fadd_rn(t.y, __fmaf_rn(x, y, -pr)));
        }
        c.mat(c.Td)[i * c.ld + j] =
            df_add(make_float2(pp_sf(c.Af)[i * lda + j], 0.f), two_sum(0.5f * h, 0.5f * e));
      });
      pp_sync<P>();
    }
    pp_mm(c, c.Vd, false, c.Td, false, c.Ud, word >= 3 ? c.Vd : -1);  // or V W
    pp_sync<P>();
    if (word == 3) {
      pp_each(c, [&](int i, int j) { c.mat(c.Vd)[i * c.ld + j] = c.mat(c.Ud)[i * c.ld + j]; });
      pp_sync<P>();
    } else {
      pp_orth(c, c.Ud, c.Td, c.Vd);
    }
    // U = V^T B V
    pp_mm(c, c.Bd, false, c.Vd, false, c.Td);
    pp_sync<P>();
    pp_mm(c, c.Vd, true, c.Td, false, c.Ud);
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

__device__ __forceinline__ float2 df_div(float2 a, float2 b) {
  const float q1 = __fdiv_rn(a.x, b.x);
  const float p = __fmul_rn(q1, b.x);
  const float e = __fmaf_rn(q1, b.y, __fmaf_rn(q1, b.x, -p));
  const float2 r = df_add(a, make_float2(-p, -e));
  return fast_two_sum(q1, __fdiv_rn(__fadd_rn(r.x, r.y), b.x));
}

// M = V [diag(s^-1/2) + F o Df] V^T for S' = diag(s) + F in c.Ud, df64 into
// c.Ud and float64 into M; status (0, or 5 if some s_i is not positive) in
// sh->flag of every CTA.
template <class P>
__device__ void pp_inv_sqrt(const PpCtx<P>& c, double* M) {
  PpSh* const sh = pp_sh();
  const int p = c.p;
  if (c.tid < 32) {
    double mx = 0.0;
    for (int i = c.tid; i < p; i += 32) {
      const double s = df_to_double(c.ldm(c.Ud + i * c.ld + i));
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
      sh->svf[i] = df_from_double(sh->sv[i]);
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
      const float2 ri = sh->svf[i], rj = sh->svf[j];
      v = df_div(df_div(df_div(pp_neg(c.mat(c.Ud)[i * c.ld + j]), ri), rj), df_add(ri, rj));
    }
    c.mat(c.Ud)[i * c.ld + j] = v;
  });
  pp_sync<P>();
  pp_mm(c, c.Vd, false, c.Ud, false, c.Td);  // V N
  pp_sync<P>();
  pp_mm(c, c.Td, false, c.Vd, true, c.Ud);   // (V N) V^T
  pp_sync<P>();
  pp_each(c, [&](int i, int j) { M[i * p + j] = df_to_double(c.mat(c.Ud)[i * c.ld + j]); });
}

// this CTA's rows of an input into a df64 matrix
template <class P, class F>
__device__ __forceinline__ void pp_load(const PpCtx<P>& c, const PpMat& a, int dsto, F f) {
  const int p = c.p;
  float2* const dst = c.mat(dsto);
  pp_each(c, [&](int i, int j) {
    float2 v;
    if (a.f) v = a.f[i * p + j];
    else if (a.sym) v = df_from_double(0.5 * (a.d[i * p + j] + a.d[j * p + i]));
    else v = df_from_double(a.d[i * p + j]);
    dst[i * c.ld + j] = f(i, j, v);
  });
}

// ---- the exact step of Alg. 3 ------------------------------------------------

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

// the search in float64 throughout, where the scaled model does not serve
static __device__ __noinline__ double pp_step_length_f64(int p, int* ev) {
  const PpSh* const sh = pp_sh();
  return get_mu_warp(p, sh->al, sh->be, sh->ga, sh->ze, ev);
}

__device__ __forceinline__ float2 df_sqrt(float2 a) {  // a >= 0
  if (!(a.x > 0.f)) return make_float2(0.f, 0.f);
  const float y = __fsqrt_rn(a.x), y2 = __fmul_rn(y, y);
  const float2 r = df_add(a, make_float2(-y2, -__fmaf_rn(y, y, -y2)));
  return fast_two_sum(y, __fdiv_rn(__fadd_rn(r.x, r.y), 2.f * y));
}
__device__ __forceinline__ float2 df_scale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
// a 2^e for |e| beyond a float's exponent
__device__ __forceinline__ float2 df_ldexp(float2 a, int e) { return make_float2(ldexpf(a.x, e), ldexpf(a.y, e)); }

// The step of get_mu_warp (alg3.cuh: bracket from the branch roots xi_i, the
// right end doubled from xi_min, Brent on phi'), one warp. The search runs in
// df64 on a model scaled by powers of two (a float64 evaluation is a chain of
// ~25 operations on a pipe with 1/64 of the float32 rate, ~5,000 cycles an
// evaluation); the root is then corrected by one Newton step from a float64
// evaluation of phi', which leaves it as accurate as a search in float64.
// Where the scaled model leaves float32's range or the Newton step is not
// small, the float64 search runs instead.
template <int MC>
__device__ __noinline__ double pp_step_length(int p, int* ev_out) {
  const PpSh* const sh = pp_sh();
  int evs = 0, *const ev = &evs;
  const int lane = threadIdx.x & 31;
  PpModel<MC> md;
  float sb = 0.f, bmax = 0.f, zmax = 0.f, dmax = 0.f;
  md.cnt = 0;
#pragma unroll
  for (int u = 0; u < MC; ++u) {
    const int i = lane + 32 * u;
    md.z[u] = md.dl[u] = md.b[u] = make_float2(0.f, 0.f);
    if (i < p) {
      md.b[u] = sh->bef[i];
      md.z[u] = sh->zef[i];
      md.dl[u] = df_add(sh->gaf[i], pp_neg(df_mul(sh->alf[i], md.b[u])));
      md.cnt = u + 1;
      sb += md.b[u].x;
      bmax = fmaxf(bmax, md.b[u].x);
      zmax = fmaxf(zmax, fabsf(md.z[u].x));
      dmax = fmaxf(dmax, fabsf(md.dl[u].x));
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    sb += __shfl_xor_sync(0xffffffffu, sb, o);
    bmax = fmaxf(bmax, __shfl_xor_sync(0xffffffffu, bmax, o));
    zmax = fmaxf(zmax, __shfl_xor_sync(0xffffffffu, zmax, o));
    dmax = fmaxf(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
  }
  sb = __shfl_sync(0xffffffffu, sb, 0);
  // t = T tau with T = min(1/sqrt(max beta), max|zeta| / max|delta|), values
  // over Sz = max|zeta|, each rounded down to a power of two
  const bool range = bmax > 1e-36f && bmax < 1e36f && zmax > 1e-36f && zmax < 1e36f && dmax < 1e36f;
  int eT = 0, eZ = 0;
  if (range) {
    eZ = ilogbf(zmax);
    eT = -((ilogbf(bmax) + 2) / 2);
    if (dmax > 0.f) eT = min(eT, eZ - ilogbf(dmax));
  }
  // (alpha and gamma enter through delta only, so that an empty bracket and a
  // model without positive zeta are the same here as in the float64 search)
  float2 xmn = make_float2(INFINITY, 0.f), xmx = make_float2(0.f, 0.f);
  bool any = false;
#pragma unroll
  for (int u = 0; u < MC; ++u) {
    const bool use = u < md.cnt && md.b[u].x > (float)ALG3_EPS * sb && md.z[u].x > 0.f;
    any = any || use;
    md.b[u] = df_ldexp(md.b[u], 2 * eT);
    md.z[u] = df_ldexp(md.z[u], -eZ);
    md.dl[u] = df_ldexp(md.dl[u], eT - eZ);
    md.bz[u] = df_mul(md.b[u], md.z[u]);
    if (use) {
      const float2 d = md.dl[u], z = md.z[u];
      const float2 disc = df_sqrt(df_add(df_mul(d, d), df_scale(df_mul(md.bz[u], z), 4.f)));
      float2 xi;
      if (d.x < 0.f) xi = df_div(df_scale(z, 2.f), df_add(disc, pp_neg(d)));
      else xi = df_div(df_add(d, disc), df_scale(md.bz[u], 2.f));
      if (!(xi.x < 1e30f)) xi = make_float2(1e30f, 0.f);  // past the largest step searched, or 2 b z underflowed
      if (df_less(xi, xmn)) xmn = xi;
      if (df_less(xmx, xi)) xmx = xi;
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    const float2 lo = make_float2(__shfl_xor_sync(0xffffffffu, xmn.x, o), __shfl_xor_sync(0xffffffffu, xmn.y, o));
    const float2 hi = make_float2(__shfl_xor_sync(0xffffffffu, xmx.x, o), __shfl_xor_sync(0xffffffffu, xmx.y, o));
    if (df_less(lo, xmn)) xmn = lo;
    if (df_less(xmx, hi)) xmx = hi;
  }
  *ev_out = 0;
  if (!range || !__any_sync(0xffffffffu, any) || !(xmn.x > 1e-9f) || !(xmn.x < 1e9f))
    return pp_step_length_f64(p, ev_out);
  const float2 fa = pp_dphi(md, xmn);
  ++*ev;
  float2 lo, flo, hi, fhi;
  if (fa.x > 0.f) {
    lo = make_float2(0.f, 0.f);
    flo = pp_dphi(md, lo);
    ++*ev;
    if (flo.x >= 0.f) return pp_step_length_f64(p, ev_out);
    hi = xmn;
    fhi = fa;
  } else {
    lo = hi = xmn;
    flo = fhi = fa;
    int k = 0;
    while (fhi.x < 0.f) {
      if (k >= 64 || hi.x > 1e18f) return pp_step_length_f64(p, ev_out);
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
  const double f = dphi_warp(t, p, sh->al, sh->be, sh->ga, sh->ze);
  ++*ev;
  // phi' over Sz and the slope are of order one; the quotient is the step in tau
  const float corr = (float)scalbn(f, -eZ) / sl;
  if (!(fabsf(corr) <= 1e-9f * tau.x)) return pp_step_length_f64(p, ev_out);
  *ev_out = evs;
  return t - scalbn((double)corr, eT);
}

// The diagonal of V^T G V (G in c.Ud, V in c.Vd) into d (shared memory of
// every CTA). The row groups' sums pass through c.Af, the ranks' through the
// control words. Synchronised on exit.
template <class P>
__device__ void pp_diag(const PpCtx<P>& c, double* d, float2* df) {
  const int p = c.p;
  float2* const part = pp_s2(c.Af / 2);
  pp_mm(c, c.Ud, false, c.Vd, false, -1, -1, 0.f, c.Vd, c.Af / 2);
  __syncthreads();
  for (int j = c.tid; j < p; j += P::NT) {
    float2 s = part[j];
    for (int g = 1; g < P::RG; ++g) s = df_add(s, part[g * p + j]);
    if constexpr (P::NC == 1) {
      d[j] = df_to_double(s);
      df[j] = s;
    } else c.gws[c.ctl + 64 + c.rank * 128 + j] = s;
  }
  pp_sync<P>();
  if constexpr (P::NC > 1) {
    for (int j = c.tid; j < p; j += P::NT) {
      const float2* const pd = c.gws + c.ctl + 64 + j;
      float2 s = __ldcg(pd);
      for (int g = 1; g < P::NC; ++g) s = df_add(s, __ldcg(pd + g * 128));
      d[j] = df_to_double(s);
      df[j] = s;
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
  PpSh* const sh = pp_sh();
  double* out = a.out;
  const bool lead = c.rank == 0 && c.tid == 0;
  const long long t0 = clock64();
  auto same = [](int, int, float2 v) { return v; };
  if (a.mode == 4) {
    pp_each(c, [&](int i, int j) { c.mat(c.Vd)[i * c.ld + j] = a.eig[i * p + j]; });
    for (int i = c.tid; i < p; i += P::NT) {
      const float2 b = a.eig[p * p + i];
      sh->bef[i] = b.x > 0.f ? b : make_float2(0.f, 0.f);
      sh->be[i] = df_to_double(sh->bef[i]);
    }
    __syncthreads();
  } else {
    if (a.scale_b) {
      float ex = 0.f;  // largest biased exponent
      for (int e = c.tid; e < p * p; e += P::NT) ex = fmaxf(ex, (float)((__double2hiint(a.B.d[e]) >> 20) & 0x7ff));
      ex = pp_bmax<P>(ex);
      const int k = ex < 2047.f ? max(1, 2046 - (int)ex) : 1023;
      const double sb = __hiloint2double(k << 20, 0);
      pp_each(c, [&](int i, int j) {
        c.mat(c.Bd)[i * c.ld + j] = df_from_double(0.5 * (sb * a.B.d[i * p + j]) + 0.5 * (sb * a.B.d[j * p + i]));
      });
    } else {
      pp_load(c, a.B, c.Bd, same);
    }
    pp_sync<P>();
    pp_eig(c, a.mode != 1, out + 8);
    if (a.mode == 0) {
      for (int i = c.tid; i < p; i += P::NT) {
        const float2 b = c.ldm(c.Ud + i * c.ld + i);
        sh->bef[i] = b.x > 0.f ? b : make_float2(0.f, 0.f);
        sh->be[i] = df_to_double(sh->bef[i]);
      }
      __syncthreads();
    }
  }
  const long long t1 = clock64();
  if (a.mode == 3) {
    pp_each(c, [&](int i, int j) {
      a.eig[i * p + j] = c.mat(c.Vd)[i * c.ld + j];
      if (i == j) a.eig[p * p + i] = c.mat(c.Ud)[i * c.ld + i];
    });
    if (lead) out[5] = (double)(t1 - t0);
    return;
  }
  if (a.mode == 2) {
    pp_each(c, [&](int i, int j) {
      a.M[i * p + j] = df_to_double(c.mat(c.Vd)[i * c.ld + j]);
      if (i == j) a.theta[i] = df_to_double(c.mat(c.Ud)[i * c.ld + i]);
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
  pp_diag(c, sh->al, sh->alf);
  pp_load(c, a.Gam, c.Ud, same);
  pp_sync<P>();
  pp_diag(c, sh->ga, sh->gaf);
  pp_load(c, a.Z, c.Ud, same);
  pp_sync<P>();
  pp_diag(c, sh->ze, sh->zef);
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
    pp_mm(c, c.Ud, false, c.Td, false, c.Bd);
  }
  pp_sync<P>();
  const long long t2 = clock64();
  if (c.tid < 32) {
    if (c.rank == 0) {
      int ev = 0;
      const double t = pp_step_length<(P::CL * P::TC * P::NCG + 31) / 32>(p, &ev);
      float2 bmax = make_float2(0.f, 0.f);
      for (int i = c.tid; i < p; i += 32)
        if (df_less(bmax, sh->bef[i])) bmax = sh->bef[i];
      for (int o = 16; o > 0; o >>= 1) {
        const float2 v = make_float2(__shfl_xor_sync(0xffffffffu, bmax.x, o), __shfl_xor_sync(0xffffffffu, bmax.y, o));
        if (df_less(bmax, v)) bmax = v;
      }
      // the model's value is reported to direct callers only
      const double ph = a.mode == 0 && a.want_phi ? phi_model_warp(t, p, sh->al, sh->be, sh->ga, sh->ze) : 0.0;
      if (c.tid == 0) {
        sh->t = t;
        if (P::NC > 1) *reinterpret_cast<double*>(c.gws + c.ctl + 2) = t;
        out[0] = t;
        out[1] = ph;
        out[2] = (double)ev;
        out[4] = df_to_double(bmax);
      }
    }
  }
  pp_sync<P>();
  const double t = P::NC == 1 ? sh->t : __ldcg(reinterpret_cast<const double*>(c.gws + c.ctl + 2));
  const long long t3 = clock64();
  // S' = V^T S V with S = XX + t (XD + XD^T) + t^2 B, summed in float64
  auto elem = [&](const PpMat& g, int i, int j) {
    return g.sym ? 0.5 * (g.d[i * p + j] + g.d[j * p + i]) : g.d[i * p + j];
  };
  pp_each(c, [&](int i, int j) {
    // X^T D as the caller holds it, where it was given
    const double xd = a.XD.d ? a.XD.d[i * p + j] + a.XD.d[j * p + i]
                             : df_to_double(c.ldm(c.Bd + i * c.ld + j)) + df_to_double(c.ldm(c.Bd + j * c.ld + i));
    c.mat(c.Ud)[i * c.ld + j] = df_from_double(fma(t, xd, elem(a.XX, i, j)) + t * t * elem(a.B, i, j));
  });
  pp_sync<P>();
  pp_mm(c, c.Ud, false, c.Vd, false, c.Td);
  pp_sync<P>();
  pp_mm(c, c.Vd, true, c.Td, false, c.Ud);
  pp_sync<P>();
  pp_inv_sqrt(c, a.M);
  if (lead) out[3] = (double)sh->flag;
  // K_next = X_new^T D = M T, T = X^T D + t D^T D, in float64: it goes into the
  // next direction and X^T D with no correction after it. The product takes
  // p^3 / 2 cycles of an SM's float64 pipe (p = 16: 3 us of a step's 98; p = 32
  // 13 of 200; on a cluster at p = 128 70 of 1640), so a solve forms it here up
  // to p = PP_K_INSIDE only and takes T for a product over many SMs beyond; the
  // batch, with a block per problem, always forms it here. T and M leave df64
  // once (a conversion costs as much as a multiply-add), in the space of T, V.
  auto t_elem = [&](int i, int j) { return fma(t, elem(a.B, i, j), df_to_double(c.mat(c.Bd)[i * c.ld + j])); };
  if (a.Tn) pp_each(c, [&](int i, int j) { a.Tn[i * p + j] = t_elem(i, j); });
  if constexpr (P::NC == 1) {
    if (a.Kd) {
      double* const T = reinterpret_cast<double*>(pp_s2(c.Td));
      double* const Md = reinterpret_cast<double*>(pp_s2(c.Vd));
      pp_each(c, [&](int i, int j) {
        T[i * p + j] = t_elem(i, j);
        Md[i * p + j] = df_to_double(c.mat(c.Ud)[i * c.ld + j]);
      });
      __syncthreads();
      pp_each(c, [&](int i, int j) {
        double v = 0.0;
#pragma unroll 4
        for (int k = 0; k < p; ++k) v = fma(Md[i * p + k], T[k * p + j], v);
        a.Kd[i * p + j] = v;
      });
    }
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
