// SVD of a centre matrix to FP64 accuracy by refining the V of FP32 sweeps with
// matrix products, over the CTAs of a cluster.
//
// The FP64 Jacobi's rounds are chains of FP64 instructions and cluster exchanges
// (10-12k cycles a round, three to ten sweeps of ncol - 1 rounds), although what is
// left after the FP32 sweeps are small rotations.  All of them at once are one
// product (Ogita and Aishima, "Iterative refinement for symmetric eigenvalue
// decomposition", 2018): with W = X V, S = W^T W and R = I - V^T V,
//   V <- V (I + E),  E_ij = R_ij / 2 + t_ij,
// t_ij (antisymmetric) the Jacobi tangent of g = S_ij + (l_i + l_j) R_ij / 2 against
// l_j - l_i.  A step squares both the cosines between the columns of W, as a Jacobi
// sweep does, and R.  Only V^T V, X V and W^T W need long sums; the correction V E is
// small, so its FP32 product is accurate enough (6e-8 of the correction).
//
// The long sums of FP32 data are compensated FP32 sums of exact products on pairs of
// floats (Ogita, Rump and Oishi's Dot2: 48 bits, 12 instructions a product), as
// GB300 does 64 FP32 operations in the time of one FP64; FP64 data take FP64.  Against 64-bit
// results nothing is lost to FP64 sums: kept against discarded directions of 80 matrices of 64 to
// 180 columns at six and nine decades, rms 1.05e-7 to 2.17e-7 with the pairs, 1.06e-7 to
// 2.19e-7 with FP64 sweeps in their place (FP32 storage rounds at 6e-8).
//
// FP32 sweeps leave the cosine of columns i, j at ~1e-7 s_0 / min(s_i, s_j): nothing
// for the small ones.  So where a tangent is not small, a second FP32 Jacobi runs on W
// itself (and a third if need be), whose columns now carry their own scale: its errors are relative to each
// column.  Its product of rotations J is applied with long sums (V <- V J).  V is
// made orthonormal first: R_ij between a large and a small column would come back
// as R_ij s_i / 2 in the small one.
//
// Pairs whose singular values agree to ~1e-5 (|t| large although the cosine is
// below 1e-5) may keep their cosine: any basis of their span serves, since V stays
// orthonormal, W = X V holds whatever the basis, and the discarded weight is the sum
// of the discarded |w_j|^2.  Where the rank rule cuts between two such columns the basis
// is the result: the caller lets the sweeps turn them (RF_TIE, RefineMem::tied).
//
// Work is split by columns: CTA c owns columns [c n / P, (c + 1) n / P) of V, W, S and
// E, all in the job's scratch (L2); a cluster barrier separates the steps.  What is
// left undone (large tangents after RF_PASSES Jacobis, no convergence in RF_STEPS)
// goes to the FP64 Jacobi sweeps, started from the V reached.
//
// Measured against FP64 sweeps from the V of FP32 sweeps (FP64 data: from V = I): 128^3
// sums of two at bond 64, mixed, 128 -> 40 ms; 64^3 sums at bond 45, FP64, 82 -> 49 ms; a step
// of a mixed 64^3 box at bond 32, 354 -> 160 ms.
#pragma once

#include "cluster.cuh"
#include "jacobi_reg.cuh"

namespace tn {

static constexpr int RF_KC = 8;          // rows of k that at least are staged at a time
static constexpr int RF_STEPS = 12;      // steps V <- V (I + E) at most
static constexpr int RF_PASSES = 2;      // FP32 Jacobis of W at most
static constexpr double RF_TIE = 2e-4;   // squared norms that agree to this may be of a pair that kept its cosine (|t| > 0.1, cosine <= 1e-5)
static constexpr int RF_MIN = 6;         // columns from which it is taken: below, the few rounds of the sweeps cost less

// A number of ~48 bits as the unevaluated sum of two floats (x = the rounded value),
// or a double: `N` below.
__device__ __forceinline__ void rf_mac(float2& a, float2 x, float2 y) {
  const float p = __fmul_rn(x.x, y.x);
  float r = fmaf(x.x, y.x, -p);
  const float t = __fadd_rn(a.x, p), b = __fadd_rn(t, -a.x);
  const float e = __fadd_rn(__fadd_rn(a.x, -__fadd_rn(t, -b)), __fadd_rn(p, -b));
  r = fmaf(x.x, y.y, r);
  r = fmaf(x.y, y.x, r);
  a.x = t;
  a.y += e + r;
}
__device__ __forceinline__ void rf_mac(double& a, double x, double y) { a = fma(x, y, a); }
__device__ __forceinline__ void rf_mac(float& a, float x, float y) { a = fmaf(x, y, a); }
__device__ __forceinline__ void rf_zero(float2& a) { a = make_float2(0.f, 0.f); }
__device__ __forceinline__ void rf_zero(double& a) { a = 0.0; }
__device__ __forceinline__ void rf_zero(float& a) { a = 0.f; }
__device__ __forceinline__ float2 rf_sum(float2 a) {       // the normalised pair
  const float h = __fadd_rn(a.x, a.y);
  return make_float2(h, __fadd_rn(a.y, -__fadd_rn(h, -a.x)));
}
__device__ __forceinline__ double rf_sum(double a) { return a; }
__device__ __forceinline__ float2 rf_add(float2 a, float v) {       // a + v, any order of magnitude
  const float t = __fadd_rn(a.x, v), b = __fadd_rn(t, -a.x);
  const float e = __fadd_rn(__fadd_rn(a.x, -__fadd_rn(t, -b)), __fadd_rn(v, -b));
  return rf_sum(make_float2(t, a.y + e));
}
__device__ __forceinline__ double rf_add(double a, float v) { return a + (double)v; }
__device__ __forceinline__ float rf_f(float2 a) { return a.x + a.y; }
__device__ __forceinline__ float rf_f(double a) { return (float)a; }
__device__ __forceinline__ double rf_d(float2 a) { return (double)a.x + (double)a.y; }
__device__ __forceinline__ double rf_d(double a) { return a; }
__device__ __forceinline__ double rf_d(float a) { return (double)a; }
// a - b, rounded to FP32 from the exact difference (up to the pairs' own error)
__device__ __forceinline__ float rf_diff(float2 a, float2 b) { return __fadd_rn(a.x, -b.x) + __fadd_rn(a.y, -b.y); }
__device__ __forceinline__ float rf_diff(double a, double b) { return (float)(a - b); }
template <typename N> __device__ __forceinline__ N rf_make(float v);
template <> __device__ __forceinline__ float2 rf_make<float2>(float v) { return make_float2(v, 0.f); }
template <> __device__ __forceinline__ double rf_make<double>(float v) { return (double)v; }
template <typename N> __device__ __forceinline__ N rf_make(double v);
template <> __device__ __forceinline__ float2 rf_make<float2>(double v) { return make_float2((float)v, 0.f); }  // v is a float
template <> __device__ __forceinline__ double rf_make<double>(double v) { return v; }
__device__ __forceinline__ float2 rf_shfl(float2 a, int o) {
  return make_float2(__shfl_xor_sync(0xffffffffu, a.x, o), __shfl_xor_sync(0xffffffffu, a.y, o));
}
__device__ __forceinline__ double rf_shfl(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ float2 rf_plus(float2 a, float2 b) {
  const float2 s = rf_add(a, b.x);
  return rf_sum(make_float2(s.x, s.y + b.y));
}
__device__ __forceinline__ double rf_plus(double a, double b) { return a + b; }

// Shared memory: the own columns of one operand (8 bytes an entry), the own columns
// of R and of E (floats), the squared norms, and at least RF_KC staged rows of the
// other operand.
__host__ __device__ inline size_t rf_fixed(int ncol, int len, int P) {
  const int big = imax(ncol, len), vi = (ncol + P - 1) / P;
  return (((size_t)big * vi + ncol) * 8 + 2 * (size_t)big * vi * 4 + 15) & ~(size_t)15;
}
__host__ __device__ inline size_t rf_bytes(int ncol, int len, int P) {
  return rf_fixed(ncol, len, P) + (size_t)RF_KC * (imax(ncol, len) + 1) * 8;
}

// Columns [0, nb) of out(i, j) = sum_k A(k, i) B(k, j), i < M, k < K, with B (K x nb,
// column j at B + j * ldb, shared memory) and A(k, i) = a(k, i) staged as far as
// `room` bytes at st allow (kfast: consecutive k are consecutive in memory).
// emit(i, j, value) gets each entry from one thread.  N: the type of the sums.
template <typename N, typename FA, typename FE>
__device__ __forceinline__ void rf_gemm(int M, int nb, int K, FA&& a, bool kfast, const N* B, int ldb, N* st, size_t room,
                                        FE&& emit) {
  const int mr = (M + 31) & ~31;                         // threads along i
  const int ng = imax(1, (int)blockDim.x / mr);
  const int lds = M | 1;
  const int kc = imin(K, (int)(room / ((size_t)lds * sizeof(N))));
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int i0 = 0; i0 < M; i0 += blockDim.x) {
    const int i = i0 + (int)threadIdx.x % mr, g = threadIdx.x / mr;
    for (int j0 = 0; j0 < nb; j0 += 4 * ng) {
      N acc[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) rf_zero(acc[q]);
      const bool act = i < M && g < ng;
      const int nq = j0 + g >= nb ? 0 : imin(4, (nb - j0 - g + ng - 1) / ng);
      for (int k0 = 0; k0 < K; k0 += kc) {
        const int nk = imin(kc, K - k0);
        if (kc < K || (i0 == 0 && j0 == 0)) {            // else it is all there
          __syncthreads();
          // four rows' (columns') loads in flight per warp
          const int n1 = kfast ? M : nk, n0 = kfast ? nk : M;
          for (int u = wid; u < n1; u += 4 * nw)
            for (int f = lane; f < n0; f += 32) {
              N t[4];
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const int w = imin(u + q * nw, n1 - 1);
                t[q] = kfast ? a(k0 + f, w) : a(k0 + w, f);
              }
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const int w = u + q * nw;
                if (w < n1) st[kfast ? (size_t)f * lds + w : (size_t)w * lds + f] = t[q];
              }
            }
          __syncthreads();
        }
        if (act && nq > 0) {
          const N* b = B + (size_t)(j0 + g) * ldb + k0;
          const N* s = st + i;
          const size_t bs = (size_t)ng * ldb;
          if (nq == 1) {
#pragma unroll 8
            for (int kk = 0; kk < nk; ++kk) rf_mac(acc[0], s[(size_t)kk * lds], b[kk]);
          } else if (nq == 2) {
#pragma unroll 4
            for (int kk = 0; kk < nk; ++kk) {
              const N x = s[(size_t)kk * lds];
              rf_mac(acc[0], x, b[kk]);
              rf_mac(acc[1], x, b[bs + kk]);
            }
          } else {
#pragma unroll 2
            for (int kk = 0; kk < nk; ++kk) {
              const N x = s[(size_t)kk * lds];
#pragma unroll
              for (int q = 0; q < 4; ++q)
                if (q < nq) rf_mac(acc[q], x, b[q * bs + kk]);
            }
          }
        }
      }
      if (act)
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (q < nq) emit(i, j0 + g + q * ng, acc[q]);
    }
  }
  __syncthreads();
}

// Largest of v over the block (v >= 0), the same in every thread.
__device__ inline float rf_block_max(float v, float* red) {
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  float m = red[threadIdx.x & ((blockDim.x >> 5) - 1)];    // a power of two of warps
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  __syncthreads();
  return m;
}

// The job's scratch for a refinement (all global, column-major).
template <typename N>
struct RefineMem {
  N *V, *V2;               // n x n, ldv
  N* W;                    // len x n, ldw
  float* J;                // n x n, ldj: the second Jacobi's rotations
  N* nrm;                  // n squared column norms
  float* stat;             // [2][CL_MAX][4] maxima of every CTA
  float2* log;
  int ldv, ldw, ldj;
  int turn;                // meetings so far (the slots of stat alternate)
  bool tied;               // pairs of equal singular values have kept their cosine
};

// All CTAs meet; the maxima over the cluster of the four values v (thread-uniform
// per CTA) come back in v.
template <typename N>
__device__ __forceinline__ bool rf_meet_max(ClusterCtx& cc, RefineMem<N>& m, float (&v)[4]) {
  int& turn = m.turn;
  if (threadIdx.x == 0) __stcg((float4*)(m.stat + ((size_t)(turn & 1) * CL_MAX + cc.rank) * 4), make_float4(v[0], v[1], v[2], v[3]));
  if (!cl_sync(cc)) return false;
  const int c = threadIdx.x & 15;
  float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
  if (c < cc.P) a = __ldcg((const float4*)(m.stat + ((size_t)(turn & 1) * CL_MAX + c) * 4));
  for (int o = 8; o > 0; o >>= 1) {
    a.x = fmaxf(a.x, __shfl_xor_sync(0xffffffffu, a.x, o));
    a.y = fmaxf(a.y, __shfl_xor_sync(0xffffffffu, a.y, o));
    a.z = fmaxf(a.z, __shfl_xor_sync(0xffffffffu, a.z, o));
    a.w = fmaxf(a.w, __shfl_xor_sync(0xffffffffu, a.w, o));
  }
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
  ++turn;
  return true;
}

// What the refinement of X (len x n, X(i, k) = x(i, k)) reached: RF_DONE: V orthonormal
// and W = X V with orthogonal columns; RF_SWEEPS: V orthonormal, the FP64 sweeps have
// to finish; RF_DEAD: this CTA has given up waiting.
enum : int { RF_DONE = 0, RF_SWEEPS = 1, RF_DEAD = 2 };

// m.V holds the start (FP32 accuracy); go_on false: it is made orthonormal, no more
// (the FP32 sweeps met the caller's limit).  kfast: consecutive k of x(i, .) are
// consecutive in memory.  ties: pairs of equal singular values may keep their
// cosine.  jacobi(): one FP32 Jacobi of W by the leader with its rotations formed in
// m.J over the cluster (false: not available).  A pair is orthogonal if its squared
// cosine is at most tol2, or if its tangent t is small enough to be W's rounding:
// own_scale: |t| <= tmin, to the columns' own scale; else |t| s_i <= tmin s_0 for its larger
// column.  W = X V carries a rounding of s_0, which turns small columns by more than
// their own scale, but the rows of a centre matrix are graded as its singular values are, and
// then small directions are as well determined as large ones: FP64 roundings need the own
// scale (with s_0, 1e-12 in the start of a porous 128^3 flow grew to 4.6e-7 in three steps at
// bond 64, where the FP64 sweeps and the own scale have 6.0e-9 and 2.9e-9).  FP32 data hold nothing
// below s_0 tmin: 128^3 sums at bond 64, mixed, 40 ms, with the own scale 57; 256^3 at bond 128,
// 142 and 232.  FP64 pays 64^3 sums at bond 45 47.9 -> 49.4 ms, 32^3 walls 13.1 -> 14.5.  Eigenproblems of
// Gram matrices (REFINE_TOP) hold nothing below s_0's rounding either.
// small: the largest |E| whose square, and whose FP32 product's error, are below
// what V has to be accurate to; ready: the |R| from which a Jacobi of W pays; none:
// squared norms (relative to the largest) of columns whose pairs carry nothing.
template <typename N, typename FX, typename FJ>
__device__ __noinline__ int rf_refine(ClusterCtx& cc, RefineMem<N>& m, int n, int len, bool go_on, FX x, bool kfast,
                                      bool ties, float tol2, float tmin, bool own_scale, float small, float ready, float none, int at, int room,
                                      FJ jacobi) {
  extern __shared__ __align__(16) unsigned char smem[];
  unsigned char* wa = smem + at;                           // the work area (`room` bytes), known to be shared memory
  __shared__ float s_red[32];
  const int v0 = cc.rank * n / cc.P, vi = (cc.rank + 1) * n / cc.P - v0;
  const int big = imax(n, len), vmax = (n + cc.P - 1) / cc.P;
  N* blk = (N*)wa;
  N* nr = blk + (size_t)big * vmax;
  float* R = (float*)(nr + n);
  float* E = R + (size_t)big * vmax;
  const size_t fixed = rf_fixed(n, len, cc.P);
  N* st = (N*)(wa + fixed);
  const size_t rm = (size_t)room - fixed;
  bool last = false;
  int passes = 0;
  auto own = [&](const N* M, int ld, int rows) {           // blk <- the own columns of M
    for (int j = threadIdx.x >> 5; j < vi; j += blockDim.x >> 5)
      for (int k = threadIdx.x & 31; k < rows; k += 32) blk[(size_t)j * rows + k] = __ldcg(M + (size_t)(v0 + j) * ld + k);
  };
  auto correct = [&]() {                                   // V2(:, own) = V(:, own) + V E, in FP32
    rf_gemm<float>(n, vi, n, [&](int k, int i) { return rf_f(__ldcg(m.V + (size_t)k * m.ldv + i)); }, false, E, n, (float*)st,
                   rm, [&](int i, int j, float v) {
                     const size_t at = (size_t)(v0 + j) * m.ldv + i;
                     __stcg(m.V2 + at, rf_add(__ldcg(m.V + at), v));
                   });
  };
  auto swap = [&]() { N* t = m.V; m.V = m.V2; m.V2 = t; };
  for (int step = 0;; ++step) {
    // R(:, own) = I - V^T V(:, own); W(:, own) = X V(:, own) and its squared norms
    own(m.V, m.ldv, n);
    float dev = 0.f;
    if (!last)
      rf_gemm<N>(n, vi, n, [&](int k, int i) { return __ldcg(m.V + (size_t)i * m.ldv + k); }, true, blk, n, st, rm,
                 [&](int i, int j, N v) {
                   const float d = i == v0 + j ? -rf_f(rf_add(v, -1.f)) : -rf_f(v);
                   R[(size_t)j * n + i] = d;
                   dev = fmaxf(dev, fabsf(d));
                 });
    rf_gemm<N>(len, vi, n, [&](int k, int i) { return x(i, k); }, kfast, blk, n, st, rm,
               [&](int i, int j, N v) { __stcg(m.W + (size_t)(v0 + j) * m.ldw + i, rf_sum(v)); });
    own(m.W, m.ldw, len);                                  // written by this CTA, ordered by the barrier in rf_gemm
    __syncthreads();
    for (int j = threadIdx.x >> 5; j < vi; j += blockDim.x >> 5) {
      N a;
      rf_zero(a);
      for (int i = threadIdx.x & 31; i < len; i += 32) rf_mac(a, blk[(size_t)j * len + i], blk[(size_t)j * len + i]);
      a = rf_sum(a);
      for (int o = 16; o > 0; o >>= 1) a = rf_plus(a, rf_shfl(a, o));
      if ((threadIdx.x & 31) == 0) __stcg(m.nrm + v0 + j, a);
    }
    if (!cl_sync(cc)) return RF_DEAD;
    if (last) return RF_DONE;
    for (int i = threadIdx.x; i < n; i += blockDim.x) nr[i] = __ldcg(m.nrm + i);
    __syncthreads();
    float nmax = 0.f;
    for (int i = threadIdx.x & 31; i < n; i += 32) nmax = fmaxf(nmax, rf_f(nr[i]));
    for (int o = 16; o > 0; o >>= 1) nmax = fmaxf(nmax, __shfl_xor_sync(0xffffffffu, nmax, o));
    const float least = none * nmax, tmin2 = tmin * tmin * nmax;
    // S(:, own) = W^T W(:, own) -> the step's E
    float mr = 0.f, mt = 0.f, mx = 0.f;                    // pairs to rotate; ties and large angles; largest |E|
    bool tied = false, large = false;
    rf_gemm<N>(n, vi, len, [&](int k, int i) { return __ldcg(m.W + (size_t)i * m.ldw + k); }, true, blk, len, st, rm,
               [&](int i, int j, N s) {
                 const int c = v0 + j;
                 const float r = R[(size_t)j * n + i];
                 float e = 0.5f * r;
                 if (i != c) {
                   const float si = rf_f(nr[i]), sc = rf_f(nr[c]);
                   const float g = rf_f(rf_add(s, 0.5f * r * (si + sc)));
                   const float sb = fmaxf(si, sc), sm = fminf(si, sc);
                   if (sb > least && sm > 1e-34f) {
                     const float cs = g * rsqrtf(si) * rsqrtf(sc), c2 = cs * cs;
                     if (c2 > tol2) {
                       const float z = rf_diff(nr[c], nr[i]) / (2.f * g), az = fabsf(z);
                       const float t = copysignf(az > 1e15f ? 0.5f / az : 1.f / (az + sqrtf(fmaf(z, z, 1.f))), z);
                       if (own_scale ? fabsf(t) <= tmin : t * t * sb <= tmin2) {
                         // nothing: W's own rounding
                       } else if (fabsf(t) <= 0.1f) {
                         e += t;
                         mr = 1.f;
                       } else if (c2 <= 1e-10f) {
                         tied = true;
                       } else {
                         large = true;
                       }
                     }
                   }
                 }
                 mx = fmaxf(mx, fabsf(e));
                 E[(size_t)j * n + i] = e;
               });
    // a column of E whose sum is large would not be a small correction
    for (int j = threadIdx.x >> 5; j < vi; j += blockDim.x >> 5) {
      float a = 0.f;
      for (int i = threadIdx.x & 31; i < n; i += 32) a += fabsf(E[(size_t)j * n + i]);
      for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
      if (!(a <= 0.4f)) large = true;
    }
    mt = (tied ? 1.f : 0.f) + (large ? 2.f : 0.f);
    float s[4] = {rf_block_max(mr, s_red), rf_block_max(mt, s_red), rf_block_max(mx, s_red), rf_block_max(dev, s_red)};
    if (!rf_meet_max(cc, m, s)) return RF_DEAD;
    m.tied = s[1] == 1.f;
    bool only_r = !go_on;                                  // E = R / 2 only
    if (!only_r && s[1] >= 2.f) {
      if (passes >= RF_PASSES || step >= RF_STEPS) {
        only_r = true;                                     // V is handed on orthonormal
      } else if (s[3] > ready) {
        for (int idx = threadIdx.x; idx < n * vi; idx += blockDim.x) E[idx] = 0.5f * R[idx];
        correct();
        if (!cl_sync(cc)) return RF_DEAD;
        swap();
        continue;
      } else {
        ++passes;
        if (!jacobi()) {
          if (cc.dead) return RF_DEAD;
          only_r = true;
        } else {
          // V <- V J, J exact FP32 numbers
          for (int j = threadIdx.x >> 5; j < vi; j += blockDim.x >> 5)
            for (int k = threadIdx.x & 31; k < n; k += 32)
              blk[(size_t)j * n + k] = rf_make<N>(__ldcg(m.J + (size_t)(v0 + j) * m.ldj + k));
          rf_gemm<N>(n, vi, n, [&](int k, int i) { return __ldcg(m.V + (size_t)k * m.ldv + i); }, false, blk, n, st, rm,
                     [&](int i, int j, N v) { __stcg(m.V2 + (size_t)(v0 + j) * m.ldv + i, rf_sum(v)); });
          if (!cl_sync(cc)) return RF_DEAD;
          swap();
          continue;
        }
      }
    }
    if (!only_r && s[1] == 1.f && !ties) only_r = true;
    // orthogonal to the tolerance, and V's own error (of order R^2 after the step that
    // made it) is done with
    if (!only_r && s[0] == 0.f && s[3] <= fmaxf(small * small, 2e-15f)) return RF_DONE;
    if (step >= RF_STEPS) only_r = true;
    if (only_r)
      for (int idx = threadIdx.x; idx < n * vi; idx += blockDim.x) E[idx] = 0.5f * R[idx];
    correct();
    if (!cl_sync(cc)) return RF_DEAD;
    swap();
    // small enough: what is left after this step is of order E^2, W = X V once more
    const bool fine = (only_r ? s[3] : s[2]) <= small;
    // (|R| squares from step to step, from 0.1 at most: 1e-2, 1e-4, 1e-8, 1e-16)
    if (only_r && (fine || step >= RF_STEPS + 8)) return RF_SWEEPS;
    if (only_r) go_on = false;                             // until V is orthonormal
    else last = fine;
  }
}

// W = X V carries the rounding of the whole X in its small columns, so their cosines are
// not below ~1e-16 s_0 / s_j (FP64) whatever V is, while Jacobi rotations of W would keep them
// small.  Where the directions of W are the orthonormal result (X is C^T), the columns are
// made orthogonal: from every column go its parts along the larger ones (first order, the
// larger ones are left as they are), W <- W (I + F).  V takes the inverse,
// V <- V (I - F^T), so that W V^T, the product of the result, stays X: those parts are up to
// 1e-16 s_0 each, and all into the same few large directions (left in W alone they took FP64
// sums of 64^3 populations from 1e-14 to 4e-14 off in single cells).  V is then orthonormal to
// |F| ~ 1e-16 s_0 / s_i only, which its caller multiplies by s_i.  A round squares the sums of
// a column's cosines and triples them: from 0.1 five rounds end below 1e-16.  Where a sum is
// larger nothing is done.  (FP32 data: up to 1.  Such columns are below 1e-9 s_0, all of
// them rounding, and rarely kept: with 0.1 their sweeps took 10 of 169 ms of a step of 64^3
// waves.)  low: squared norms (relative to the largest) of columns that are
// all rounding; they are left out.  RF_DONE; RF_SWEEPS: the sweeps have to finish; or RF_DEAD.
template <typename N>
__device__ __noinline__ int rf_polish(ClusterCtx& cc, RefineMem<N>& m, int n, int len, float low, float tol2, int at,
                                       int room) {
  extern __shared__ __align__(16) unsigned char smem[];
  unsigned char* wa = smem + at;
  __shared__ float s_red[32];
  const int v0 = cc.rank * n / cc.P, vi = (cc.rank + 1) * n / cc.P - v0;
  const int big = imax(n, len), vmax = (n + cc.P - 1) / cc.P;
  N* blk = (N*)wa;
  N* nr = blk + (size_t)big * vmax;
  float* F = (float*)(nr + n);
  const size_t fixed = rf_fixed(n, len, cc.P);
  N* st = (N*)(wa + fixed);
  const size_t rm = (size_t)room - fixed;
  for (int i = threadIdx.x; i < n; i += blockDim.x) nr[i] = __ldcg(m.nrm + i);
  for (int j = threadIdx.x >> 5; j < vi; j += blockDim.x >> 5)
    for (int k = threadIdx.x & 31; k < len; k += 32) blk[(size_t)j * len + k] = __ldcg(m.W + (size_t)(v0 + j) * m.ldw + k);
  __syncthreads();
  float nmax = 0.f;
  for (int i = threadIdx.x & 31; i < n; i += 32) nmax = fmaxf(nmax, rf_f(nr[i]));
  for (int o = 16; o > 0; o >>= 1) nmax = fmaxf(nmax, __shfl_xor_sync(0xffffffffu, nmax, o));
  const float least = low * nmax;
  for (int it = 0;; ++it) {
    float mx = 0.f;
    rf_gemm<N>(n, vi, len, [&](int k, int i) { return __ldcg(m.W + (size_t)i * m.ldw + k); }, true, blk, len, st, rm,
               [&](int i, int j, N s) {
                 const int c = v0 + j;
                 const float si = rf_f(nr[i]), sc = rf_f(nr[c]), g = rf_f(s);
                 float f = 0.f;
                 if (i != c && si > least && sc > least) {
                   const float cs = g * rsqrtf(si) * rsqrtf(sc), c2 = cs * cs;
                   mx = fmaxf(mx, c2);
                   if (c2 > 0.25f * tol2 && (si > sc || (si == sc && i < c))) f = -g / si;
                 }
                 F[(size_t)j * n + i] = f;
                 __stcg(m.J + (size_t)c * m.ldj + i, f);
               });
    float sum = 0.f;                                       // of the cosines that F takes off a column
    for (int j = threadIdx.x >> 5; j < vi; j += blockDim.x >> 5) {
      float a = 0.f;
      for (int i = threadIdx.x & 31; i < n; i += 32) a += fabsf(F[(size_t)j * n + i]) * sqrtf(rf_f(nr[i]));
      for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
      sum = a > 0.f ? fmaxf(sum, a * rsqrtf(rf_f(nr[v0 + j]))) : sum;
    }
    float s[4] = {rf_block_max(mx, s_red), rf_block_max(sum, s_red), 0.f, 0.f};
    if (!rf_meet_max(cc, m, s)) return RF_DEAD;
    if (s[0] <= tol2) return RF_DONE;
    if (s[1] > (std::is_same<N, double>::value ? 0.1f : 1.f) || it == 6) return RF_SWEEPS;
    rf_gemm<float>(len, vi, n, [&](int k, int i) { return rf_f(__ldcg(m.W + (size_t)k * m.ldw + i)); }, false, F, n, (float*)st, rm,
                   [&](int i, int j, float v) { blk[(size_t)j * len + i] = rf_add(blk[(size_t)j * len + i], v); });
    // V2(:, own) = V(:, own) - V F^T(:, own)
    for (int k = threadIdx.x >> 5; k < n; k += blockDim.x >> 5)
      for (int j = threadIdx.x & 31; j < vi; j += 32) F[(size_t)j * n + k] = __ldcg(m.J + (size_t)k * m.ldj + v0 + j);
    rf_gemm<float>(n, vi, n, [&](int k, int i) { return rf_f(__ldcg(m.V + (size_t)k * m.ldv + i)); }, false, F, n, (float*)st, rm,
                   [&](int i, int j, float v) {
                     const size_t at = (size_t)(v0 + j) * m.ldv + i;
                     __stcg(m.V2 + at, rf_add(__ldcg(m.V + at), -v));
                   });
    if (!cl_sync(cc)) return RF_DEAD;                        // W, V and F have been read everywhere
    { N* t = m.V; m.V = m.V2; m.V2 = t; }
    for (int j = threadIdx.x >> 5; j < vi; j += blockDim.x >> 5)
      for (int k = threadIdx.x & 31; k < len; k += 32) __stcg(m.W + (size_t)(v0 + j) * m.ldw + k, blk[(size_t)j * len + k]);
    if (!cl_sync(cc)) return RF_DEAD;
  }
}

}  // namespace tn
