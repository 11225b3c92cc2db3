// FP32 one-sided Jacobi of up to 256 columns of up to 512 entries over the CTAs of a
// cluster, V along with W: the start of an FP64-accurate SVD that is too large for
// one CTA's registers (jacobi_reg.cuh).
//
// The columns form 2 U blocks of b <= 16 (U = min(P, 8) CTAs at work); in each of the
// 2 U - 1 rounds of a sweep a CTA holds two blocks, a column of each per warp, W and V in
// registers, and passes the second block's columns once round its warps through
// shared memory: b steps meet all cross pairs.  The first round of a sweep is an
// odd-even transposition of all 2 b columns, which meets the pairs inside the
// blocks too.  256 columns: 15 rounds of 16 steps (31 in the first), 256 steps
// where 255 is the least.  Blocks travel through L2 (64 KB per CTA and round) between
// cluster barriers.
//
// W and V are rotated as packed pairs of FP32 (fma.rn.f32x2: the same roundings, half
// the instructions).  A step is a chain of an inner product's shuffles, the
// angle, the rotation and the hand-over, ~600 cycles.
//
// Measured against one CTA's FP32 sweeps through shared memory and FP64 sweeps of the
// cluster: 256^3 sums of two at bond 128, mixed, two jobs on clusters of 16 (256 x 256 centre
// matrices): 1015 -> 142 ms; 128^3 at bond 100, nine jobs: 446 -> 86 ms; 64^3 at bond 80, FP64,
// two jobs: 196 -> 103 ms.
#pragma once

#include "cluster.cuh"
#include "jacobi_reg.cuh"

namespace tn {

// round-robin pair p of round rnd over np (even) indices, a < b
__device__ __forceinline__ void rr_pair(int rnd, int p, int np, int& a, int& b) {
  if (p == 0) { a = rnd; b = np - 1; }
  else { a = (rnd + p) % (np - 1); b = (rnd - p + (np - 1)) % (np - 1); }
  if (a > b) { const int t = a; a = b; b = t; }
}

static constexpr int JW_CTAS = 8, JW_COLS = 256, JW_LEN = 512, JW_SWEEPS = 16;

__host__ __device__ inline int jacobi_wide_ctas(int P) { return P < JW_CTAS ? P : JW_CTAS; }
__host__ __device__ inline int jacobi_wide_block(int ncol, int P) {
  const int u2 = 2 * jacobi_wide_ctas(P);
  return (ncol + u2 - 1) / u2;
}
__host__ __device__ inline bool jacobi_wide_fits(int ncol, int len, int P) {
  return P >= 2 && ncol <= JW_COLS && len <= JW_LEN && jacobi_wide_block(ncol, P) <= 16;
}
// Leading dimensions and columns (padded to whole blocks) of W and V.
__host__ __device__ inline int jacobi_wide_ldw(int len) { return len <= 256 ? 256 : 512; }
__host__ __device__ inline int jacobi_wide_cols(int ncol) { return ncol + 2 * JW_CTAS; }
// Floats that W and V take for column counts and lengths up to these.
__host__ __device__ inline size_t jacobi_wide_floats(int ncol, int len) {
  return (size_t)jacobi_wide_cols(imin(ncol, JW_COLS)) * (jacobi_wide_ldw(imin(len, JW_LEN)) + JW_COLS);
}

typedef unsigned long long jw2;          // two FP32 numbers
__device__ __forceinline__ jw2 jw_pack(float a, float b) {
  jw2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 jw_split(jw2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ jw2 jw_fma(jw2 a, jw2 b, jw2 c) {
  jw2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ jw2 jw_mul(jw2 a, jw2 b) {
  jw2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// One column of 64 H entries, 2 H of them a lane's.
template <int H>
__device__ __forceinline__ void jw_get(const float* p, jw2 (&x)[H], int lane) {
#pragma unroll
  for (int e = 0; e < H; e += 2) {
    const ulonglong2 v = *(const ulonglong2*)(p + e * 64 + 4 * lane);
    x[e] = v.x;
    x[e + 1] = v.y;
  }
}
template <int H>
__device__ __forceinline__ void jw_get_l2(const float* p, jw2 (&x)[H], int lane) {
#pragma unroll
  for (int e = 0; e < H; e += 2) {
    const float4 v = __ldcg((const float4*)(p + e * 64 + 4 * lane));
    x[e] = jw_pack(v.x, v.y);
    x[e + 1] = jw_pack(v.z, v.w);
  }
}
template <int H>
__device__ __forceinline__ void jw_put(float* p, const jw2 (&x)[H], int lane) {
#pragma unroll
  for (int e = 0; e < H; e += 2) *(ulonglong2*)(p + e * 64 + 4 * lane) = make_ulonglong2(x[e], x[e + 1]);
}
template <int H>
__device__ __forceinline__ void jw_put_l2(float* p, const jw2 (&x)[H], int lane) {
#pragma unroll
  for (int e = 0; e < H; e += 2) {
    const float2 a = jw_split(x[e]), b = jw_split(x[e + 1]);
    __stcg((float4*)(p + e * 64 + 4 * lane), make_float4(a.x, a.y, b.x, b.y));
  }
}
template <int H>
__device__ __forceinline__ float jw_dot(const jw2 (&x)[H], const jw2 (&y)[H]) {
  jw2 a = jw_mul(x[0], y[0]), b = jw_mul(x[1], y[1]);
#pragma unroll
  for (int e = 2; e < H; e += 2) {
    a = jw_fma(x[e], y[e], a);
    b = jw_fma(x[e + 1], y[e + 1], b);
  }
  const float2 p = jw_split(a), q = jw_split(b);
  float s = (p.x + p.y) + (q.x + q.y);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}
template <int H>
__device__ __forceinline__ void jw_rot(jw2 (&x)[H], jw2 (&y)[H], jw2 c, jw2 s, jw2 ms) {
#pragma unroll
  for (int e = 0; e < H; ++e) {
    const jw2 u = jw_fma(c, x[e], jw_mul(ms, y[e]));
    y[e] = jw_fma(c, y[e], jw_mul(s, x[e]));
    x[e] = u;
  }
}

// Sweeps on W (column j at Wg + j * 64 HW, zero beyond the column count and length) with
// V (Vg + j * JW_COLS) taking the same rotations, both in global memory, written by the
// cluster before (and ordered by a cluster barrier).  At most maxsw sweeps; returns those that
// rotated anything (maxsw if the last one still did, or this CTA has given up).  sm:
// shared memory of jacobi_wide_smem bytes.  All threads of every CTA.
static constexpr size_t jacobi_wide_smem(int ld) { return (size_t)2 * 16 * (ld + JW_COLS + 4) * 4; }

template <int HW>
__device__ __noinline__ int jacobi_wide_run(ClusterCtx& cc_, float* Wg, float* Vg, int ncol, int len, int maxsw, float* sm) {
  constexpr int HV = JW_COLS / 64, LW = 64 * HW, SLOT = LW + JW_COLS + 4;
  __builtin_assume(__isShared(sm));
  ClusterCtx cc = cc_;                                         // in registers
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int U = jacobi_wide_ctas(cc.P), nblk = 2 * U, b = jacobi_wide_block(ncol, cc.P);
  const bool work = cc.rank < U && wid < b;
  const float tol = 4.f * Eps<float>::v * sqrtf((float)len);
  __shared__ int s_any;
  auto slot = [&](int buf, int w) -> float* { return sm + (size_t)(buf * 16 + w) * SLOT; };
  auto meet = [&]() { asm volatile("bar.sync 1, %0;" ::"r"(b * 32) : "memory"); };
  jw2 xw[HW], yw[HW], xv[HV], yv[HV];
  float al = 0.f, be = 0.f;
  bool rot = false;
  auto rotate = [&]() {
    const float ga = jw_dot<HW>(xw, yw);
    float c, s;
    if (!jr_angle(al, be, ga, tol, c, s)) return;              // the same in every lane
    rot = true;
    const jw2 cp = jw_pack(c, c), sp = jw_pack(s, s), mp = jw_pack(-s, -s);
    jw_rot<HW>(xw, yw, cp, sp, mp);
    jw_rot<HV>(xv, yv, cp, sp, mp);
  };
  auto send = [&](float* p, const jw2 (&w)[HW], const jw2 (&v)[HV], float n) {
    jw_put<HW>(p, w, lane);
    jw_put<HV>(p + LW, v, lane);
    if (lane == 0) p[LW + JW_COLS] = n;
  };
  auto take = [&](const float* p, jw2 (&w)[HW], jw2 (&v)[HV], float& n) {
    jw_get<HW>(p, w, lane);
    jw_get<HV>(p + LW, v, lane);
    n = p[LW + JW_COLS];
  };
  int sweep = 0;
  for (; sweep < maxsw; ++sweep) {
    rot = false;
    for (int rnd = 0; rnd < nblk - 1; ++rnd) {
      if (work && !cc.dead) {
        int A, B;
        rr_pair(rnd, cc.rank, nblk, A, B);
        int ca = A * b + wid, cb = B * b + wid;
        jw_get_l2<HW>(Wg + (size_t)ca * LW, xw, lane);
        jw_get_l2<HV>(Vg + (size_t)ca * JW_COLS, xv, lane);
        jw_get_l2<HW>(Wg + (size_t)cb * LW, yw, lane);
        jw_get_l2<HV>(Vg + (size_t)cb * JW_COLS, yv, lane);
        al = jw_dot<HW>(xw, xw);
        be = jw_dot<HW>(yw, yw);
        if (rnd == 0) {
          // all pairs of the two blocks (the order of jacobi_reg_run with B = 1)
          for (int ph = 0; ph < b; ++ph) {
            rotate();
            send(slot(0, wid == 0 ? b - 1 : wid - 1), yw, yv, be);
            meet();
            take(slot(0, wid), yw, yv, be);
            if (wid + 1 < b) {
              rotate();
              send(slot(1, wid + 1), xw, xv, al);
            } else {
              send(slot(1, 0), yw, yv, be);
#pragma unroll
              for (int e = 0; e < HW; ++e) yw[e] = xw[e];
#pragma unroll
              for (int e = 0; e < HV; ++e) yv[e] = xv[e];
              be = al;
            }
            meet();
            take(slot(1, wid), xw, xv, al);
          }
          // reversed: X is the column that began as Y of warp b - 1 - wid
          ca = B * b + (b - 1 - wid);
          cb = A * b + (b - 1 - wid);
        } else {
          for (int s = 0; s < b; ++s) {
            rotate();
            if (b == 1) break;
            send(slot(s & 1, wid + 1 == b ? 0 : wid + 1), yw, yv, be);
            meet();
            take(slot(s & 1, wid), yw, yv, be);
          }
        }
        jw_put_l2<HW>(Wg + (size_t)ca * LW, xw, lane);
        jw_put_l2<HV>(Vg + (size_t)ca * JW_COLS, xv, lane);
        jw_put_l2<HW>(Wg + (size_t)cb * LW, yw, lane);
        jw_put_l2<HV>(Vg + (size_t)cb * JW_COLS, yv, lane);
      }
      if (rnd == nblk - 2) {
        // this CTA's flag into every CTA's slot (double buffered by sweep)
        const int any = __syncthreads_or(work && rot);
        if (cl_alive(cc) && threadIdx.x < (unsigned)cc.P) cl_store_remote(&cc.sh->flags[sweep & 1][cc.rank], threadIdx.x, any);
      }
      if (!cl_sync(cc)) {
        cc_ = cc;
        return maxsw;
      }
    }
    if (threadIdx.x < 32) {
      const int f = threadIdx.x < (unsigned)cc.P ? ((volatile int*)cc.sh->flags[sweep & 1])[threadIdx.x] : 0;
      const int any = __any_sync(0xffffffffu, f);
      if (threadIdx.x == 0) s_any = any;
    }
    __syncthreads();
    const int any = s_any;
    __syncthreads();
    if (!any) break;
  }
  cc_ = cc;
  return sweep;
}

__device__ __forceinline__ int jacobi_wide(ClusterCtx& cc, float* Wg, float* Vg, int ncol, int len, int maxsw, float* sm) {
  return len <= 256 ? jacobi_wide_run<4>(cc, Wg, Vg, ncol, len, maxsw, sm)
                    : jacobi_wide_run<8>(cc, Wg, Vg, ncol, len, maxsw, sm);
}

}  // namespace tn
