// FP32 one-sided Jacobi with the columns held in registers.
//
// jacobi_cols_h4 reads and writes both columns of every pair (and of V) through
// shared memory in every round, which bounds it by the shared-memory port: 256 KB
// per round of 64 pairs of 128 entries, ~2050 of its ~2800 cycles.  Here a warp
// keeps 2 B columns (two blocks of B) in its registers, rotates the B x B pairs
// of the two blocks in B steps without leaving them, and then passes one block on
// to its neighbour through shared memory: 1 / (2 B) of that traffic and one
// block barrier per B rounds.
//
// Order of the pairs: odd-even transposition of the 2 W blocks of W warps.  In an
// even phase warp w holds positions (2 w, 2 w + 1), in an odd phase
// (2 w + 1, 2 w + 2); the two blocks of a warp trade places after they met, so in
// 2 W phases every two blocks meet exactly once (the order of the blocks ends
// reversed, which the caller does not see: columns are not ordered).  The
// pairs inside a block are rotated at the start of a sweep.
//
// Measured (128^3 sums of two at bond 64, 9 jobs, 128 x 128 centre matrices):
// the rounding 67.5 -> 34.7 ms; 3.4 M -> 0.9 M cycles per SVD of a 64^3 step at
// bond 64.  ~140 instructions per warp and step of 64 pairs, of which 64 are the
// rotation's arithmetic; four warps a scheduler do not hide the chain of a step (inner
// products, shuffles, angle): over the whole FP32 rounding 44 % of the issue slots of a busy SM
// are used, an issue waits 2.3 times on barriers, 1.8 on shuffles and shared memory and
// 1.7 on fixed latencies (ncu).
#pragma once

#include "linalg.cuh"

namespace tn {

// Totals over the warp of v[0..B): lane group q = lane / (32 / B) gets that of v[q].
template <int B>
__device__ __forceinline__ float jr_reduce(float (&v)[B], int lane) {
  constexpr unsigned F = 0xffffffffu;
  float r;
  if constexpr (B == 4) {
    const bool h = lane & 16;
    const float s0 = h ? v[0] : v[2], s1 = h ? v[1] : v[3];
    const float k0 = (h ? v[2] : v[0]) + __shfl_xor_sync(F, s0, 16);
    const float k1 = (h ? v[3] : v[1]) + __shfl_xor_sync(F, s1, 16);
    const bool g = lane & 8;
    r = (g ? k1 : k0) + __shfl_xor_sync(F, g ? k0 : k1, 8);
  } else if constexpr (B == 2) {
    const bool h = lane & 16;
    r = (h ? v[1] : v[0]) + __shfl_xor_sync(F, h ? v[0] : v[1], 16);
    r += __shfl_xor_sync(F, r, 8);
  } else {
    r = v[0] + __shfl_xor_sync(F, v[0], 16);
    r += __shfl_xor_sync(F, r, 8);
  }
  r += __shfl_xor_sync(F, r, 4);
  r += __shfl_xor_sync(F, r, 2);
  r += __shfl_xor_sync(F, r, 1);
  return r;
}

// Rutishauser's rotation zeroing the inner product ga of columns with squared
// norms al, be (c = 1, s = 0 if they count as orthogonal: |ga| <= tol sqrt(al)
// sqrt(be), or one carries nothing).  al, be are updated to the rotated norms.
// MUFU reciprocal and square root (2 ulp): the rotation is off orthogonal by
// ~2e-7, which scales a column of W by that much and turns it not at all; the
// caller takes directions, not lengths, from W where it needs more.
__device__ __forceinline__ bool jr_angle(float& al, float& be, float ga, float tol, float& c, float& s) {
  c = 1.f;
  s = 0.f;
  // the FP32 floor of jacobi_cols_hw: below it zeta could overflow
  if (!(al >= 1e-24f) || !(be >= 1e-24f) || !(fabsf(ga) * (rsqrtf(al) * rsqrtf(be)) > tol)) return false;
  const float z = __fdividef(be - al, 2.f * ga), az = fabsf(z);
  const float q = fmaf(z, z, 1.f);
  const float t = copysignf(az > 1e15f ? __fdividef(0.5f, az) : __fdividef(1.f, az + q * rsqrtf(q)), z);
  c = rsqrtf(fmaf(t, t, 1.f));
  s = c * t;
  al -= t * ga;
  be += t * ga;
  return true;
}

// One step: the pairs (X[i], Y[(i + S) % B]) of two blocks, their squared norms
// na (of X[q]) and nb (of Y[q]) kept by lane group q.
// LOG: lane group q puts the pair's (c, s) at its log.
template <int B, int EPL, int S, bool LOG>
__device__ __forceinline__ bool jr_cross(float (&X)[B][EPL], float (&Y)[B][EPL], float& na, float& nb, float tol,
                                         int lane, float2* log) {
  constexpr unsigned F = 0xffffffffu;
  constexpr int G = 32 / B;
  float d[B];
#pragma unroll
  for (int i = 0; i < B; ++i) {
    float a = 0.f;
#pragma unroll
    for (int e = 0; e < EPL; ++e) a = fmaf(X[i][e], Y[(i + S) % B][e], a);
    d[i] = a;
  }
  const float ga = jr_reduce<B>(d, lane);
  float be = S == 0 ? nb : __shfl_sync(F, nb, (lane + S * G) & 31);
  float c, s;
  const bool go = jr_angle(na, be, ga, tol, c, s);
  if (LOG && lane % G == 0) *log = make_float2(c, s);
  if (!__any_sync(F, go)) return false;
  nb = S == 0 ? be : __shfl_sync(F, be, (lane + 32 - S * G) & 31);
#pragma unroll
  for (int i = 0; i < B; ++i) {
    const float ci = B == 1 ? c : __shfl_sync(F, c, i * G), si = B == 1 ? s : __shfl_sync(F, s, i * G);
#pragma unroll
    for (int e = 0; e < EPL; ++e) {
      const float x = X[i][e], y = Y[(i + S) % B][e];
      X[i][e] = ci * x - si * y;
      Y[(i + S) % B][e] = si * x + ci * y;
    }
  }
  return true;
}

// The pairs inside the two blocks, (X[i0], X[i1]), (X[i2], X[i3]) and the same of
// Y (B = 4), or (X[0], X[1]) and (Y[0], Y[1]) (B = 2).
template <int B, int EPL, int I0, int I1, int I2, int I3, bool LOG>
__device__ __forceinline__ bool jr_inner(float (&X)[B][EPL], float (&Y)[B][EPL], float tol, int lane, float2* log) {
  constexpr unsigned F = 0xffffffffu;
  constexpr int G = 32 / B, H = B / 2;
  float d[B], na[B], nb[B];
#pragma unroll
  for (int q = 0; q < B; ++q) {
    const int i = (q % H) == 0 ? I0 : I2, j = (q % H) == 0 ? I1 : I3;
    float a = 0.f, x2 = 0.f, y2 = 0.f;
#pragma unroll
    for (int e = 0; e < EPL; ++e) {
      const float x = q < H ? X[i][e] : Y[i][e], y = q < H ? X[j][e] : Y[j][e];
      a = fmaf(x, y, a);
      x2 = fmaf(x, x, x2);
      y2 = fmaf(y, y, y2);
    }
    d[q] = a;
    na[q] = x2;
    nb[q] = y2;
  }
  const float ga = jr_reduce<B>(d, lane);
  float al = jr_reduce<B>(na, lane), be = jr_reduce<B>(nb, lane), c, s;
  const bool go = jr_angle(al, be, ga, tol, c, s);
  if (LOG && lane % G == 0) *log = make_float2(c, s);
  if (!__any_sync(F, go)) return false;
#pragma unroll
  for (int q = 0; q < B; ++q) {
    const int i = (q % H) == 0 ? I0 : I2, j = (q % H) == 0 ? I1 : I3;
    const float ci = __shfl_sync(F, c, q * G), si = __shfl_sync(F, s, q * G);
#pragma unroll
    for (int e = 0; e < EPL; ++e) {
      const float x = q < H ? X[i][e] : Y[i][e], y = q < H ? X[j][e] : Y[j][e];
      const float u = ci * x - si * y, w = si * x + ci * y;
      if (q < H) { X[i][e] = u; X[j][e] = w; }
      else { Y[i][e] = u; Y[j][e] = w; }
    }
  }
  return true;
}

// A block of B columns in shared memory: EPL consecutive entries of a column per lane.
template <int B, int EPL>
__device__ __forceinline__ void jr_store(float* p, const float (&X)[B][EPL], int lane) {
#pragma unroll
  for (int i = 0; i < B; ++i)
#pragma unroll
    for (int e = 0; e < EPL; e += 4) {
      if constexpr (EPL % 4 == 0)
        *(float4*)(p + (size_t)i * 32 * EPL + e * 32 + 4 * lane) = make_float4(X[i][e], X[i][e + 1], X[i][e + 2], X[i][e + 3]);
      else if constexpr (EPL == 2)
        *(float2*)(p + (size_t)i * 64 + 2 * lane) = make_float2(X[i][0], X[i][1]);
      else
        p[(size_t)i * 32 + lane] = X[i][0];
    }
}
template <int B, int EPL>
__device__ __forceinline__ void jr_load(const float* p, float (&X)[B][EPL], int lane) {
#pragma unroll
  for (int i = 0; i < B; ++i)
#pragma unroll
    for (int e = 0; e < EPL; e += 4) {
      if constexpr (EPL % 4 == 0) {
        const float4 v = *(const float4*)(p + (size_t)i * 32 * EPL + e * 32 + 4 * lane);
        X[i][e] = v.x; X[i][e + 1] = v.y; X[i][e + 2] = v.z; X[i][e + 3] = v.w;
      } else if constexpr (EPL == 2) {
        const float2 v = *(const float2*)(p + (size_t)i * 64 + 2 * lane);
        X[i][0] = v.x; X[i][1] = v.y;
      } else {
        X[i][0] = p[(size_t)i * 32 + lane];
      }
    }
}

// Sweeps on the columns W[j * 32 EPL + i] (shared memory; zero beyond the column
// count and length, columns padded to a multiple of 2 B), at most maxsw.  Returns
// the sweeps that rotated anything (maxsw if the last one still did).  W is the
// exchange buffer meanwhile: 2 W blocks are one block out and one block in per
// warp, so a sending phase alternates between its halves.  A sweep reverses the
// blocks; they are stored back in their first order.
// log (LOG) receives the (c, s) of every pair of every sweep,
// log[((sweep * jr_steps + step) * B + q) * nw + w] for pair q of warp w, which
// jacobi_reg_apply reads.
template <int B>
__host__ __device__ constexpr int jr_steps(int nw) { return B - 1 + 2 * nw * B; }

template <int B, int EPL, bool LOG>
__device__ __noinline__ int jacobi_reg_run(float* W, int ncol, int len, int maxsw, float2* log) {
  __builtin_assume(__isShared(W));
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nw = (ncol + 2 * B - 1) / (2 * B);              // warps that hold columns
  constexpr int BS = B * 32 * EPL;                          // floats of a block
  // a few ulps above the round-off of a fresh pair; as a start for a refinement
  // (LOG), which wants small cosines, closer to it
  const float tol = (LOG ? 4.f : 16.f) * Eps<float>::v * sqrtf((float)len);
  __shared__ int s_rot[2];
  if (threadIdx.x < 2) s_rot[threadIdx.x] = 0;
  __syncthreads();
  int sweep = 0;
  if (wid < nw) {
    float X[B][EPL], Y[B][EPL];
    jr_load<B, EPL>(W + (size_t)(2 * wid) * BS, X, lane);
    jr_load<B, EPL>(W + (size_t)(2 * wid + 1) * BS, Y, lane);
    float* buf[2] = {W, W + (size_t)nw * BS};
    auto meet = [&]() { asm volatile("bar.sync 1, %0;" ::"r"(nw * 32) : "memory"); };
    const int lstep = B * nw;
    float2* lg = log + (LOG ? (size_t)(lane / (32 / B)) * nw + wid : 0);
    auto next = [&]() { if (LOG) lg += lstep; };
    // all cross pairs of the two blocks, with norms taken afresh
    auto cross = [&]() -> bool {
      float na[B], nb[B];
#pragma unroll
      for (int i = 0; i < B; ++i) {
        float a = 0.f, b = 0.f;
#pragma unroll
        for (int e = 0; e < EPL; ++e) {
          a = fmaf(X[i][e], X[i][e], a);
          b = fmaf(Y[i][e], Y[i][e], b);
        }
        na[i] = a;
        nb[i] = b;
      }
      float al = jr_reduce<B>(na, lane), be = jr_reduce<B>(nb, lane);
      bool r = jr_cross<B, EPL, 0, LOG>(X, Y, al, be, tol, lane, lg);
      next();
      if constexpr (B >= 2) {
        r |= jr_cross<B, EPL, 1, LOG>(X, Y, al, be, tol, lane, lg);
        next();
      }
      if constexpr (B == 4) {
        r |= jr_cross<B, EPL, 2, LOG>(X, Y, al, be, tol, lane, lg);
        next();
        r |= jr_cross<B, EPL, 3, LOG>(X, Y, al, be, tol, lane, lg);
        next();
      }
      return r;
    };
    meet();
    for (; sweep < maxsw; ++sweep) {
      bool rot = false;
      if constexpr (B == 4) {
        rot |= jr_inner<B, EPL, 0, 1, 2, 3, LOG>(X, Y, tol, lane, lg);
        next();
        rot |= jr_inner<B, EPL, 0, 2, 1, 3, LOG>(X, Y, tol, lane, lg);
        next();
        rot |= jr_inner<B, EPL, 0, 3, 1, 2, LOG>(X, Y, tol, lane, lg);
        next();
      } else if constexpr (B == 2) {
        rot |= jr_inner<B, EPL, 0, 1, 0, 1, LOG>(X, Y, tol, lane, lg);
        next();
      }
      for (int ph = 0; ph < nw; ++ph) {
        // even phase; the blocks trade places: Y (now first) goes to the left
        // neighbour's right hand (warp 0's parks with the last warp)
        rot |= cross();
        jr_store<B, EPL>(buf[0] + (size_t)(wid == 0 ? nw - 1 : wid - 1) * BS, Y, lane);
        meet();
        jr_load<B, EPL>(buf[0] + (size_t)wid * BS, Y, lane);
        // odd phase: the last warp holds the two ends, which do not meet; its X
        // stays the last position, so it leaves as the others' Y stays
        if (wid + 1 < nw) {
          rot |= cross();
          jr_store<B, EPL>(buf[1] + (size_t)(wid + 1) * BS, X, lane);
        } else {
          if (LOG) lg += B * lstep;                          // no pairs here: the log has a gap
          jr_store<B, EPL>(buf[1], Y, lane);
#pragma unroll
          for (int i = 0; i < B; ++i)
#pragma unroll
            for (int e = 0; e < EPL; ++e) Y[i][e] = X[i][e];
        }
        meet();
        jr_load<B, EPL>(buf[1] + (size_t)wid * BS, X, lane);
      }
      if (rot && lane == 0) s_rot[sweep & 1] = 1;
      meet();
      const int any = s_rot[sweep & 1];
      if (threadIdx.x == 0) s_rot[(sweep + 1) & 1] = 0;     // read two meetings ago
      meet();
      if (!any) break;
    }
    const int done = sweep < maxsw ? sweep + 1 : sweep;     // the last one rotated nothing
    const int px = done & 1 ? 2 * nw - 1 - 2 * wid : 2 * wid, py = done & 1 ? px - 1 : px + 1;
    jr_store<B, EPL>(W + (size_t)px * BS, X, lane);
    jr_store<B, EPL>(W + (size_t)py * BS, Y, lane);
  }
  __shared__ int s_sweeps;
  if (threadIdx.x == 0) s_sweeps = sweep;
  __syncthreads();
  sweep = s_sweeps;
  __syncthreads();
  return sweep;
}

// Shapes that jacobi_reg takes with 512 threads: 16 warps of 8 columns, eight
// entries per lane (2 x 4 x 8 = 64 registers of data).
__host__ __device__ inline bool jacobi_reg_fits(int ncol, int len) { return ncol <= 128 && len <= 256; }
// Leading dimension of W, and its columns (padded to whole warps of blocks).
__host__ __device__ inline int jacobi_reg_ld(int len) { return len <= 32 ? 32 : len <= 64 ? 64 : len <= 128 ? 128 : 256; }
__host__ __device__ inline int jacobi_reg_block(int ncol) { return ncol <= 32 ? 1 : ncol <= 64 ? 2 : 4; }
__host__ __device__ inline int jacobi_reg_cols(int ncol) {
  const int b2 = 2 * jacobi_reg_block(ncol);
  return (ncol + b2 - 1) / b2 * b2;
}

// One-sided FP32 Jacobi of the padded columns in W (see jacobi_reg_run).  Blocks
// of 4 columns when more than 64 are there, of 2 or 1 below so that all 16 warps
// have columns.
template <bool LOG>
__device__ __forceinline__ int jacobi_reg(float* W, int ncol, int len, int maxsw, float2* log) {
  const int b = jacobi_reg_block(ncol);
#define JR(B, LOG)                                                              \
  (len <= 32    ? jacobi_reg_run<B, 1, LOG>(W, ncol, len, maxsw, log)           \
   : len <= 64  ? jacobi_reg_run<B, 2, LOG>(W, ncol, len, maxsw, log)           \
   : len <= 128 ? jacobi_reg_run<B, 4, LOG>(W, ncol, len, maxsw, log)           \
                : jacobi_reg_run<B, 8, LOG>(W, ncol, len, maxsw, log))
  return b == 1 ? JR(1, LOG) : b == 2 ? JR(2, LOG) : JR(4, LOG);
#undef JR
}

// Pairs of a sweep's log, and the sweeps that are logged at most (the ones that
// an FP32 Jacobi needs are about ten; what is left at the limit is the FP64
// sweeps' work).
static constexpr int JR_LOG_SWEEPS = 16;
__host__ __device__ inline size_t jacobi_reg_log_sweep(int ncol) {
  const int b = jacobi_reg_block(ncol), nw = (ncol + 2 * b - 1) / (2 * b);
  return (size_t)(b - 1 + 2 * nw * b) * b * nw;
}

// Rows [r0, r0 + nr) of the product J of the logged rotations (J = I before), as
// entries of its columns: out[c * ld + r] for c, r < ncol.  Rows of J are
// independent, so the CTAs of a cluster share them.  A half-warp holds a row: its
// lane w the columns that warp w of jacobi_reg_run held, and passes them on to its
// neighbours as that warp did.  A sweep of the log is staged in shared memory (st,
// two sweeps long) while the one before is applied.  ~40 cycles a step, the latency
// of its dependent rotations.
template <typename O> __device__ __forceinline__ O jr_out(float v) { return (O)v; }
template <> __device__ __forceinline__ float2 jr_out<float2>(float v) { return make_float2(v, 0.f); }   // v as a pair

template <int B, typename O>
__device__ __noinline__ void jacobi_reg_apply_run(const float2* log, int sweeps, int ncol, int r0, int nr, O* out,
                                                  int ld, float2* st) {
  __builtin_assume(__isShared(st));
  constexpr unsigned F = 0xffffffffu;
  const int nw = (ncol + 2 * B - 1) / (2 * B), per = B * nw, size = jr_steps<B>(nw) * per;
  const int w = threadIdx.x & 15, hw = threadIdx.x >> 4, nhw = blockDim.x >> 4;
  const int lane = threadIdx.x & 31, half = lane & 16;
  const int wl = imin(w, nw - 1);
  const int left = half | (w == 0 ? nw - 1 : w - 1), right = half | (w == nw - 1 ? 0 : imin(w + 1, 15));
  const bool last = w + 1 >= nw;
  auto stage = [&](int sw) {
    const float2* lg = log + (size_t)sw * size;
    float2* d = st + (size_t)(sw & 1) * size;
    // 16 bytes (`size` is even) past L1, which may hold an earlier site's log
    for (int i = 2 * threadIdx.x; i < size; i += 2 * blockDim.x)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(d + i)), "l"(lg + i)
                   : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  auto rot = [](float& x, float& y, float2 g) {
    const float u = g.x * x - g.y * y, v = g.y * x + g.x * y;
    x = u;
    y = v;
  };
  for (int base = r0; base < r0 + nr; base += nhw) {
    const int row = base + hw;
    float X[B], Y[B];
#pragma unroll
    for (int i = 0; i < B; ++i) {
      X[i] = (2 * w) * B + i == row ? 1.f : 0.f;
      Y[i] = (2 * w + 1) * B + i == row ? 1.f : 0.f;
    }
    if (sweeps > 0) stage(0);
    for (int sw = 0; sw < sweeps; ++sw) {
      if (sw + 1 < sweeps) {
        stage(sw + 1);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
      } else {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
      }
      __syncthreads();
      if ((hw & ~1) + base < r0 + nr) {                      // the warp holds a row
        const float2* p = st + (size_t)(sw & 1) * size + wl;
        float2 g[B];
        auto get = [&]() {
#pragma unroll
          for (int q = 0; q < B; ++q) g[q] = p[q * nw];
          p += per;
        };
        if constexpr (B == 4) {
          get(); rot(X[0], X[1], g[0]); rot(X[2], X[3], g[1]); rot(Y[0], Y[1], g[2]); rot(Y[2], Y[3], g[3]);
          get(); rot(X[0], X[2], g[0]); rot(X[1], X[3], g[1]); rot(Y[0], Y[2], g[2]); rot(Y[1], Y[3], g[3]);
          get(); rot(X[0], X[3], g[0]); rot(X[1], X[2], g[1]); rot(Y[0], Y[3], g[2]); rot(Y[1], Y[2], g[3]);
        } else if constexpr (B == 2) {
          get(); rot(X[0], X[1], g[0]); rot(Y[0], Y[1], g[1]);
        }
        float2 e[B][B], o[B][B];                             // the phase's pairs, loaded ahead
        auto fetch = [&](float2 (&f)[B][B]) {
#pragma unroll
          for (int S = 0; S < B; ++S)
#pragma unroll
            for (int q = 0; q < B; ++q) f[S][q] = p[(S * B + q) * nw];
          p += B * per;
        };
        fetch(e);
        for (int ph = 0; ph < nw; ++ph) {
          fetch(o);
#pragma unroll
          for (int S = 0; S < B; ++S)
#pragma unroll
            for (int i = 0; i < B; ++i) rot(X[i], Y[(i + S) % B], e[S][i]);
#pragma unroll
          for (int i = 0; i < B; ++i) Y[i] = __shfl_sync(F, Y[i], right);
          if (ph + 1 < nw) fetch(e);
#pragma unroll
          for (int S = 0; S < B; ++S)
#pragma unroll
            for (int i = 0; i < B; ++i) rot(X[i], Y[(i + S) % B], last ? make_float2(1.f, 0.f) : o[S][i]);
#pragma unroll
          for (int i = 0; i < B; ++i) {
            // the last lane's X is the last position and stays as Y; its Y is the first
            const float give = last ? Y[i] : X[i], stay = last ? X[i] : Y[i];
            X[i] = __shfl_sync(F, give, left);
            Y[i] = stay;
          }
        }
      }
      __syncthreads();                                       // st is refilled two sweeps on
    }
    if (row < r0 + nr && w < nw) {
      const int px = sweeps & 1 ? 2 * nw - 1 - 2 * w : 2 * w, py = sweeps & 1 ? px - 1 : px + 1;
#pragma unroll
      for (int i = 0; i < B; ++i) {
        if (px * B + i < ncol) __stcg(out + (size_t)(px * B + i) * ld + row, jr_out<O>(X[i]));
        if (py * B + i < ncol) __stcg(out + (size_t)(py * B + i) * ld + row, jr_out<O>(Y[i]));
      }
    }
  }
  __syncthreads();
}

// st: shared memory of 2 jacobi_reg_log_sweep(ncol) pairs.
template <typename O>
__device__ __forceinline__ void jacobi_reg_apply(const float2* log, int sweeps, int ncol, int r0, int nr, O* out,
                                                 int ld, float2* st) {
  const int b = jacobi_reg_block(ncol);
  if (b == 1) jacobi_reg_apply_run<1, O>(log, sweeps, ncol, r0, nr, out, ld, st);
  else if (b == 2) jacobi_reg_apply_run<2, O>(log, sweeps, ncol, r0, nr, out, ld, st);
  else jacobi_reg_apply_run<4, O>(log, sweeps, ncol, r0, nr, out, ld, st);
}

}  // namespace tn
