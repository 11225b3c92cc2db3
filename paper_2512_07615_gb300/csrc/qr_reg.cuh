// FP32 blocked Householder QR with the panels in registers.
//
// householder_qr_blk walks a panel column by column through shared memory with
// four to five block barriers a column, and its trailing products load eight
// operands for sixteen multiply-adds.  Here a thread holds one row (two above 512
// rows) of the 16-column panel in registers, and one reduction per column gives
// everything the column needs at once: its norm, its products with the columns
// still to come (the update) and with the reflectors already there (the T
// factor), so a column costs one block barrier.  The trailing update runs a
// thread per column and row group: a row of V is read as four broadcast 16-byte
// loads for sixteen multiply-adds, and T is folded into V (V T^T or V T) instead of
// being applied to the product.
#pragma once

#include "linalg.cuh"

namespace tn {

static constexpr int QRT = 512;          // threads of the CTAs that call qr_reg

// Totals over the warp of v[0..16): lanes 2 q and 2 q + 1 get that of v[q].
__device__ __forceinline__ float qr_reduce16(float (&v)[16], int lane) {
  constexpr unsigned F = 0xffffffffu;
#pragma unroll
  for (int o = 16, n = 8; n >= 1; o >>= 1, n >>= 1) {
    const bool h = lane & o;
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (i < n) {
        const float keep = h ? v[i + n] : v[i], give = h ? v[i] : v[i + n];
        v[i] = keep + __shfl_xor_sync(F, give, o);
      }
  }
  return v[0] + __shfl_xor_sync(F, v[0], 1);
}

// Shared scratch of a call: V (rows of the panel), then the partial products.
__host__ __device__ inline size_t qr_reg_vbytes(int m) { return (size_t)m * 16 * sizeof(float); }
// (the most that G - 1 partial sums of ncw column groups take: G ncw <= 16)
static constexpr size_t QR_PART_BYTES = (size_t)15 * 32 * 16 * sizeof(float);
__host__ __device__ inline size_t qr_reg_bytes(int m) { return qr_reg_vbytes(m) + QR_PART_BYTES; }

// X (mr x nx, ld) <- X - VT (V^T X) for the panel V (mr x 16, shared memory),
// where VT = V T (or V T^T) replaces V in place once V^T X is formed.  The column
// groups are 32 wide; the 16 warps share the rows of each in G groups whose
// partial sums are added in group order.
__device__ __forceinline__ void qr_reg_update(float* V, int mr, float* X, int ld, int nx, const float (*sT)[17],
                                              bool transposed, float* part) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  auto fold_t = [&]() {                  // V <- V T^T (transposed) or V T, row by row
    for (int r = threadIdx.x; r < mr; r += QRT) {
      float v[16], o[16];
      float4* p = (float4*)(V + (size_t)r * 16);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 x = p[i];
        v[4 * i] = x.x; v[4 * i + 1] = x.y; v[4 * i + 2] = x.z; v[4 * i + 3] = x.w;
      }
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        float a = 0.f;
        if (transposed) {
#pragma unroll
          for (int k = q; k < 16; ++k) a = fmaf(v[k], sT[q][k], a);
        } else {
#pragma unroll
          for (int k = 0; k <= q; ++k) a = fmaf(v[k], sT[k][q], a);
        }
        o[q] = a;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) p[i] = make_float4(o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
    }
  };
  // all columns in one go up to 512 of them (16 warps of 32); V is replaced by
  // V T only when the products of every column are there, so wider matrices
  // form the products of all their chunks first
  const int ncw = imin((nx + 31) / 32, 16), G = 16 / ncw;
  const int cw = wid % ncw, g = wid / ncw, rc = (mr + G - 1) / G;
  const int r0 = imin(mr, g * rc), r1 = imin(mr, r0 + rc);
  const int pld = ncw * 32;
  const int c = cw * 32 + lane;
  const bool act = g < G && c < nx;
  float a[16];
#pragma unroll
  for (int q = 0; q < 16; ++q) a[q] = 0.f;
  if (act) {
    const float* x = X + c;
#pragma unroll 4
    for (int r = r0; r < r1; ++r) {
      const float xv = x[(size_t)r * ld];
      const float4* v = (const float4*)(V + (size_t)r * 16);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 w = v[i];
        a[4 * i] = fmaf(w.x, xv, a[4 * i]);
        a[4 * i + 1] = fmaf(w.y, xv, a[4 * i + 1]);
        a[4 * i + 2] = fmaf(w.z, xv, a[4 * i + 2]);
        a[4 * i + 3] = fmaf(w.w, xv, a[4 * i + 3]);
      }
    }
    if (g > 0) {
#pragma unroll
      for (int q = 0; q < 16; ++q) part[((size_t)(g - 1) * 16 + q) * pld + c] = a[q];
    }
  }
  __syncthreads();
  fold_t();
  if (G > 1) {
    if (act && g == 0) {
      for (int h = 1; h < G; ++h)
#pragma unroll
        for (int q = 0; q < 16; ++q) a[q] += part[((size_t)(h - 1) * 16 + q) * pld + c];
#pragma unroll
      for (int q = 0; q < 16; ++q) part[(size_t)q * pld + c] = a[q];
    }
    __syncthreads();
    if (act && g > 0) {
#pragma unroll
      for (int q = 0; q < 16; ++q) a[q] = part[(size_t)q * pld + c];
    }
  } else {
    __syncthreads();
  }
  if (act) {
    float* x = X + c;
#pragma unroll 4
    for (int r = r0; r < r1; ++r) {
      // the change first: taken from X term by term it would round sixteen times at X's size
      // (directions of mixed roundings 8-16 % further off)
      float s = 0.f;
      const float4* v = (const float4*)(V + (size_t)r * 16);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 w = v[i];
        s = fmaf(w.x, a[4 * i], s);
        s = fmaf(w.y, a[4 * i + 1], s);
        s = fmaf(w.z, a[4 * i + 2], s);
        s = fmaf(w.w, a[4 * i + 3], s);
      }
      x[(size_t)r * ld] -= s;
    }
  }
  __syncthreads();
}

// Shapes qr_reg takes: two rows a thread, columns in one pass of the 16 warps.
__host__ __device__ inline bool qr_reg_fits(int m, int n) { return m <= 2 * QRT && n <= 512; }

// Same factorisation, outputs, sign rule and zero floor as householder_qr_blk
// (scaled FP32 norms, columns below 2^-60 of the largest entry are zero) for A
// (m x n, lda; shared or global memory) with qr_reg_fits(m, n); Q == nullptr: R only.
// V and part: shared memory of qr_reg_vbytes(m) and QR_PART_BYTES; Tg:
// 16 n + 256 floats (any memory) that keep the T factors for the Q pass; sm: 4 KB
// of shared memory.  Called by all QRT threads of the block.
template <int RP, bool SH>
__device__ __noinline__ void qr_reg_run(float* A, int m, int n, int lda, float* Q, int ldq, float* R, int ldr, float* V,
                                        float* part, float* Tg, float* sm) {
  __builtin_assume(__isShared(V));
  __builtin_assume(__isShared(part));
  __builtin_assume(__isShared(sm));
  if (SH) __builtin_assume(__isShared(A));
  float (*sT)[17] = (float (*)[17])sm;
  float (*s_part)[16][16] = (float (*)[16][16])(sm + 272);
  float (*s_row)[16] = (float (*)[16])(sm + 784);
  float* s_max = sm + 816;
  signed char* s_neg = (signed char*)(sm + 832);          // 512
  constexpr unsigned F = 0xffffffffu;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int kk = imin(m, n);
  float amax = 0.f;
  for (int idx = tid; idx < m * n; idx += QRT) amax = fmaxf(amax, fabsf(A[(size_t)(idx / n) * lda + idx % n]));
  for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(F, amax, o));
  if (lane == 0) s_max[wid] = amax;
  __syncthreads();
  float mx = s_max[lane & 15];
  for (int o = 8; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(F, mx, o));
  int ex = 0;
  if (mx > 0.f && isfinite(mx)) frexpf(mx, &ex);
  const float sc2 = ldexpf(1.f, -ex);                // max |A| sc2 in [0.5, 1)
  const float isc2 = 1.f / sc2;
  const float floor2 = (float)m * 7.523164e-37f;     // m (2^-60)^2 in scaled units
  for (int p0 = 0; p0 < kk; p0 += 16) {
    const int pb = imin(16, kk - p0), mr = m - p0;
    const int nwr = imin(16, (mr + 31) / 32);        // warps that hold rows
    float a[RP][16];
#pragma unroll
    for (int h = 0; h < RP; ++h) {
      const int r = tid + h * QRT;
#pragma unroll
      for (int q = 0; q < 16; ++q) a[h][q] = (r < mr && q < pb) ? A[(size_t)(p0 + r) * lda + p0 + q] : 0.f;
    }
    float trow[16];                                  // row `lane` of T (warp 0, lanes 0..15)
#pragma unroll
    for (int q = 0; q < 16; ++q) trow[q] = 0.f;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      if (j >= pb) break;
      const int b = j & 1;
      if (wid < nwr) {
        float v[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) {
          float s = 0.f;
#pragma unroll
          for (int h = 0; h < RP; ++h)
            if (h > 0 || tid > j) {
              const float x = q == j ? a[h][j] * sc2 : a[h][j];
              s = fmaf(x, q == j ? x : a[h][q], s);
            }
          v[q] = s;
        }
        const float t = qr_reduce16(v, lane);
        if (!(lane & 1)) s_part[b][wid][lane >> 1] = t;
        if (tid == j) {
#pragma unroll
          for (int q = 0; q < 16; ++q) s_row[b][q] = a[0][q];
        }
      }
      __syncthreads();
      if (wid < nwr) {
        const int q = lane & 15;
        float s = 0.f;
        for (int w = lane >> 4; w < nwr; w += 2) s += s_part[b][w][q];
        s += __shfl_xor_sync(F, s, 16);
        const float rowq = s_row[b][q];
        const float sig2 = __shfl_sync(F, s, j);
        const float alpha = s_row[b][j] * sc2;
        float tau = 0.f, sc = 0.f, beta = alpha;
        const bool zero = sig2 <= floor2;
        if (!zero) {
          beta = -copysignf(sqrtf(alpha * alpha + sig2), alpha);
          tau = (beta - alpha) / beta;
          sc = sc2 / (alpha - beta);
        }
        // lane q: products of the reflector with column q (q > j), with
        // reflector q (q < j: the entry of the T factor)
        const float wq = rowq + sc * s, uq = wq * tau;
        if (wid == 0) {
          // T[i][j] = -tau_j sum_{k = i}^{j - 1} T[i][k] (V_k^T v_j), T[j][j] = tau_j
          float z = 0.f;
#pragma unroll
          for (int k = 0; k < 16; ++k)
            if (k < j) z = fmaf(trow[k], __shfl_sync(F, wq, k), z);
          trow[j] = lane < j ? -tau * z : lane == j ? tau : 0.f;
        }
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          if (c <= j) continue;
          const float u = __shfl_sync(F, uq, c);
#pragma unroll
          for (int h = 0; h < RP; ++h) {
            if (h > 0 || tid > j) a[h][c] = fmaf(-u * sc, a[h][j], a[h][c]);
            else if (tid == j) a[h][c] -= u;
          }
        }
#pragma unroll
        for (int h = 0; h < RP; ++h) {
          if (h > 0 || tid > j) a[h][j] *= sc;       // the reflector; zero columns (sc = 0) are zeroed
          else if (tid == j && !zero) a[h][j] = beta * isc2;
        }
      }
    }
    // the panel back to A (R and the reflectors), and V with its unit diagonal
#pragma unroll
    for (int h = 0; h < RP; ++h) {
      const int r = tid + h * QRT;
      if (r < mr) {
#pragma unroll
        for (int q = 0; q < 16; ++q) {
          if (q < pb) A[(size_t)(p0 + r) * lda + p0 + q] = a[h][q];
          V[(size_t)r * 16 + q] = (q >= pb || r < q) ? 0.f : r == q ? 1.f : a[h][q];
        }
      }
    }
    if (wid == 0 && lane < 16) {
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        sT[lane][q] = trow[q];
        Tg[(size_t)(p0 / 16) * 256 + lane * 16 + q] = trow[q];
      }
    }
    __syncthreads();
    if (n - p0 - pb > 0)
      qr_reg_update(V, mr, A + (size_t)p0 * lda + p0 + pb, lda, n - p0 - pb, sT, true, part);
  }
  // R with non-negative diagonal; the signs go to Q
  for (int idx = tid; idx < kk * n; idx += QRT) {
    const int i = idx / n, c = idx % n;
    const bool neg = A[(size_t)i * lda + i] < 0.f;
    const float v = c >= i ? A[(size_t)i * lda + c] : 0.f;
    R[(size_t)i * ldr + c] = neg ? -v : v;
    if (c == i) s_neg[i] = neg ? 1 : 0;
  }
  __syncthreads();
  if (Q == nullptr) return;
  // Q = (I - V_0 T_0 V_0^T) ... [I; 0], backwards in place of the reflectors
  for (int p0 = ((kk - 1) / 16) * 16; p0 >= 0; p0 -= 16) {
    const int pb = imin(16, kk - p0), mr = m - p0;
    for (int r = tid; r < mr; r += QRT)
#pragma unroll
      for (int q = 0; q < 16; ++q)
        V[(size_t)r * 16 + q] = (q >= pb || r < q) ? 0.f : r == q ? 1.f : A[(size_t)(p0 + r) * lda + p0 + q];
    if (tid < 256) sT[tid >> 4][tid & 15] = Tg[(size_t)(p0 / 16) * 256 + tid];
    __syncthreads();
    for (int idx = tid; idx < m * pb; idx += QRT) {
      const int i = idx / pb, c = p0 + idx % pb;
      A[(size_t)i * lda + c] = i == c ? 1.f : 0.f;
    }
    __syncthreads();
    qr_reg_update(V, mr, A + (size_t)p0 * lda + p0, lda, kk - p0, sT, false, part);
  }
  for (int idx = tid; idx < m * kk; idx += QRT) {
    const int i = idx / kk, c = idx % kk;
    const float q = A[(size_t)i * lda + c];
    Q[(size_t)i * ldq + c] = s_neg[c] ? -q : q;
  }
  __syncthreads();
}

__device__ __forceinline__ void qr_reg(float* A, int m, int n, int lda, float* Q, int ldq, float* R, int ldr, float* V,
                                       float* part, float* Tg, float* sm) {
  if (m <= QRT && __isShared(A)) qr_reg_run<1, true>(A, m, n, lda, Q, ldq, R, ldr, V, part, Tg, sm);
  else if (m <= QRT) qr_reg_run<1, false>(A, m, n, lda, Q, ldq, R, ldr, V, part, Tg, sm);
  else qr_reg_run<2, false>(A, m, n, lda, Q, ldq, R, ldr, V, part, Tg, sm);
}

}  // namespace tn
