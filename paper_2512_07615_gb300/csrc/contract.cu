// Contraction of an MPS to a dense [x][y][z] field (Eq. MPS) and the sums of
// populations to rho and j that outputs are made of.
//
// The chain is split at h = L / 2: f(l, q) = sum_j Lm(l, j) Rt(q, j) with the
// 2^h prefixes l and the 2^(L-h) suffixes q.  All sums carry 53 bits whatever the
// storage type: FP32 products of L cores would bias sums over the lattice at the
// 1e-6 level.
//
// FP64 runs at two multiply-adds a clock and SM on GB300, so that is what the
// work is counted in.
//  - Prefixes and suffixes: a CTA forms 2^TREE_BITS neighbouring rows: their common
//    sites once, then a site at a time doubles the rows (one row alone would redo
//    all L / 2 sites).  128^3 at bond 64: 86 k multiply-adds for eight rows, not 330 k.
//  - The join, 2^L r multiply-adds (134 M at 128^3 and bond 64: 0.23 ms of FP64), for FP32
//    storage on the tensor cores, exactly: every row is cut into seven signed
//    base-256 digits relative to its largest entry (55 bits), BF16 holds a digit,
//    a product of two has 14 bits, and the sum of the at most 7 x 128 products of one weight
//    24: an FP32 accumulator holds it exactly (Ozaki, Ogita, Oishi and Rump, "Error-free
//    transformations of matrix multiplication", 2012).  The columns of both sides are first
//    balanced by powers of two.  The 34 digit products of
//    weight 256^-7 and more go to eight accumulators in tensor memory, which the epilogue
//    adds as integers: one rounding per value, four FP64 instructions in place of r.
//    What is left out, relative to the product of the two rows' largest entries: the products of
//    weight 256^-8 and less, at most 5 x 128 x 2^-64 and a little, 2^-54.7; and the cut of the
//    entries to 55 bits, at most 2 x 128 x 2^-56 = 2^-48 (an FP64 sum of 128 rounded products:
//    2^-46).
// The digits lie in global memory in the order of the MMA's shared-memory layout
// (8 x 16-byte core matrices, no swizzle), one bulk copy per operand and K chunk,
// and the rows of both sides in the order of their coordinates, z fastest, so that a
// thread's outputs are runs of z.
//
// Measured per 128^3 field at bond 64: rows 0.11 ms, digits 0.01 ms, join 0.05 ms (0.09 with
// the sums to rho and j), where a row per CTA and an FP64 join took 0.8 ms; rho and u of
// 19 populations on the host: 19.6 -> 7.6 ms.  Against the sums in rational arithmetic u is
// off by 1e-18 to 7e-18, with the FP64 join by 8e-18 to 2.5e-17 (u ~ 1e-4).
#include <algorithm>

#include "fit.cuh"
#include "tcgemm.cuh"

namespace tn {

static constexpr int TREE_BITS = 3;      // rows of a CTA: 2^TREE_BITS
static constexpr int TREE_THREADS = 256;
static constexpr int TREE_KC = 32;       // staged entries of a row of the right cores
static constexpr int DIGITS = 7;         // base-256 digits of an entry
static constexpr int GROUPS = 8;         // digit products p + q < GROUPS are kept
static constexpr int JM = 128, JN = 32, JK = 32;   // prefixes, suffixes, bonds of a tile
static constexpr int J_MAXR = 128;       // bonds up to which the sums of digit products are exact
static constexpr int J_A = DIGITS * JM * JK, J_B = DIGITS * JN * JK;   // digits of a tile's chunk
static constexpr int E_NONFINITE = 1 << 20;
static constexpr int J_SMEM = 100 * 1024;     // not the ~71 KB used: two CTAs an SM, as the tensor memory holds
static_assert((J_A + J_B) * 2 + 1024 <= J_SMEM, "a chunk of both operands");

// x in FP64.  Normal numbers by moving their bits: the conversion instruction runs on
// the FP64 pipes, which bound these kernels.
__device__ __forceinline__ double wide(double x) { return x; }
__device__ __forceinline__ double wide(float x) {
  const unsigned u = __float_as_uint(x), e = u & 0x7f800000u;
  if (e == 0u || e == 0x7f800000u) return (u << 1) == 0u ? 0.0 : (double)x;
  return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(u << 29));
}

// ---------------------------------------------------------------- prefixes and suffixes
// One site: in (R rows of the near bond) -> out (R rows of the far bond for one index
// value s, 2 R for s < 0).  Columns over the threads, the sum over the near bond split
// when there are fewer columns than threads.
// Left: out row 2 row + s, out[., j] = sum_i in[row, i] A(i, s, j).
template <typename T, int R>
__device__ __forceinline__ void tree_left(const T* __restrict__ A, int r0, int r1, int s, const double* in, double* out,
                                          int ld, double* part) {
  const int nc = s < 0 ? 2 * r1 : r1;
  const T* Ab = A + (s < 0 ? 0 : (size_t)s * r1);
  const int ncp = (imin(nc, TREE_THREADS) + 31) & ~31, G = TREE_THREADS / ncp;
  for (int c0 = 0; c0 < nc; c0 += TREE_THREADS) {
    const int cl = threadIdx.x % ncp, c = c0 + cl, g = threadIdx.x / ncp;
    const bool act = c < nc && g < G;
    double acc[R];
#pragma unroll
    for (int q = 0; q < R; ++q) acc[q] = 0.0;
    if (act)
#pragma unroll 8
      for (int i = g; i < r0; i += G) {
        const double a = wide(Ab[(size_t)i * 2 * r1 + c]);
#pragma unroll
        for (int q = 0; q < R; ++q) acc[q] = fma(in[(size_t)q * ld + i], a, acc[q]);
      }
    if (G > 1) {
      if (act)
#pragma unroll
        for (int q = 0; q < R; ++q) part[(g * R + q) * ncp + cl] = acc[q];
      __syncthreads();
    }
    if (c < nc && g == 0) {
      const int sc = s < 0 ? c / r1 : 0, j = s < 0 ? c - sc * r1 : c;
#pragma unroll
      for (int q = 0; q < R; ++q) {
        double v = acc[q];
        for (int p = 1; p < G; ++p) v += part[(p * R + q) * ncp + cl];
        out[(size_t)(s < 0 ? 2 * q + sc : q) * ld + j] = v;
      }
    }
    if (G > 1) __syncthreads();
  }
  __syncthreads();
}

// Right: out row s R + row, out[., i] = sum_j A(i, s, j) in[row, j].  The rows of A are
// staged TREE_KC entries at a time (they are read across otherwise).
template <typename T, int R>
__device__ __forceinline__ void tree_right(const T* __restrict__ A, int r0, int r1, int s, const double* in, double* out,
                                           int ld, double* part, T* st) {
  const int nc = s < 0 ? 2 * r0 : r0;
  const int ncp = (imin(nc, TREE_THREADS) + 31) & ~31, G = TREE_THREADS / ncp;
  for (int c0 = 0; c0 < nc; c0 += TREE_THREADS) {
    const int cl = threadIdx.x % ncp, c = c0 + cl, g = threadIdx.x / ncp;
    const int here = imin(nc - c0, TREE_THREADS);
    const bool act = c < nc && g < G;
    double acc[R];
#pragma unroll
    for (int q = 0; q < R; ++q) acc[q] = 0.0;
    for (int j0 = 0; j0 < r1; j0 += TREE_KC) {
      const int nk = imin(TREE_KC, r1 - j0);
      __syncthreads();
#pragma unroll 8
      for (int e = threadIdx.x; e < here * TREE_KC; e += TREE_THREADS) {
        const int w = e / TREE_KC, kk = e % TREE_KC, row = s < 0 ? c0 + w : 2 * (c0 + w) + s;
        if (kk < nk) st[w * (TREE_KC + 1) + kk] = A[(size_t)row * r1 + j0 + kk];
      }
      __syncthreads();
      if (act)
        for (int kk = g; kk < nk; kk += G) {
          const double a = wide(st[cl * (TREE_KC + 1) + kk]);
#pragma unroll
          for (int q = 0; q < R; ++q) acc[q] = fma(in[(size_t)q * ld + j0 + kk], a, acc[q]);
        }
    }
    if (G > 1) {
      if (act)
#pragma unroll
        for (int q = 0; q < R; ++q) part[(g * R + q) * ncp + cl] = acc[q];
      __syncthreads();
    }
    if (c < nc && g == 0) {
      const int sc = s < 0 ? c & 1 : 0, i = s < 0 ? c >> 1 : c;
#pragma unroll
      for (int q = 0; q < R; ++q) {
        double v = acc[q];
        for (int p = 1; p < G; ++p) v += part[(p * R + q) * ncp + cl];
        out[(size_t)(sc * R + q) * ld + i] = v;
      }
    }
    if (G > 1) __syncthreads();
  }
  __syncthreads();
}

static constexpr int TREE_PART = 4 * TREE_THREADS;       // partial sums: G R ncp <= 4 x 256
template <typename T>
static size_t tree_smem(int ld) {
  return ((size_t)2 * (1 << TREE_BITS) * ld + TREE_PART) * sizeof(double) +
         (size_t)TREE_THREADS * (TREE_KC + 1) * sizeof(T);
}

// Rows of both sides: CTAs [0, nl) the prefixes, the rest the suffixes.  tops (if not null):
// the largest exponent field of every column of Lm, then of Rt (ld apart).
template <typename T>
__global__ void __launch_bounds__(TREE_THREADS) tree_kernel(MpsRef X, int L, int h, int nl, int ld, double* __restrict__ Lm,
                                                            double* __restrict__ Rt, int* __restrict__ tops) {
  extern __shared__ __align__(16) unsigned char tsm[];
  double* a = (double*)tsm;
  double* b = a + (size_t)(1 << TREE_BITS) * ld;
  double* part = b + (size_t)(1 << TREE_BITS) * ld;
  T* st = (T*)(part + TREE_PART);
  const bool left = (int)blockIdx.x < nl;
  const int sites = left ? h : L - h, bits = imin(TREE_BITS, sites);
  const int idx = left ? blockIdx.x : blockIdx.x - nl;
  if (threadIdx.x == 0) a[0] = 1.0;
  __syncthreads();
  size_t off = left ? 0 : mps_size(L, X.cap);
  int rows = 1, far = 1;
  for (int c = 0; c < sites; ++c) {
    const int k = left ? c : L - 1 - c;
    const int r0 = X.ranks[k], r1 = X.ranks[k + 1];
    const size_t size = (size_t)bond_cap(L, X.cap, k) * 2 * bond_cap(L, X.cap, k + 1);
    if (!left) off -= size;
    const T* A = (const T*)X.base + off;
    if (left) off += size;
    const int s = c < sites - bits ? (idx >> (left ? sites - bits - 1 - c : c)) & 1 : -1;
    if (left) {
      if (rows == 1) tree_left<T, 1>(A, r0, r1, s, a, b, ld, part);
      else if (rows == 2) tree_left<T, 2>(A, r0, r1, s, a, b, ld, part);
      else tree_left<T, 4>(A, r0, r1, s, a, b, ld, part);
    } else {
      if (rows == 1) tree_right<T, 1>(A, r0, r1, s, a, b, ld, part, st);
      else if (rows == 2) tree_right<T, 2>(A, r0, r1, s, a, b, ld, part, st);
      else tree_right<T, 4>(A, r0, r1, s, a, b, ld, part, st);
    }
    if (s < 0) rows *= 2;
    double* t = a; a = b; b = t;
    far = left ? r1 : r0;
  }
  for (int j = threadIdx.x; j < far; j += TREE_THREADS) {
    int top = 0;
    for (int w = 0; w < rows; ++w) {
      const double v = a[(size_t)w * ld + j];
      top = imax(top, (__double2hiint(v) >> 20) & 0x7ff);
      if (left) Lm[(((size_t)idx << bits) + w) * ld + j] = v;
      else Rt[(((size_t)w << (sites - bits)) + idx) * ld + j] = v;
    }
    if (tops) atomicMax(tops + (left ? 0 : ld) + j, top);
  }
}

// ---------------------------------------------------------------- join, FP64
template <typename T>
__global__ void join_kernel(const int* ranks, int n, int h, const double* Lm, const double* Rt, int ld, T* out) {
  const int L = 3 * n;
  const size_t N = (size_t)1 << n;
  const size_t total = N * N * N;
  const int rh = ranks[h];
  for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < total;
       idx += (size_t)gridDim.x * blockDim.x) {
    const int z = (int)(idx % N), y = (int)((idx / N) % N), x = (int)(idx / (N * N));
    const size_t si = site_index(x, y, z, n);
    const size_t l = si >> (L - h), q = si & (((size_t)1 << (L - h)) - 1);
    const double* a = Lm + l * ld;
    const double* b = Rt + q * ld;
    double acc = 0.0;
    for (int j = 0; j < rh; ++j) acc += a[j] * b[j];
    out[idx] = (T)acc;
  }
}

// ---------------------------------------------------------------- join by digits
// Coordinate bits of the sites [k0, k1) of each axis.
__host__ __device__ inline int axis_bits(int k0, int k1, int axis) {
  int c = 0;
  for (int k = k0; k < k1; ++k) c += k % 3 == axis;
  return c;
}

// A row's place among the rows of its side (sites [k0, k1), first site in the highest
// bit) when they are ordered by (x, y, z), z fastest; and back.
__device__ inline int coord_order(int row, int k0, int k1) {
  int v[3] = {0, 0, 0};
  for (int k = k0; k < k1; ++k) v[k % 3] = 2 * v[k % 3] + ((row >> (k1 - 1 - k)) & 1);
  return (((v[0] << axis_bits(k0, k1, 1)) | v[1]) << axis_bits(k0, k1, 2)) | v[2];
}
__device__ inline int site_order(int place, int k0, int k1) {
  const int by = axis_bits(k0, k1, 1), bz = axis_bits(k0, k1, 2);
  int v[3] = {place >> (by + bz), (place >> bz) & ((1 << by) - 1), place & ((1 << bz) - 1)};
  int row = 0;
  for (int k = k1 - 1; k >= k0; --k) {
    row |= (v[k % 3] & 1) << (k1 - 1 - k);
    v[k % 3] >>= 1;
  }
  return row;
}

struct JoinBuf {
  uint16_t *a, *b;         // digits of the prefixes and suffixes, by tile, chunk and digit
  int *ea, *eb;            // exponents of their rows (E_NONFINITE: a row that is not finite)
  int chunks;              // K chunks per tile that there is room for
};

// Digits of a row (one warp): entries x = q 2^(e - 55) with |x| <= 2^e.
__global__ void __launch_bounds__(256) digits_kernel(const int* __restrict__ ranks, int L, int h, int ld,
                                                     const double* __restrict__ Lm, const double* __restrict__ Rt,
                                                     const int* __restrict__ tops, JoinBuf J) {
  const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (w >= (1 << h) + (1 << (L - h))) return;
  const bool left = w < (1 << h);
  const int row = left ? w : w - (1 << h), r = ranks[h];
  const double* x = (left ? Lm : Rt) + (size_t)row * ld;
  // column j of Lm times 2^s, of Rt times 2^-s: their largest entries become alike, so that the
  // digits of a row resolve each term of the sum to the same part of its bound
  auto at = [&](int j) -> double {
    const int tl = tops[j], tr = tops[ld + j];
    if (tl == 0 || tr == 0 || tl == 0x7ff || tr == 0x7ff) return x[j];
    const int s = imax(-500, imin(500, (tr - tl) / 2));
    return x[j] * __hiloint2double((1023 + (left ? s : -s)) << 20, 0);
  };
  const int place = left ? coord_order(row, 0, h) : coord_order(row, h, L);
  double m = 0.0;
  bool bad = false;
  for (int j = lane; j < r; j += 32) {
    const double v = at(j);
    m = fmax(m, fabs(v));
    bad |= !isfinite(v);
  }
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  int e = 0;
  if (m > 0.0) frexp(m, &e);
  // beyond this the scales could leave the FP64 range: such a row is summed in FP64
  bad = __any_sync(0xffffffffu, bad) || e > 400 || e < -400;
  if (lane == 0) (left ? J.ea : J.eb)[place] = bad ? E_NONFINITE : e;
  const double scl = bad ? 0.0 : __hiloint2double((1023 + 55 - e) << 20, 0);
  const int rows = left ? JM : JN;
  uint16_t* d = (left ? J.a : J.b) + (size_t)(place / rows) * J.chunks * (left ? J_A : J_B);
  const int rt = place % rows;
  for (int j = lane; j < (r + JK - 1) / JK * JK; j += 32) {
    long long q = j < r && !bad ? __double2ll_rn(at(j) * scl) : 0;
    const int kk = j % JK;
    uint16_t* p = d + (size_t)(j / JK) * (left ? J_A : J_B) + ((rt >> 3) * (JK / 8) + kk / 8) * 64 + (rt & 7) * 8 + kk % 8;
#pragma unroll
    for (int g = DIGITS - 1; g >= 0; --g) {
      const int v = g > 0 ? (int)(signed char)(q & 255) : (int)q;
      q = (q - v) >> 8;
      p[(size_t)g * rows * JK] = tc_bf16((float)v);
    }
  }
}

__device__ __forceinline__ void tc_ld8(uint32_t addr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(addr));
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t mbar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(mbar)
               : "memory");
}
// An integer below 2^51 in FP64 (one addition; the conversion costs more).
__device__ __forceinline__ double whole(long long v) {
  return __longlong_as_double(0x4338000000000000LL + v) - 6755399441055744.0;
}

// Where the values go: a field, or the sums over populations: rho (+)= f, j_d (+)= c_d f.
template <typename T>
struct FieldOut {
  T* out;
  __device__ __forceinline__ void put(size_t at, const double (&v)[8]) const {
    if constexpr (sizeof(T) == 4) {
      *(float4*)(out + at) = make_float4((float)v[0], (float)v[1], (float)v[2], (float)v[3]);
      *(float4*)(out + at + 4) = make_float4((float)v[4], (float)v[5], (float)v[6], (float)v[7]);
    } else {
#pragma unroll
      for (int i = 0; i < 8; i += 2) *(double2*)(out + at + i) = make_double2(v[i], v[i + 1]);
    }
  }
};
struct MomentOut {
  double* m[4];            // rho, jx, jy, jz
  int c[3];
  int first;
  __device__ __forceinline__ void put(size_t at, const double (&v)[8]) const {
#pragma unroll
    for (int d = 0; d < 4; ++d) {
      const int f = d == 0 ? 1 : c[d - 1];
      bool need = first || f != 0;
#pragma unroll
      for (int i = 0; i < 8; ++i) need |= !isfinite(v[i]);           // 0 * v is then NaN
      if (!need) continue;
      double2* p = (double2*)(m[d] + at);
#pragma unroll
      for (int i = 0; i < 8; i += 2) {
        double2 o = first ? make_double2(0.0, 0.0) : p[i / 2];
        const double x = f == 1 ? v[i] : f == -1 ? -v[i] : f * v[i], y = f == 1 ? v[i + 1] : f == -1 ? -v[i + 1] : f * v[i + 1];
        o.x = first ? x : o.x + x;
        o.y = first ? y : o.y + y;
        p[i / 2] = o;
      }
    }
  }
};

// 128 prefixes x 32 suffixes per CTA; two CTAs an SM, so that one's products run under
// the other's epilogue.  Bound by the epilogue's FP64 instructions.
template <typename Out>
__global__ void __launch_bounds__(256, 2) join_digits_kernel(const int* __restrict__ ranks, int n, int h,
                                                             const double* __restrict__ Lm, const double* __restrict__ Rt,
                                                             int ld, JoinBuf J, Out out, int* status) {
  extern __shared__ __align__(1024) unsigned char jsm[];
  __shared__ __align__(8) uint64_t s_bar[2];
  __shared__ uint32_t s_tmem;
  __shared__ int s_fail;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t full = tc_smem(&s_bar[0]), done = tc_smem(&s_bar[1]);
  const uint32_t sa = (tc_smem(jsm) + 1023u) & ~1023u, sb = sa + J_A * 2;
  const int r = ranks[h], nch = (r + JK - 1) / JK;
  const int nbt = (1 << (3 * n - h)) / JN, ta = blockIdx.x / nbt, tb = blockIdx.x % nbt;
  if (tid == 0) {
    s_fail = 0;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(full));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(done));
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_smem(&s_tmem)),
                 "r"(GROUPS * JN));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = s_tmem;
  if (tid == 0) {
    const uint32_t idesc = tc_idesc(JM, JN, true), sbo = (JK / 8) * 128;
    bool ok = true;
    int ch = 0;
    for (; ch < nch; ++ch) {
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(full), "r"((J_A + J_B) * 2) : "memory");
      bulk_load(sa, J.a + ((size_t)ta * J.chunks + ch) * J_A, J_A * 2, full);
      bulk_load(sb, J.b + ((size_t)tb * J.chunks + ch) * J_B, J_B * 2, full);
      ok = tc_wait(full, ch & 1);
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int steps = (imin(JK, r - ch * JK) + 15) / 16;              // the rest of the chunk is zero
#pragma unroll 1
      for (int g = 0; g < GROUPS; ++g)
#pragma unroll 1
        for (int p = imax(0, g - DIGITS + 1); p <= imin(g, DIGITS - 1); ++p)
#pragma unroll 1
          for (int s = 0; s < steps; ++s) {
            const uint64_t da = tc_sdesc(sa + p * (JM * JK * 2) + s * 256, 128, sbo);
            const uint64_t db = tc_sdesc(sb + (g - p) * (JN * JK * 2) + s * 256, 128, sbo);
            const uint32_t acc = ch > 0 || s > 0 || p > imax(0, g - DIGITS + 1);
            asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                         "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                         ::"r"(tmem + g * JN), "l"(da), "l"(db), "r"(idesc), "r"(acc));
          }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(done) : "memory");
      ok = tc_wait(done, ch & 1);
      if (!ok) break;
    }
    if (!ok) {
      // what is in flight ends before this CTA's memory is given back
      tc_wait(full, ch & 1);
      tc_wait(done, ch & 1);
      s_fail = 1;
    }
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (s_fail) {
    if (tid == 0) atomicOr(status, ST_TIMEOUT);
  } else {
    const int L = 3 * n, N = 1 << n;
    const int ly = axis_bits(0, h, 1), lz = axis_bits(0, h, 2);
    const int qx = axis_bits(h, L, 0), qy = axis_bits(h, L, 1), qz = axis_bits(h, L, 2);
    const int l = ta * JM + 32 * (warp & 3) + lane, c0 = (JN / 2) * (warp >> 2);
    const int lxv = l >> (ly + lz), lyv = (l >> lz) & ((1 << ly) - 1), lzv = l & ((1 << lz) - 1);
    const int ea = J.ea[l];
#pragma unroll 1
    for (int b = 0; b < JN / 2; b += 8) {
      uint32_t G[GROUPS][8];
#pragma unroll
      for (int g = 0; g < GROUPS; ++g) tc_ld8(tmem + ((uint32_t)(32 * (warp & 3)) << 16) + g * JN + c0 + b, G[g]);
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      const int q0 = tb * JN + c0 + b;                                  // eight z in a row
      double v[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int e = ea + J.eb[q0 + i];
        if (e < E_NONFINITE / 2) {
          long long hi = 0, lo = 0;
#pragma unroll
          for (int g = 0; g < GROUPS / 2; ++g) {
            hi = hi * 256 + __float2int_rn(__uint_as_float(G[g][i]));
            lo = lo * 256 + __float2int_rn(__uint_as_float(G[g + GROUPS / 2][i]));
          }
          v[i] = fma(whole(hi), 4294967296.0, whole(lo)) * __hiloint2double((1023 + e - 70) << 20, 0);
        } else {
          const double* x = Lm + (size_t)site_order(l, 0, h) * ld;
          const double* y = Rt + (size_t)site_order(q0 + i, h, L) * ld;
          double a = 0.0;
          for (int j = 0; j < r; ++j) a += x[j] * y[j];
          v[i] = a;
        }
      }
      const int qxv = q0 >> (qy + qz), qyv = (q0 >> qz) & ((1 << qy) - 1), qzv = q0 & ((1 << qz) - 1);
      out.put(((size_t)((lxv << qx) | qxv) * N + ((lyv << qy) | qyv)) * N + ((lzv << qz) | qzv), v);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(GROUPS * JN));
}

// ---------------------------------------------------------------- host
// The digits from 64^3 on (the eight outputs of a thread's step are then z neighbours),
// up to the bond at which their sums stay exact.  Below, FP64 joins
// 32^3 x 64 in 4 us, and FP64 storage carries more bits than a row's digits hold of its
// small entries.
template <typename T>
static bool by_digits(int n_bits, int cap) {
  return sizeof(T) == 4 && n_bits >= 6 && cap <= J_MAXR;
}

struct ContractPlan {
  int L, h, ld, chunks;
  size_t lm, rt, a, b, ea, eb, tops, total;      // byte offsets in the scratch, after the status word
};
// The size is no monotonic function of cap: the digits come with the caps that take them.
static ContractPlan contract_plan(int n_bits, int cap, bool digits) {
  ContractPlan p;
  p.L = 3 * n_bits;
  p.h = p.L / 2;
  p.ld = bond_cap(p.L, cap, p.h);
  p.chunks = (p.ld + JK - 1) / JK;
  const size_t nl = (size_t)1 << p.h, nr = (size_t)1 << (p.L - p.h);
  size_t o = 256;
  auto take = [&](size_t bytes) { const size_t at = o; o += (bytes + 255) & ~(size_t)255; return at; };
  p.lm = take(nl * p.ld * sizeof(double));
  p.rt = take(nr * p.ld * sizeof(double));
  if (digits) {
    p.a = take(nl / JM * p.chunks * J_A * sizeof(uint16_t));
    p.b = take(nr / JN * p.chunks * J_B * sizeof(uint16_t));
    p.ea = take(nl * sizeof(int));
    p.eb = take(nr * sizeof(int));
    p.tops = take((size_t)2 * p.ld * sizeof(int));
  } else {
    p.a = p.b = p.ea = p.eb = p.tops = 0;
  }
  p.total = o;
  return p;
}

size_t contract_scratch_bytes(int n_bits, int cap, size_t elem) {
  return contract_plan(n_bits, cap, elem == 4 && by_digits<float>(n_bits, cap)).total;
}

static int contract_short() {
  set_error("the scratch of a contraction is too small");
  return TNLBM_E_ARG;
}

// Prefix and suffix rows of X (and their digits).
template <typename T>
static void contract_rows(const MpsRef& X, int n_bits, const ContractPlan& p, unsigned char* scr, cudaStream_t st) {
  double* Lm = (double*)(scr + p.lm);
  double* Rt = (double*)(scr + p.rt);
  const size_t smem = tree_smem<T>(p.ld);
  cudaFuncSetAttribute(tree_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  const int nl = 1 << (p.h - imin(TREE_BITS, p.h)), nr = 1 << (p.L - p.h - imin(TREE_BITS, p.L - p.h));
  const bool digits = by_digits<T>(n_bits, X.cap);
  int* tops = digits ? (int*)(scr + p.tops) : nullptr;
  if (digits) cudaMemsetAsync(tops, 0, (size_t)2 * p.ld * sizeof(int), st);
  tree_kernel<T><<<nl + nr, TREE_THREADS, smem, st>>>(X, p.L, p.h, nl, p.ld, Lm, Rt, tops);
  if (digits) {
    const JoinBuf J{(uint16_t*)(scr + p.a), (uint16_t*)(scr + p.b), (int*)(scr + p.ea), (int*)(scr + p.eb), p.chunks};
    const int rows = (1 << p.h) + (1 << (p.L - p.h));
    digits_kernel<<<(rows + 7) / 8, 256, 0, st>>>(X.ranks, p.L, p.h, p.ld, Lm, Rt, tops, J);
  }
}

template <typename Out>
static void join_digits(const MpsRef& X, int n_bits, const ContractPlan& p, unsigned char* scr, const Out& out,
                        cudaStream_t st) {
  const JoinBuf J{(uint16_t*)(scr + p.a), (uint16_t*)(scr + p.b), (int*)(scr + p.ea), (int*)(scr + p.eb), p.chunks};
  cudaFuncSetAttribute(join_digits_kernel<Out>, cudaFuncAttributeMaxDynamicSharedMemorySize, J_SMEM);
  const unsigned tiles = (1u << p.h) / JM * ((1u << (p.L - p.h)) / JN);
  join_digits_kernel<Out><<<tiles, 256, J_SMEM, st>>>(X.ranks, n_bits, p.h, (const double*)(scr + p.lm),
                                                      (const double*)(scr + p.rt), p.ld, J, out, (int*)scr);
}

template <typename T, typename OutT>
static int contract_to(const MpsRef& X, int n_bits, OutT* d_dense, void* d_scratch, size_t scratch_bytes, cudaStream_t st) {
  const bool digits = by_digits<T>(n_bits, X.cap);
  const ContractPlan p = contract_plan(n_bits, X.cap, digits);
  if (p.total > scratch_bytes) return contract_short();
  unsigned char* scr = (unsigned char*)d_scratch;
  contract_rows<T>(X, n_bits, p, scr, st);
  if (digits && (size_t)d_dense % 16 == 0)
    join_digits(X, n_bits, p, scr, FieldOut<OutT>{d_dense}, st);
  else
    join_kernel<OutT><<<152 * 16, 256, 0, st>>>(X.ranks, n_bits, p.h, (const double*)(scr + p.lm), (const double*)(scr + p.rt),
                                                p.ld, d_dense);
  return 0;
}

void contract_begin(void* d_scratch, cudaStream_t st) { cudaMemsetAsync(d_scratch, 0, sizeof(int), st); }

int contract_end(const void* d_scratch, cudaStream_t st, const char* what) {
  int status = 0;
  cudaError_t e = cudaMemcpyAsync(&status, d_scratch, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaGetLastError();
  const cudaError_t s = cudaStreamSynchronize(st);
  if (e == cudaSuccess) e = s;
  if (e != cudaSuccess) return cuda_fail(e, what);
  if (status & ST_TIMEOUT) {
    set_error(std::string("a bounded wait ran out in ") + what);
    return TNLBM_E_TIMEOUT;
  }
  return 0;
}

template <typename T>
int contract_dense(const MpsRef& X, int n_bits, T* d_dense, void* d_scratch, size_t scratch_bytes, cudaStream_t st) {
  return contract_to<T, T>(X, n_bits, d_dense, d_scratch, scratch_bytes, st);
}

template <typename T>
int contract_dense_f64(const MpsRef& X, int n_bits, double* d_dense, void* d_scratch, size_t scratch_bytes,
                       cudaStream_t st) {
  return contract_to<T, double>(X, n_bits, d_dense, d_scratch, scratch_bytes, st);
}

template <typename T>
int contract_moments(const MpsRef& X, int n_bits, double* tmp, void* d_scratch, size_t scratch_bytes, double* rho,
                     double* jx, double* jy, double* jz, int cx, int cy, int cz, int first, cudaStream_t st) {
  if (by_digits<T>(n_bits, X.cap)) {
    const ContractPlan p = contract_plan(n_bits, X.cap, true);
    if (p.total > scratch_bytes) return contract_short();
    contract_rows<T>(X, n_bits, p, (unsigned char*)d_scratch, st);
    join_digits(X, n_bits, p, (unsigned char*)d_scratch, MomentOut{{rho, jx, jy, jz}, {cx, cy, cz}, first}, st);
    return 0;
  }
  const int rc = contract_to<T, double>(X, n_bits, tmp, d_scratch, scratch_bytes, st);
  if (!rc) launch_accum_moments<double>(tmp, (size_t)1 << (3 * n_bits), rho, jx, jy, jz, cx, cy, cz, first, st);
  return rc;
}

#define INST(T)                                                                                    \
  template int contract_dense<T>(const MpsRef&, int, T*, void*, size_t, cudaStream_t);            \
  template int contract_dense_f64<T>(const MpsRef&, int, double*, void*, size_t, cudaStream_t);    \
  template int contract_moments<T>(const MpsRef&, int, double*, void*, size_t, double*, double*, double*, double*, int, \
                                   int, int, int, cudaStream_t);
INST(float)
INST(double)

}  // namespace tn
