// TT-rounding of linear combinations of exactly formed terms (one CTA per job).
//
// For a job sum_t coef_t X_t the wide MPS is the block-diagonal sum of Eq. (add);
// its cores are never stored as a whole: at site k the term blocks are formed
// (plain copy, rank-1 mask product, Kronecker product of Eq. (mul), or the shift
// MPO x MPS contraction of Eq. (applympo) with the cores of Sec. 2.5), multiplied
// from the left by the R factor carried from site k-1, and QR-factorised
// (left-orthogonalising sweep, Eq. lorg).  The right-to-left sweep then moves the
// canonical centre back to site 0 with SVDs (Eq. svd-move) and truncates at the
// centre to chi / eps.
#include <algorithm>
#include <type_traits>

#include "cluster.cuh"
#include "jacobi_reg.cuh"
#include "jacobi_wide.cuh"
#include "linalg.cuh"
#include "qr_reg.cuh"
#include "refine64.cuh"
#include "rows_layout.cuh"

namespace tn {

static constexpr int RT = 512;                      // threads per rounding CTA
static constexpr int MAXK = 1024;                   // max columns of a QR / SVD

size_t round_smem_bytes() { return SM_SMALL + SM_WORK; }

// ---------------------------------------------------------------- layout (host)
void plan_round_job(RoundJob& j, int L, int n_bits, size_t eb) {
  for (int k = 0; k <= L; ++k) {
    int s = 0;
    for (int t = 0; t < j.nterms; ++t) s += term_bond_bound(j.t[t], L, n_bits, k);
    j.rw[k] = (k == 0 || k == L) ? 1 : s;
  }
  // QR-sweep bonds: q_0 = 1, q_{k+1} <= min(2 q_k, rw_{k+1})
  j.qb[0] = 1;
  for (int k = 0; k < L; ++k) j.qb[k + 1] = imin(2 * j.qb[k], j.rw[k + 1]);
  j.qb[L] = 1;
  size_t off = 0;
  auto al = [&](size_t n) { size_t o = off; off += (n + 31) & ~(size_t)31; return o; };
  for (int k = 0; k < L; ++k) j.lay.q_off[k] = al((size_t)2 * j.qb[k] * (k == L - 1 ? 1 : j.qb[k + 1]));
  size_t wmax = 0, mmax = 0, rmax = 0, cmax = 0, jw = 0, jv = 0, us = 0, rz = 0, qw = 0;
  for (int k = 0; k < L; ++k) {
    size_t w = 0;
    for (int t = 0; t < j.nterms; ++t)
      w += (size_t)term_bond_bound(j.t[t], L, n_bits, k) * 2 * term_bond_bound(j.t[t], L, n_bits, k + 1);
    wmax = w > wmax ? w : wmax;
    size_t m = (size_t)j.qb[k] * 2 * j.rw[k + 1];
    mmax = m > mmax ? m : mmax;
    // blocked QR of M (2 q_k x rw_{k+1}): panel reflectors and products
    const size_t qs = qr_blk_scratch<float>(2 * j.qb[k], j.rw[k + 1]);
    qw = qs > qw ? qs : qw;
    size_t r = (size_t)j.qb[k + 1] * j.rw[k + 1];
    rmax = r > rmax ? r : rmax;
    // right sweep at site k: C is q_k x 2 r_{k+1}, r_{k+1} <= min(chi, q_{k+1})
    size_t rn = (size_t)imin(j.chi, j.qb[k + 1]);
    size_t cm = (size_t)j.qb[k] * 2 * rn;
    cmax = cm > cmax ? cm : cmax;
    size_t ncol = imin(j.qb[k], (int)(2 * rn));
    size_t len = j.qb[k] > (int)(2 * rn) ? j.qb[k] : 2 * rn;
    // Jacobi matrices with 16-byte row strides (up to 16 / eb - 1 padding)
    const size_t pad = 16 / eb;
    jw = ncol * (len + pad) > jw ? ncol * (len + pad) : jw;
    jv = ncol * (ncol + pad) > jv ? ncol * (ncol + pad) : jv;
    // range-finder power step (n x l), then B (l x n) of the randomized step
    rz = (2 * rn + pad) * ncol > rz ? (2 * rn + pad) * ncol : rz;
    size_t u = (size_t)j.qb[k] * imin(j.chi, (int)ncol);
    us = u > us ? u : us;
    // C' = Q_{k-1} (2 q_{k-1} x q_k) * US: 2 q_{k-1} x r
    size_t c2 = (size_t)(k > 0 ? j.qb[k - 1] : 1) * 2 * imin(j.chi, (int)ncol);
    cmax = c2 > cmax ? c2 : cmax;
  }
  j.lay.w_off = al(wmax);
  j.lay.m_off = al(mmax);
  j.lay.r_off = al(rmax > 1 ? rmax : 1);
  j.lay.c_off = al(cmax);
  j.lay.jw_off = al(jw);
  j.lay.jv_off = al(jv);
  j.lay.us_off = al(us);
  j.lay.rz_off = al(rz);
  j.lay.qw_off = al(qw);
  if (eb == 8) {
    j.lay.jw64_off = j.lay.jw_off;                 // the FP64 Jacobi matrices are the Jacobi matrices
    j.lay.jv64_off = j.lay.jv_off;
  } else if (j.svd64) {
    size_t w64 = 0, v64 = 0;                       // doubles, in units of T (two floats each)
    for (int k = 0; k < L; ++k) {
      const int rn = imin(j.chi, j.qb[k + 1]);
      const int ncol = imin(j.qb[k], 2 * rn), len = imax(j.qb[k], 2 * rn);
      w64 = std::max(w64, (size_t)ncol * jacobi_ld<double>(len));
      v64 = std::max(v64, (size_t)ncol * jacobi_ld<double>(ncol));
    }
    j.lay.jw64_off = al(2 * w64);
    j.lay.jv64_off = al(2 * v64);
  } else {
    j.lay.jw64_off = j.lay.jv64_off = 0;
  }
  if (j.refine) {
    size_t lg = 0, j32 = 0, vb = 0;                // float pairs, floats, doubles
    for (int k = 0; k < L; ++k) {
      const int ncol = imin(j.qb[k], 2 * imin(j.chi, j.qb[k + 1]));
      lg = std::max(lg, jacobi_reg_log_sweep(imin(ncol, 128)));
      j32 = std::max(j32, (size_t)ncol * jacobi_ld<float>(ncol));
      vb = std::max(vb, (size_t)ncol * jacobi_ld<double>(ncol) + ncol);
    }
    const size_t fpe = eb / 4;                     // floats per element
    j.lay.log_off = al(2 * lg * JR_LOG_SWEEPS / fpe);
    j.lay.j32_off = al((j32 + fpe - 1) / fpe);
    j.lay.vb64_off = al((2 * vb + CL_MAX * 8) / fpe);
    size_t wide = 0;                               // floats
    for (int k = 0; k < L; ++k) {
      const int rn = imin(j.chi, j.qb[k + 1]);
      const int ncol = imin(j.qb[k], 2 * rn), len = imax(j.qb[k], 2 * rn);
      if (!jacobi_reg_fits(ncol, len)) wide = std::max(wide, jacobi_wide_floats(ncol, len));
    }
    j.lay.wide_off = al((wide + fpe - 1) / fpe);
  }
  j.lay.total = off;
}

// ---------------------------------------------------------------- device helpers
__device__ inline void flag(int* st, int code) { atomicOr(st, code); }

template <typename T>
__device__ inline const T* core_ptr(const MpsRef& m, int L, int k) {
  return (const T*)m.base + core_offset(L, m.cap, k);
}

// Input index s of the shift MPO block (w, s_out, w') at site k, or -1 (zero).
// 1-D cores (Sec. 2.5): first [I X], middle [[I j],[0 j']], last [j; j'],
// X = P (cyclic) or j (non-cyclic); (j, j') = (J, J') for offset +1, swapped for -1.
// Non-axis sites carry the identity and pass the bond through.
__device__ inline int shift_src(const Term& t, int n_bits, int k, int w, int so, int w2) {
  if (k % 3 != t.axis) return (w == w2) ? so : -1;             // identity padding
  const int lev = k / 3;
  // 2x2 blocks as functions out -> in: I: s; J: out0<-in1; J': out1<-in0; P: 1-s
  const int jJ = (t.offset == 1) ? 0 : 1;   // 0: j = J, 1: j = J'
  auto blockJ = [&](int which) -> int {     // which 0 = j, 1 = j'
    int isJ = (which == 0) ? (jJ == 0) : (jJ == 1);
    if (isJ) return so == 0 ? 1 : -1;      // J: (0,1)
    return so == 1 ? 0 : -1;               // J': (1,0)
  };
  if (n_bits == 1) {                        // single 2x2 operator
    if (t.cyclic) return 1 - so;
    return blockJ(0);
  }
  if (lev == 0) {                           // [I  X], 1 x 2
    if (w2 == 0) return so;
    if (t.cyclic) return 1 - so;
    return blockJ(0);
  }
  if (lev == n_bits - 1) {                  // [j; j'], 2 x 1
    return blockJ(w == 0 ? 0 : 1);
  }
  if (w == 0 && w2 == 0) return so;         // [[I j],[0 j']]
  if (w == 0 && w2 == 1) return blockJ(0);
  if (w == 1 && w2 == 1) return blockJ(1);
  return -1;
}

__device__ inline int shift_w(const Term& t, int n_bits, int k) {   // MPO bond at bond k
  int first = t.axis, last = t.axis + 3 * (n_bits - 1);
  return (k > first && k <= last) ? 2 : 1;
}

__device__ inline int term_bond(const Term& t, int n_bits, int k) {
  switch (t.kind) {
    case T_ONES: return 1;
    case T_PLAIN:
    case T_MASK1: return t.x.ranks[k];
    case T_KRON: return t.x.ranks[k] * t.y.ranks[k];
    case T_SHIFT: return shift_w(t, n_bits, k) * t.x.ranks[k];
  }
  return 0;
}

// element (i, s, j) of term t's core k (coefficient not applied)
template <typename T>
__device__ inline T term_elem(const Term& t, int L, int n_bits, int k, int i, int s, int j,
                              const T* masks) {
  switch (t.kind) {
    case T_ONES: return (T)1;
    case T_PLAIN: {
      const int r1 = t.x.ranks[k + 1];
      return core_ptr<T>(t.x, L, k)[((size_t)i * 2 + s) * r1 + j];
    }
    case T_MASK1: {
      const int r1 = t.x.ranks[k + 1];
      return core_ptr<T>(t.x, L, k)[((size_t)i * 2 + s) * r1 + j] *
             masks[((size_t)t.mask_id * TN_MAXL + k) * 2 + s];
    }
    case T_KRON: {
      const int rb = t.y.ranks[k], rb1 = t.y.ranks[k + 1], ra1 = t.x.ranks[k + 1];
      const int a = i / rb, b = i % rb, a1 = j / rb1, b1 = j % rb1;
      return core_ptr<T>(t.x, L, k)[((size_t)a * 2 + s) * ra1 + a1] *
             core_ptr<T>(t.y, L, k)[((size_t)b * 2 + s) * rb1 + b1];
    }
    case T_SHIFT: {
      const int ra = t.x.ranks[k], ra1 = t.x.ranks[k + 1];
      const int w = i / ra, a = i % ra, w2 = j / ra1, a1 = j % ra1;
      const int si = shift_src(t, n_bits, k, w, s, w2);
      if (si < 0) return (T)0;
      return core_ptr<T>(t.x, L, k)[((size_t)a * 2 + si) * ra1 + a1];
    }
  }
  return (T)0;
}

// ---------------------------------------------------------------- the kernel
// Shared memory map (bytes): [0,16K) bond bookkeeping; then 32 doubles of
// reduction scratch, tau[MAXK], sig[MAXK] (doubles), wv[MAXK] (T); the rest is
// the work area holding the QR panel (left sweep) or the Jacobi pair W, V
// (right sweep) whenever they fit.
static constexpr int SM_RED = 16 * 1024;
static constexpr int SM_TAU = SM_RED + 256;
static constexpr int SM_SIG = SM_TAU + (MAXK + 8) * 8;   // tau also holds tails at [2, MAXK+2)
static constexpr int SM_WV = SM_SIG + MAXK * 8;
static_assert(SM_WV + MAXK * 8 <= SM_SMALL, "bookkeeping overlaps the work area");
static_assert(16 * 1024 >= (2 * TN_MAXT * (TN_MAXL + 1) + TN_MAXT + 2 * (TN_MAXL + 1) + MAXK) * 4, "bond tables");

// phase timer of thread 0 (profiling only)
// Phase timers and counters of thread 0, kept in shared memory so that they
// hold no registers across the kernel (slots: PH_*).
struct PhaseClock {
  long long t0 = 0;
  double* acc;
  bool on;
  __device__ PhaseClock(bool enable, double* sh) : acc(sh), on(enable && threadIdx.x == 0) {
    if (on) {
      for (int p = 0; p < PH_COUNT; ++p) acc[p] = 0.0;
      t0 = clock64();
    }
  }
  __device__ void lap(int ph) {
    if (!on) return;
    const long long t = clock64();
    acc[ph] += (double)(t - t0);
    t0 = t;
  }
};

// Lap timer of the cluster Jacobi's sub-phases (thread 0 of the leader CTA;
// acc null elsewhere).
struct RxClock {
  double* acc;
  long long t0;
  __device__ explicit RxClock(double* a) : acc(threadIdx.x == 0 ? a : nullptr), t0(0) {
    if (acc) t0 = clock64();
  }
  __device__ void lap(int ph) {
    if (!acc) return;
    const long long t = clock64();
    acc[ph] += (double)(t - t0);
    t0 = t;
  }
};

// ---------------------------------------------------------------- row-partitioned FP64 SVD
template <typename S>
__device__ __forceinline__ S fmx(S a, S b, S c) {
  if constexpr (sizeof(S) == 8) return fma(a, b, c);
  else return fmaf(a, b, c);
}

// Sum of n values x[0], x[s], x[2s], ... in a fixed order with four
// independent accumulators; the same inputs give the same result in every CTA.
template <typename S>
__device__ __forceinline__ S sum4(const S* x, int n, int s) {
  S a0 = 0, a1 = 0, a2 = 0, a3 = 0;
  int c = 0;
  for (; c + 3 < n; c += 4) {
    a0 += x[(size_t)c * s];
    a1 += x[(size_t)(c + 1) * s];
    a2 += x[(size_t)(c + 2) * s];
    a3 += x[(size_t)(c + 3) * s];
  }
  for (; c < n; ++c) a0 += x[(size_t)c * s];
  return (a0 + a1) + (a2 + a3);
}

// Column norms of the S-typed rows Wl over the cluster, in S arithmetic:
// every CTA sums its rows, sends the partial sums to every CTA, and every CTA
// adds them in rank order (the same values in every CTA).  Ends with nrm[]
// valid everywhere.
template <typename S>
__device__ inline void rows_norms(ClusterCtx& cc, const RowsLayout& R, unsigned char* wa, const S* Wl, int ncol,
                                  int li) {
  S* nb = (S*)(wa + R.nbuf);
  S* nrm = (S*)(wa + R.nrm);
  S* loc = (S*)(wa + R.gl);
  cl_xchg_expect(cc, (unsigned)(ncol * cc.P * sizeof(S)));
  for (int j = threadIdx.x; j < ncol; j += blockDim.x) {
    const S* w = Wl + (size_t)j * R.lw;
    S v0 = 0, v1 = 0, v2 = 0, v3 = 0;
    int ii = 0;
    for (; ii + 3 < li; ii += 4) {
      v0 = fmx(w[ii], w[ii], v0);
      v1 = fmx(w[ii + 1], w[ii + 1], v1);
      v2 = fmx(w[ii + 2], w[ii + 2], v2);
      v3 = fmx(w[ii + 3], w[ii + 3], v3);
    }
    for (; ii < li; ++ii) v0 = fmx(w[ii], w[ii], v0);
    const S v = (v0 + v1) + (v2 + v3);
    if (cc.P == 1) nb[j] = v;
    else loc[j] = v;
  }
  // stores into the other CTAs follow the last exchange by at most a round,
  // far less than a CTA that gave up waits at the exit barrier
  if (cc.P > 1) {
    __syncthreads();
    if (!cc.dead)
      for (int idx = threadIdx.x; idx < ncol * cc.P; idx += blockDim.x) {
        const int j = idx / cc.P, d = idx % cc.P;
        cl_xchg_send(cc, nb + (size_t)j * cc.P + cc.rank, d, loc[j]);
      }
  }
  cl_xchg_wait(cc);
  for (int j = threadIdx.x; j < ncol; j += blockDim.x) nrm[j] = sum4<S>(nb + (size_t)j * cc.P, cc.P, 1);
  __syncthreads();
}

// This CTA's parts of the inner products of the pairs of round rnd (S sums;
// four lanes per pair, so that the FP64 work of a round is spread over four
// warps), sent to every CTA's exchange slots xq[p][rank]; then the wait for
// the other CTAs' parts.
template <typename S>
__device__ inline bool rows_pair_dots(ClusterCtx& cc, const RowsLayout& R, unsigned char* wa, const S* Wl,
                                      S* xq, int rnd, int np, int ncol, int li, RxClock& rx) {
  const int npairs = np / 2;
  S* loc = (S*)(wa + R.gl);
  cl_xchg_expect(cc, (unsigned)(npairs * cc.P * sizeof(S)));
  for (int t = threadIdx.x; t < npairs * 4; t += blockDim.x) {
    const int p = t >> 2, q = t & 3;
    const unsigned grp = 0xfu << (threadIdx.x & 28);
    int a, b;
    rr_pair(rnd, p, np, a, b);
    S g0 = 0, g1 = 0;
    if (b < ncol) {
      const S* x = Wl + (size_t)a * R.lw;
      const S* y = Wl + (size_t)b * R.lw;
      int ii = q;
      for (; ii + 4 < li; ii += 8) {
        g0 = fmx(x[ii], y[ii], g0);
        g1 = fmx(x[ii + 4], y[ii + 4], g1);
      }
      if (ii < li) g0 = fmx(x[ii], y[ii], g0);
    }
    S g = g0 + g1;
    g += __shfl_xor_sync(grp, g, 1, 4);
    g += __shfl_xor_sync(grp, g, 2, 4);
    if (q == 0) {
      if (cc.P == 1) xq[p] = g;
      else loc[p] = g;
    }
  }
  if (cc.P > 1) {
    __syncthreads();
    if (!cc.dead)
      for (int idx = threadIdx.x; idx < npairs * cc.P; idx += blockDim.x) {
        const int p = idx / cc.P, d = idx % cc.P;
        cl_xchg_send(cc, xq + (size_t)p * cc.P + cc.rank, d, loc[p]);
      }
  }
  rx.lap(PH_RX_DOT);
  const bool ok = cl_xchg_wait(cc);
  rx.lap(PH_RX_WAIT);
  return ok;
}

// (c, s) of FP32 values renormalised in FP64: (c, s) (1 + d)^(-1/2) with
// d = c^2 + s^2 - 1 (exact in FP64: the squares have 48 bits) and the series
// to d^2 (error O(d^3) ~ 1e-20): orthogonal to FP64 rounding.
__device__ __forceinline__ void renorm64(float cf, float sf, double& c, double& s) {
  const double c0 = (double)cf, s0 = (double)sf;
  const double dr = fma(c0, c0, s0 * s0) - 1.0;
  const double h = fma(dr, fma(0.375, dr, -0.5), 1.0);
  c = c0 * h;
  s = s0 * h;
}

// Rotation of a pair with norms al, be and inner product g (exchanged FP64
// values, identical in every CTA): false if the pair counts as orthogonal
// (g^2 <= tol2 al be) or a column is negligible.  t = tan(theta) is
// Rutishauser's root of the FP32 quotient zeta = (be - al) / (2 g) of the
// FP64 difference (a quotient outside the FP32 range is formed in FP64, with
// t = 1 / (2 zeta) once |zeta| > 1e18).  (c, s) = (1, t) (1 + t^2)^(-1/2)
// orthogonal to FP64 rounding: for |t| < 2^-14 by the series c = 1 - t^2/2,
// s = t c; else the FP32 (c, s) renormalised in FP64 (renorm64).  The new
// norms are al - t g and be + t g (exact for the exact root; recomputed every
// sweep); rel2 = g^2 / (al be) and tan = |t| for the stopping rule.
// A warp's FP64 instruction takes 64 cycles of its scheduler (0.5 lanes a clock), and a
// round waits for this chain: 30 of them took 4 k of a round's 9 k cycles.  So where al, be
// and g are within 2^+-100 and al, be within 2^100 of each other, the test and the quotient
// are FP32, conversions of normal numbers move bits, and ten FP64 instructions are left:
// 4.0 k -> 3.2 k cycles.
__device__ __forceinline__ float narrow_bits(double x) {    // |x| in 2^+-126, truncated
  const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
  return __uint_as_float((h & 0x80000000u) | (((h & 0x7fffffffu) - 0x38000000u) << 3) | (l >> 29));
}
__device__ __forceinline__ double widen_bits(float x) {     // a normal number
  const unsigned u = __float_as_uint(x);
  return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(u << 29));
}
__device__ __forceinline__ bool rows_angle(double al, double be, double g, double tol2, double& cw, double& sw,
                                           double& na, double& nb, float& rel2, float& tan) {
  const int xa = __double2hiint(al) >> 20, xb = __double2hiint(be) >> 20, xg = (__double2hiint(g) >> 20) & 0x7ff;
  if (xa > 923 && xa < 1123 && xb > 923 && xb < 1123 && xg > 923 && xg < 1123 && xa - xb < 100 && xb - xa < 100) {
    const float gf = narrow_bits(g);
    const float cs = fabsf(gf) * (rsqrtf(narrow_bits(al)) * rsqrtf(narrow_bits(be)));
    if (!(cs > sqrtf((float)tol2))) return false;
    rel2 = cs * cs;
    const float z = (float)(be - al) / (2.f * gf), az = fabsf(z);
    const float tf = copysignf(az > 1e18f ? 0.5f / az : 1.f / (az + sqrtf(fmaf(z, z, 1.f))), z);
    const double t = widen_bits(tf);                        // at least 2^-100: normal
    tan = fabsf(tf);
    if (fabsf(tf) < 6.1035156e-05f) {
      cw = fma(-0.5 * t, t, 1.0);                           // c^2 + s^2 = 1 - 3 t^4 / 4 + ...
      sw = t * cw;
    } else {
      const float cf = rsqrtf(fmaf(tf, tf, 1.f));
      const double c0 = widen_bits(cf), s0 = widen_bits(cf * tf);
      const double dr = fma(c0, c0, fma(s0, s0, -1.0)), h = fma(dr, fma(0.375, dr, -0.5), 1.0);
      cw = c0 * h;
      sw = s0 * h;
    }
    na = fma(-t, g, al);
    nb = fma(t, g, be);
    return true;
  }
  const double gg = g * g, ab = al * be;
  if (g == 0.0 || !(al > 1e-250) || !(be > 1e-250) || gg <= tol2 * ab) return false;
  rel2 = (float)gg / (float)ab;                         // +inf if al be leaves the FP32 range
  const double d = be - al;
  float tf = 0.f;
  double t;
  bool tiny = false;
  if (fabs(d) > 1e18 * fabs(g) || fabs(g) < 1e-30) {
    const double zd = d / (2.0 * g);                    // outside the FP32 range: FP64 (rare)
    if (fabs(zd) > 1e18) {
      t = 0.5 / zd;
      tiny = true;
    } else {
      const float z = (float)zd;
      tf = copysignf(1.f / (fabsf(z) + sqrtf(fmaf(z, z, 1.f))), z);
      t = (double)tf;
    }
  } else {
    const float z = (float)d / (2.f * (float)g);
    tf = copysignf(1.f / (fabsf(z) + sqrtf(fmaf(z, z, 1.f))), z);
    t = (double)tf;
  }
  tan = fabsf((float)t);
  if (tiny) {
    cw = 1.0;                                           // 1 + t^2 rounds to 1 for |t| < 1e-18
    sw = t;
  } else if (fabsf(tf) < 6.1035156e-05f) {
    // c^2 + s^2 = 1 - 3 t^4 / 4 + ...: orthogonal to FP64 rounding
    const double c = fma(-0.5 * t, t, 1.0);
    cw = c;
    sw = t * c;
  } else {
    const float cf = rsqrtf(fmaf(tf, tf, 1.f)), sf = cf * tf;
    renorm64(cf, sf, cw, sw);
  }
  na = al - t * g;
  nb = be + t * g;
  return true;
}

// Cyclic one-sided Jacobi sweeps (round-robin order) on the cluster's FP64
// rows of W and V; nrot counts rotations.  Per round: each CTA's parts of the
// pair inner products go to every CTA, four lanes per pair add them in rank
// order, lane 0 takes the angle, and every CTA rotates its rows of W and V.
// Stopping rule: a sweep that rotates nothing (every pair within the tolerance), or a
// sweep whose cosines c and tangents t were small: c below 5e-9 and the largest c times the
// largest t below a tenth of the tolerance.  A rotation turns t c of its columns' cosines
// with others onto one another, so that is what a sweep leaves (and the FP32 angle's residual
// 1.2e-7 x 5e-9, under the tolerance 16 eps_64 sqrt(len) >= 5e-15), and the confirming
// sweep is skipped.  Columns of close singular values turn far on small cosines: with c alone,
// eight of them 1e-9 apart kept cosines of up to 9e-10 after a refinement.  Every CTA sees the
// same values, so every CTA stops at the same sweep.  Returns the sweeps used; *converged
// tells whether the rule was met within maxsw sweeps.
template <typename S>
__device__ __noinline__ int rows_sweeps(ClusterCtx& cc_, const RowsLayout& R_, unsigned char* wa, S* Wl, double* Vl, int ncol,
                           int li, int vi, int maxsw, S tol2, unsigned* nrot, double* phase_acc, bool* converged,
                           int* rounds_out = nullptr) {
  static_assert(sizeof(S) == 8, "the cluster sweeps run on FP64 rows");
  // in registers: behind the references they are in local memory, read again in each of
  // the exchanges that a round is made of
  ClusterCtx cc = cc_;
  const RowsLayout R = R_;
  __shared__ float s_mrel[32], s_mtan[32];
  RxClock rx(phase_acc);
  unsigned q = 0;                                  // rounds so far (exchange buffer parity)
  S* nrm = (S*)(wa + R.nrm);
  S* xb = (S*)(wa + R.xb);
  S* pcw = (S*)(wa + R.pcw);
  S* psw = (S*)(wa + R.psw);
  int* pfl = (int*)(wa + R.pf);
  const int np = (ncol + 1) & ~1, npairs = np / 2;
  int sweep = 0, rounds = 0;
  *converged = true;
  if (ncol < 2) return 0;
  *converged = false;
  // rotation of this CTA's rows of V by round rnd's pairs
  auto rotate_v = [&](int rnd) {
    for (int idx = threadIdx.x; idx < npairs * vi; idx += blockDim.x) {
      const int p = idx / vi, ii = idx - p * vi;
      if (!pfl[p]) continue;
      int a, b;
      rr_pair(rnd, p, np, a, b);
      const double cs = pcw[p], sn = psw[p];
      double* pa = Vl + (size_t)a * R.lv + ii;
      double* pb = Vl + (size_t)b * R.lv + ii;
      const double u = *pa, w = *pb;
      *pa = cs * u - sn * w;
      *pb = sn * u + cs * w;
    }
  };
  for (; sweep < maxsw; ++sweep) {
    rows_norms<S>(cc, R, wa, Wl, ncol, li);
    rx.lap(PH_RX_NORM);
    int any = 0;
    float mrel = 0.f, mtan = 0.f;                  // largest g^2 / (al be) and |t| this thread rotated this sweep
    bool ok = rows_pair_dots<S>(cc, R, wa, Wl, xb + (size_t)(q & 1) * npairs * cc.P, 0, np, ncol, li, rx);
    for (int rnd = 0; rnd < np - 1 && ok; ++rnd, ++q) {
      const S* xq = xb + (size_t)(q & 1) * npairs * cc.P;
      ++rounds;
      int rot = 0;
      for (int t = threadIdx.x; t < npairs * 4; t += blockDim.x) {
        const int p = t >> 2, l = t & 3;
        const unsigned grp = 0xfu << (threadIdx.x & 28);
        // the partials of pair p in rank order: lane l adds ranks l, l+4, ...,
        // then the four lanes combine (the same order in every CTA)
        S g = 0;
        if (cc.P == 1) {
          g = xq[p];
        } else {
          for (int c = l; c < cc.P; c += 4) g += xq[(size_t)p * cc.P + c];
          g += __shfl_xor_sync(grp, g, 1, 4);
          g += __shfl_xor_sync(grp, g, 2, 4);
        }
        if (l != 0) continue;
        int a, b;
        rr_pair(rnd, p, np, a, b);
        int go = 0;
        if (b < ncol) {
          S cw, sw, na, nb;
          float rel2 = 0.f, tan = 0.f;
          if (rows_angle(nrm[a], nrm[b], g, tol2, cw, sw, na, nb, rel2, tan)) {
            mrel = fmaxf(mrel, rel2);
            mtan = fmaxf(mtan, tan);
            nrm[a] = na;
            nrm[b] = nb;
            pcw[p] = cw;
            psw[p] = sw;
            go = 1;
            atomicAdd(nrot, 1u);
          }
        }
        pfl[p] = go;
        rot |= go;
      }
      any |= __syncthreads_or(rot);
      rx.lap(PH_RX_ANGLE);
      // the rotations of W, one element pair per thread
      for (int idx = threadIdx.x; idx < npairs * li; idx += blockDim.x) {
        const int p = idx / li, ii = idx - p * li;
        if (!pfl[p]) continue;
        int a, b;
        rr_pair(rnd, p, np, a, b);
        const S cs = pcw[p], sn = psw[p];
        S* pa = Wl + (size_t)a * R.lw + ii;
        S* pb = Wl + (size_t)b * R.lw + ii;
        const S u = *pa, w = *pb;
        *pa = cs * u - sn * w;
        *pb = sn * u + cs * w;
      }
      rotate_v(rnd);
      __syncthreads();
      rx.lap(PH_RX_ROT);
      if (rnd + 1 < np - 1)
        ok = rows_pair_dots<S>(cc, R, wa, Wl, xb + (size_t)((q + 1) & 1) * npairs * cc.P, rnd + 1, np, ncol, li,
                               rx);
    }
    if (cc.dead) break;
    if (!any) { *converged = true; break; }
    // the sweep's largest cosine (squared) and tangent (the same in every CTA)
    for (int o = 16; o > 0; o >>= 1) {
      mrel = fmaxf(mrel, __shfl_xor_sync(0xffffffffu, mrel, o));
      mtan = fmaxf(mtan, __shfl_xor_sync(0xffffffffu, mtan, o));
    }
    if ((threadIdx.x & 31) == 0) { s_mrel[threadIdx.x >> 5] = mrel; s_mtan[threadIdx.x >> 5] = mtan; }
    __syncthreads();
    float m = 0.f, mt = 0.f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) { m = fmaxf(m, s_mrel[w]); mt = fmaxf(mt, s_mtan[w]); }
    __syncthreads();
    if (m < 2.5e-17f && sqrtf(m) * mt < 0.1f * sqrtf((float)tol2)) { *converged = true; ++sweep; break; }
  }
  if (phase_acc && threadIdx.x == 0) phase_acc[PH_ROUNDS64] += rounds;
  if (rounds_out) *rounds_out = rounds;
  cc_ = cc;
  if (cc.dead) { *converged = false; return maxsw; }
  return sweep;
}

// Stage rows [k0, k0 + nk) of every column of the ncol x ncol matrix V
// (global, column c at V + c * ld, type S) in shared memory as doubles:
// st[c * kc + kk] = V(k0 + kk, c).
template <typename S>
__device__ inline void stage_rows(const S* V, int ld, int ncol, int k0, int nk, int kc, double* st) {
  for (int idx = threadIdx.x; idx < ncol * nk; idx += blockDim.x) {
    const int c = idx / nk, kk = idx - c * nk;
    st[(size_t)c * kc + kk] = rf_d(__ldcg(V + (size_t)c * ld + k0 + kk));
  }
}

// One Newton-Schulz step towards the orthogonal polar factor, in FP64, on
// this CTA's block of columns J = [v0, v0 + vi): G(:, J) = V0^T V0(:, J),
// V1(:, J) = V0 (3/2 I - 1/2 G)(:, J).  V0 (type S, ld0) and V1 (FP64, ld1)
// are global; V0 is read in staged row chunks.  With V0^T V0 = I + E the
// step leaves V1^T V1 = I + O(E^2) (3/4 E^2 to second order).
template <typename S>
__device__ inline void rows_ns_step(const RowsLayout& R, unsigned char* wa, const S* V0, int ld0, double* V1,
                                    int ld1, int ncol, int v0, int vi) {
  double* G = (double*)(wa + R.gb);                      // G[jj * ncol + i] = G(i, v0 + jj)
  double* st = (double*)(wa + R.st);
  const int kc = R.kc;
  for (int idx = threadIdx.x; idx < ncol * vi; idx += blockDim.x) G[idx] = 0.0;
  for (int k0 = 0; k0 < ncol; k0 += kc) {
    const int nk = imin(kc, ncol - k0);
    __syncthreads();
    stage_rows<S>(V0, ld0, ncol, k0, nk, kc, st);
    __syncthreads();
    for (int idx = threadIdx.x; idx < ncol * vi; idx += blockDim.x) {
      const int jj = idx / ncol, i = idx - jj * ncol;
      const double* x = st + (size_t)i * kc;
      const double* y = st + (size_t)(v0 + jj) * kc;
      double a0 = 0.0, a1 = 0.0;
      int kk = 0;
      for (; kk + 1 < nk; kk += 2) {
        a0 = fma(x[kk], y[kk], a0);
        a1 = fma(x[kk + 1], y[kk + 1], a1);
      }
      if (kk < nk) a0 = fma(x[kk], y[kk], a0);
      G[idx] += a0 + a1;
    }
  }
  __syncthreads();
  for (int idx = threadIdx.x; idx < ncol * vi; idx += blockDim.x) {
    const int jj = idx / ncol, i = idx - jj * ncol;
    G[idx] = (i == v0 + jj ? 1.5 : 0.0) - 0.5 * G[idx];  // H = 3/2 I - 1/2 G
  }
  for (int k0 = 0; k0 < ncol; k0 += kc) {
    const int nk = imin(kc, ncol - k0);
    __syncthreads();
    stage_rows<S>(V0, ld0, ncol, k0, nk, kc, st);
    __syncthreads();
    for (int idx = threadIdx.x; idx < nk * vi; idx += blockDim.x) {
      const int jj = idx / nk, kk = idx - jj * nk;
      const double* h = G + (size_t)jj * ncol;
      double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
      int i = 0;
      for (; i + 3 < ncol; i += 4) {
        a0 = fma(st[(size_t)i * kc + kk], h[i], a0);
        a1 = fma(st[(size_t)(i + 1) * kc + kk], h[i + 1], a1);
        a2 = fma(st[(size_t)(i + 2) * kc + kk], h[i + 2], a2);
        a3 = fma(st[(size_t)(i + 3) * kc + kk], h[i + 3], a3);
      }
      for (; i < ncol; ++i) a0 = fma(st[(size_t)i * kc + kk], h[i], a0);
      __stcg(V1 + (size_t)(v0 + jj) * ld1 + k0 + kk, (a0 + a1) + (a2 + a3));
    }
  }
  __syncthreads();
}

// W = X V for this CTA's rows (FP64): X(i, k) = scl C(i, k) (C^T when the
// Jacobi runs on the columns of C^T) for the rows [i0, i0 + li), read from
// the job's scratch, and V (ncol x ncol, FP64, column c at V + c * ld), both
// staged in chunks of kc indices k.
template <typename T, typename N>
__device__ inline void rows_xv(const RowsLayout& R, unsigned char* wa, const T* C, int n, bool trans, double scl,
                               int i0, int li, const N* V, int ld, double* W, int ncol) {
  double* st = (double*)(wa + R.st);
  double* xs = (double*)(wa + R.xs);                      // xs[kk * li + ii] = X(i0 + ii, k0 + kk)
  const int kc = R.kc;
  for (int idx = threadIdx.x; idx < ncol * li; idx += blockDim.x) W[(size_t)(idx / li) * R.lw + idx % li] = 0.0;
  for (int k0 = 0; k0 < ncol; k0 += kc) {
    const int nk = imin(kc, ncol - k0);
    __syncthreads();
    stage_rows<N>(V, ld, ncol, k0, nk, kc, st);
    for (int idx = threadIdx.x; idx < nk * li; idx += blockDim.x) {
      const int kk = idx / li, ii = idx - kk * li, i = i0 + ii, k = k0 + kk;
      xs[idx] = scl * (double)__ldcg(trans ? C + (size_t)i * n + k : C + (size_t)k * n + i);
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < ncol * li; idx += blockDim.x) {
      const int j = idx / li, ii = idx - j * li;
      const double* v = st + (size_t)j * kc;
      double a0 = 0.0, a1 = 0.0;
      int kk = 0;
      for (; kk + 1 < nk; kk += 2) {
        a0 = fma(xs[kk * li + ii], v[kk], a0);
        a1 = fma(xs[(kk + 1) * li + ii], v[kk + 1], a1);
      }
      if (kk < nk) a0 = fma(xs[kk * li + ii], v[kk], a0);
      W[(size_t)j * R.lw + ii] += a0 + a1;
    }
  }
  __syncthreads();
}

// FP64 one-sided Jacobi SVD of the centre matrix C (m x n, T, global) with the
// rows of the Jacobi matrices split over the CTAs of the cluster and held in
// shared memory.  X = the columns of C (n <= m) or of C^T, scaled by scl;
// V accumulates the rotations (FP64).  CTA c owns entries
// [c len / P, (c+1) len / P) of every column of W and [c ncol / P,
// (c+1) ncol / P) of every column of V.  Every CTA sums the exchanged parts
// in the same order, so every CTA takes the same rotations.
// The start, by sw32:
// >= 0: the leader has run FP32 sweeps on X alone and logged their rotations; every
//   CTA forms its rows of their product V0 from the log, and rf_refine takes V0 to an
//   orthonormal V with W = X V and orthogonal columns, to 48 (FP32 data) or 53 bits;
//   the FP64 sweeps run only where it could not finish, from the V it reached;
// SW_WIDE: the same with FP32 sweeps over the cluster, V along (jacobi_wide), where X
//   does not fit one CTA's registers;
// SW_SCRATCH (FP32 data beyond that too): the leader's V0 is in the job's scratch;
//   one FP64 Newton-Schulz step, spread over the CTAs by blocks of columns, makes it
//   orthogonal to ~1e-12, W = X V is formed in FP64 and the FP64 sweeps finish;
// SW_PLAIN: FP64 sweeps from W = X, V = I.
// Column norms are recomputed exactly at the start of every sweep and at the end.
// Every CTA then finds the same singular values, order and kept rank (the rank rule
// of Eq.
// svd-move with delta) and writes its rows of core k (V^T[:r], r x n) and of
// U S (m x r).  Called by all threads of every CTA with equal arguments;
// returns the kept rank (0 if it exceeds the bond capacity), the FP64
// sweeps, whether their limit was reached, and the FP64 FLOPs executed.
template <typename T>
__device__ __noinline__ int svd64_rows(ClusterCtx& cc, const RoundJob& J, int L, int k, int m, int n, double scl, double delta,
                          int maxsw, int sw32, int* sweeps_out, bool* noconv, double* exec_flops = nullptr,
                          double* phase_acc = nullptr) {
  constexpr bool two_phase = sizeof(T) == 4;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ unsigned s_nrot;
  if (threadIdx.x == 0) s_nrot = 0;
  unsigned char* wa = smem + SM_SMALL;
  T* scr = (T*)J.scratch;
  const T* C = scr + J.lay.c_off;
  T* US = scr + J.lay.us_off;
  T* out = (T*)J.dst.base + core_offset(L, J.dst.cap, k);
  const int ncol = imin(m, n), len = imax(m, n);
  const bool trans = (n <= m);
  const RowsLayout R = rows_layout(ncol, len, cc.P, rows_stage(sizeof(T), sw32));
  double* Wl = (double*)(wa + R.wl);
  double* Vl = (double*)(wa + R.vl);
  double* nrm = (double*)(wa + R.nrm);
  double* sig = (double*)(wa + R.sig);
  int* perm = (int*)(wa + R.perm);
  double* tail = (double*)(wa + R.tail);
  const int i0 = cc.rank * len / cc.P, li = (cc.rank + 1) * len / cc.P - i0;
  const int v0 = cc.rank * ncol / cc.P, vi = (cc.rank + 1) * ncol / cc.P - v0;
  double* W = Wl;
  const double tol64 = 16.0 * 2.220446049250313e-16 * sqrt((double)len);
  auto xat = [&](int i, int kk) -> double { return scl * (double)__ldcg(trans ? C + (size_t)i * n + kk : C + (size_t)kk * n + i); };
  const int ld1 = jacobi_ld<double>(ncol);
  int state = RF_SWEEPS;
  bool tied = false;
  // squared norms relative to the largest below which a refined W is rounding only
  constexpr float low = two_phase ? 1e-22f : 1e-27f;
  if (sw32 >= 0 || sw32 == SW_WIDE) {
    // start from FP32 sweeps, refine by products
    const bool wide = sw32 == SW_WIDE;
    const int ldw32 = wide ? jacobi_wide_ldw(len) : jacobi_reg_ld(len);
    float* Wg = (float*)(scr + J.lay.wide_off);
    float* Vg = Wg + (size_t)jacobi_wide_cols(ncol) * ldw32;
    // FP32 sweeps of x(i, j) over the cluster, Vg their product
    auto sweep_wide = [&](auto&& x) -> int {
      const int nc = 2 * jacobi_wide_ctas(cc.P) * jacobi_wide_block(ncol, cc.P);
      for (int j = cc.rank; j < nc; j += cc.P) {
        for (int i = threadIdx.x; i < ldw32; i += blockDim.x)
          __stcg(Wg + (size_t)j * ldw32 + i, j < ncol && i < len ? x(i, j) : 0.f);
        for (int i = threadIdx.x; i < JW_COLS; i += blockDim.x) __stcg(Vg + (size_t)j * JW_COLS + i, i == j && j < ncol ? 1.f : 0.f);
      }
      if (!cl_sync(cc)) return maxsw;
      return jacobi_wide(cc, Wg, Vg, ncol, len, imin(maxsw, JW_SWEEPS), (float*)wa);
    };
    const long long t0 = clock64();
    using N = typename std::conditional<two_phase, float2, double>::type;
    RefineMem<N> rm;
    rm.V = (N*)(scr + J.lay.jv64_off);
    rm.stat = (float*)(scr + J.lay.vb64_off);     // 16-byte aligned, then V2 and the norms
    rm.V2 = (N*)(rm.stat + CL_MAX * 8);
    rm.W = (N*)(scr + J.lay.jw64_off);
    rm.J = (float*)(scr + J.lay.j32_off);
    rm.ldv = ld1;
    rm.ldw = jacobi_ld<double>(len);
    rm.ldj = jacobi_ld<float>(ncol);
    rm.nrm = rm.V2 + (size_t)ncol * ld1;
    rm.log = (float2*)(scr + J.lay.log_off);
    rm.turn = 0;
    rm.tied = false;
    if (wide) {
      sw32 = sweep_wide([&](int i, int j) { return (float)xat(i, j); });
      for (int idx = threadIdx.x; idx < ncol * vi; idx += blockDim.x)
        __stcg(rm.V + (size_t)(v0 + idx / ncol) * ld1 + idx % ncol, rf_make<N>(__ldcg(Vg + (size_t)(v0 + idx / ncol) * JW_COLS + idx % ncol)));
    } else {
      jacobi_reg_apply(rm.log, sw32, ncol, v0, vi, rm.V, ld1, (float2*)wa);
    }
    cl_sync(cc);
    // one more FP32 Jacobi, of W: the leader's sweeps, their product over the cluster
    auto jacobi = [&]() -> bool {
      int sw = 0;
      if (wide) {
        sweep_wide([&](int i, int j) { return 1048576.f * rf_f(__ldcg(rm.W + (size_t)j * rm.ldw + i)); });
        for (int idx = threadIdx.x; idx < ncol * vi; idx += blockDim.x)
          __stcg(rm.J + (size_t)(v0 + idx / ncol) * rm.ldj + idx % ncol, __ldcg(Vg + (size_t)(v0 + idx / ncol) * JW_COLS + idx % ncol));
        return cl_sync(cc);
      }
      if (cc.rank == 0) {
        float* Wf = (float*)wa;
        const int ncp = jacobi_reg_cols(ncol);
        for (int idx = threadIdx.x; idx < ncp * ldw32; idx += blockDim.x) {
          const int jj = idx / ldw32, i = idx % ldw32;
          // 2^20: columns down to 1e-18 of the scale are above the Jacobi's floor
          Wf[idx] = jj < ncol && i < len ? 1048576.f * rf_f(__ldcg(rm.W + (size_t)jj * rm.ldw + i)) : 0.f;
        }
        __syncthreads();
        sw = jacobi_reg<true>(Wf, ncol, len, imin(maxsw, JR_LOG_SWEEPS), rm.log);
        if (cl_alive(cc) && threadIdx.x < (unsigned)cc.P) cl_store_remote(&cc.sh->cmd.sw32, threadIdx.x, sw);
      }
      if (!cl_sync(cc)) return false;
      sw = *(volatile int*)&cc.sh->cmd.sw32;
      __syncthreads();
      jacobi_reg_apply(rm.log, sw, ncol, v0, vi, rm.J, rm.ldj, (float2*)wa);
      return cl_sync(cc);
    };
    const T tscl = (T)scl;                        // exact: a power of two
    auto xn = [&](int i, int kk) -> N { return rf_make<N>(tscl * __ldcg(trans ? C + (size_t)i * n + kk : C + (size_t)kk * n + i)); };
    const bool own = !two_phase && J.refine != REFINE_TOP;
    // the sums of FP32 data carry 48 bits
    const float tol2r = (two_phase ? 256.f : 1.f) * (float)(tol64 * tol64);
    state = rf_refine<N>(cc, rm, ncol, len, sw32 < maxsw, xn, trans, trans, tol2r,
                         two_phase ? 2e-13f : own ? 4e-16f : 1e-16f, own, two_phase ? 2e-6f : 2e-9f, two_phase ? 1e-11f : 1e-14f,
                         two_phase ? 1e-22f : 1e-28f, SM_SMALL, SM_WORK, jacobi);
    const bool has_w = state == RF_DONE;          // rm.W V^T = X
    tied = rm.tied;
    if (state == RF_DONE && !trans) state = rf_polish<N>(cc, rm, ncol, len, low, tol2r, SM_SMALL, SM_WORK);
    if (phase_acc && threadIdx.x == 0) phase_acc[PH_NS] += (double)(clock64() - t0);
    const long long t1 = clock64();
    for (int idx = threadIdx.x; idx < ncol * vi; idx += blockDim.x) {
      const int j = idx / vi, ii = idx % vi;
      Vl[(size_t)j * R.lv + ii] = rf_d(__ldcg(rm.V + (size_t)j * ld1 + v0 + ii));
    }
    if (has_w) {
      for (int idx = threadIdx.x; idx < ncol * li; idx += blockDim.x) {
        const int j = idx / li, ii = idx % li;
        Wl[(size_t)j * R.lw + ii] = rf_d(__ldcg(rm.W + (size_t)j * rm.ldw + i0 + ii));
      }
      __syncthreads();
    } else {
      rows_xv(R, wa, C, n, trans, scl, i0, li, rm.V, ld1, W, ncol);
    }
    cl_sync(cc);                                  // the staging space is the exchange buffers' again
    if (phase_acc && threadIdx.x == 0) phase_acc[PH_XV] += (double)(clock64() - t1);
  } else if (two_phase && sw32 == SW_SCRATCH) {
    const long long t0 = clock64();
    float* V0 = (float*)(scr + J.lay.jv_off);
    const int ld0 = jacobi_ld<float>(ncol);
    double* V1 = (double*)(scr + J.lay.jv64_off);
    rows_ns_step(R, wa, V0, ld0, V1, ld1, ncol, v0, vi);
    cl_sync(cc);                                  // every block of V1 written (cluster-scope fence)
    if (phase_acc && threadIdx.x == 0) phase_acc[PH_NS] += (double)(clock64() - t0);
    const long long t1 = clock64();
    for (int idx = threadIdx.x; idx < ncol * vi; idx += blockDim.x) {
      const int j = idx / vi, ii = idx % vi;
      Vl[(size_t)j * R.lv + ii] = __ldcg(V1 + (size_t)j * ld1 + v0 + ii);
    }
    rows_xv(R, wa, C, n, trans, scl, i0, li, V1, ld1, W, ncol);
    cl_sync(cc);                                  // the staging space is the exchange buffers' again
    if (phase_acc && threadIdx.x == 0) phase_acc[PH_XV] += (double)(clock64() - t1);
  } else {
    // own rows of X (promoted, scaled by a power of two: exact)
    for (int idx = threadIdx.x; idx < ncol * li; idx += blockDim.x) {
      const int j = idx / li, ii = idx % li;
      Wl[(size_t)j * R.lw + ii] = xat(i0 + ii, j);
    }
    for (int idx = threadIdx.x; idx < ncol * vi; idx += blockDim.x) {
      const int j = idx / vi, ii = idx % vi;
      Vl[(size_t)j * R.lv + ii] = (j == v0 + ii) ? 1.0 : 0.0;
    }
    __syncthreads();
  }
  bool conv = state == RF_DONE;
  int rounds = 0, sw = 0;
  if (state != RF_DONE)
    sw = rows_sweeps<double>(cc, R, wa, W, Vl, ncol, li, vi, maxsw, tol64 * tol64, &s_nrot, phase_acc, &conv, &rounds);
  *sweeps_out = sw;
  *noconv = !conv || cc.dead;
  if (exec_flops && threadIdx.x == 0) {
    // over the whole cluster, FP64 only: 6 per rotated element pair of W and
    // V, 2 per element of every pair's inner product and of the norms; for
    // FP32 data the Newton-Schulz step (two ncol^3 products) and X V
    const int np = (ncol + 1) & ~1, npairs = np / 2;
    const double sweeps = (double)rounds / (double)imax(np - 1, 1);
    *exec_flops = 6.0 * (double)s_nrot * (len + ncol) + 2.0 * (double)rounds * npairs * len +
                  2.0 * (sweeps + 1) * ncol * len;
    if (two_phase) *exec_flops += 4.0 * (double)ncol * ncol * ncol + 2.0 * (double)len * ncol * ncol;
  }
  // exact norms -> singular values, order and rank (identical in every CTA);
  // non-finite values order last and are reported
  __shared__ int s_r;
  for (bool again = false;; again = true) {
    rows_norms<double>(cc, R, wa, W, ncol, li);
    for (int j = threadIdx.x; j < ncol; j += blockDim.x) {
      const double sv = sqrt(nrm[j]) / scl;
      if (!(sv >= 0.0) || isinf(sv)) { sig[j] = -1.0; atomicOr(cc.status, ST_NAN); }
      else sig[j] = sv;
    }
    __syncthreads();
    for (int j = threadIdx.x; j < ncol; j += blockDim.x) {
      int rank = 0;
      const double sj = sig[j];
      for (int o = 0; o < ncol; ++o) rank += (sig[o] > sj) || (sig[o] == sj && o < j);
      perm[rank] = j;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      const int rmax = imin(J.chi, ncol);
      double tail2 = 0.0;
      for (int p = ncol - 1; p >= 1; --p) {
        const double sv = sig[perm[p]];
        tail2 += sv * sv;
        tail[2 + p] = tail2;
      }
      int rr = rmax;
      for (int qq = 1; qq <= rmax; ++qq) {
        const double t2 = (qq < ncol) ? tail[2 + qq] : 0.0;
        if (sqrt(t2) <= delta) { rr = qq; break; }
      }
      s_r = rr > bond_cap(L, J.dst.cap, k) ? 0 : rr;
    }
    __syncthreads();
    // the sweeps finish like any others: kept columns of W that are all rounding and have no
    // directions (a tolerance below the refinement's resolution), and pairs that kept their
    // cosine on both sides of the cut (of a Gram matrix, whose cut is its caller's: anywhere
    // above its rounding)
    if (again || state != RF_DONE || s_r < 1 || cc.dead) break;
    const double s0 = sig[perm[0]], sl = sig[perm[s_r - 1]];
    bool more = !trans && sl * sl <= (double)low * s0 * s0;
    if (tied) {
      const bool top = J.refine == REFINE_TOP;
      const double least = top ? 64.0 * 2.220446049250313e-16 * ncol * s0 : 0.0;
      for (int p = top ? 1 : s_r; p < (top ? ncol : imin(s_r + 1, ncol)); ++p) {
        const double a = sig[perm[p - 1]], b = sig[perm[p]];
        more |= b > least && a * a - b * b <= RF_TIE * a * a;
      }
    }
    if (!more) break;
    cl_sync(cc);                                  // the norms' slots have been read everywhere
    sw = rows_sweeps<double>(cc, R, wa, W, Vl, ncol, li, vi, maxsw, tol64 * tol64, &s_nrot, phase_acc, &conv, &rounds);
    *sweeps_out = sw;
    *noconv = !conv || cc.dead;
  }
  const int r = s_r;
  if (r > 0 && !cc.dead) {
    if (trans) {
      // core: rows of V^T (entries c in this CTA's V rows); U S: this CTA's rows of W
      for (int idx = threadIdx.x; idx < r * vi; idx += blockDim.x) {
        const int jr = idx / vi, ii = idx % vi;
        __stcg(out + (size_t)jr * n + v0 + ii, (T)Vl[(size_t)perm[jr] * R.lv + ii]);
      }
      for (int idx = threadIdx.x; idx < li * r; idx += blockDim.x) {
        const int ii = idx / r, jr = idx % r;
        __stcg(US + (size_t)(i0 + ii) * r + jr, (T)(W[(size_t)perm[jr] * R.lw + ii] * (1.0 / scl)));
      }
    } else {
      for (int idx = threadIdx.x; idx < r * li; idx += blockDim.x) {
        const int jr = idx / li, ii = idx % li;
        const int pj = perm[jr];
        const double sg = sig[pj] * scl;
        const double v = sg > 0.0 ? W[(size_t)pj * R.lw + ii] / sg : (i0 + ii == jr ? 1.0 : 0.0);
        __stcg(out + (size_t)jr * n + i0 + ii, (T)v);
      }
      for (int idx = threadIdx.x; idx < vi * r; idx += blockDim.x) {
        const int ii = idx / r, jr = idx % r;
        const int pj = perm[jr];
        __stcg(US + (size_t)(v0 + ii) * r + jr, (T)(Vl[(size_t)pj * R.lv + ii] * sig[pj]));
      }
    }
  }
  cl_sync(cc);
  return r;
}

// Shared-memory pointers of the leader CTA that the FP64 centre SVD uses.
struct SiteShared {
  double* red;
  double* tau;     // [1] scale, [2..] tails
  double* sig;
  int* perm;
  int* bad;
  int* rank;
  double* flops;
};

// Centre SVD of one right-to-left step in FP64 (FP32 data promoted, or FP64
// data on a cluster): C (m x n, T, global) = U S V^T by one-sided Jacobi in
// FP64 on the columns of C (n <= m) or of C^T; the rank rule and the
// discarded tail in FP64; writes core k = V^T[:r] (r x n) to out and U S
// (m x r) to US, both in T.  The Jacobi matrices sit in the leader's shared
// memory when the job has one CTA and they fit, else in the job's global
// scratch, where every CTA of the cluster works on them.  Returns the kept
// rank, or 0 after flagging an error.
template <typename T>
__device__ __noinline__ int svd64_site(const RoundJob& J, int L, int k, const T* C, int m, int n, T* out, T* US,
                                       T* scr, T* work, const SiteShared& sh, ClusterCtx& cc, int* status,
                                       const LearnCtx* lc, PhaseClock& pc, double delta) {
  const int ncol = imin(m, n), len = imax(m, n);
  const bool trans = (n <= m);
  const int ldw = jacobi_ld<double>(len), ldv = jacobi_ld<double>(ncol);
  const size_t need = ((size_t)ncol * ldw + (size_t)ncol * ldv) * sizeof(double);
  const bool in_smem = cc.P == 1 && need <= (size_t)SM_WORK;
  double* Wm = in_smem ? (double*)work : (double*)(scr + J.lay.jw64_off);
  double* Vm = in_smem ? (double*)work + (size_t)ncol * ldw : (double*)(scr + J.lay.jv64_off);
  // exact power-of-two scale so that max |C| is in [1, 2) (as the T path)
  T amax = (T)0;
  for (int idx = threadIdx.x; idx < m * n; idx += blockDim.x) amax = fmax(amax, fabs(C[idx]));
  for (int o = 16; o > 0; o >>= 1) amax = fmax(amax, __shfl_xor_sync(0xffffffffu, amax, o));
  if ((threadIdx.x & 31) == 0) sh.red[threadIdx.x >> 5] = (double)amax;
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) a = fmax(a, sh.red[w]);
    int e = 0;
    if (a > 0.0 && isfinite(a)) frexp(a, &e);
    sh.tau[1] = ldexp(1.0, 1 - e);
  }
  __syncthreads();
  const double scl = sh.tau[1];
  const int maxsw = J.max_sweeps > 0 ? J.max_sweeps : 60;
  // few columns: the sweeps of this CTA alone (a cluster of one)
  const Svd64Path path = cc.P > 1 ? svd64_path(ncol, len, cc.P, sizeof(T), J.refine) : Svd64Path{};
  const bool solo = path.solo;
  ClusterCtx one = cc;
  one.P = 1;
  one.rank = 0;
  if (solo || path.rows) {
    // rows of the Jacobi matrices spread over the cluster, in shared memory
    pc.lap(PH_SVD_OUT);
    int sw32 = 0;
    bool logged = false;
    if (path.reg || (sizeof(T) == 4 && !path.plain && !path.wide)) {
      // FP32 sweeps on X by this CTA alone (its own stopping rule, a
      // sweep limit, convergence not required).  In registers where X fits: W only,
      // the rotations logged for the cluster to form V0 (a row of V0 per half-warp,
      // ~1/16 of the sweeps' time on 16 CTAs, where carrying V along would double
      // the sweeps' work)
      if (path.reg) {
        float* Wf = (float*)work;
        const int ldw32 = jacobi_reg_ld(len), ncp = jacobi_reg_cols(ncol);
        for (int idx = threadIdx.x; idx < ncp * ldw32; idx += blockDim.x) {
          const int jj = idx / ldw32, i = idx % ldw32;
          Wf[idx] = jj < ncol && i < len ? (float)(scl * (double)(trans ? C[(size_t)i * n + jj] : C[(size_t)jj * n + i]))
                                         : 0.f;
        }
        __syncthreads();
        sw32 = jacobi_reg<true>(Wf, ncol, len, imin(maxsw, JR_LOG_SWEEPS), (float2*)(scr + J.lay.log_off));
        logged = true;
        __threadfence();                          // the log, before the workers are told of it
      } else if constexpr (sizeof(T) == 4) {
        // larger: the in-CTA Jacobi of the FP32 path, V0 left in the job's scratch
        const int ldw32 = jacobi_ld<float>(len), ldv32 = jacobi_ld<float>(ncol);
        const size_t need32 = ((size_t)ncol * ldw32 + (size_t)ncol * ldv32) * sizeof(float);
        float* Vg = (float*)(scr + J.lay.jv_off);
        // W (the hot operand: len entries per rotated column) in shared memory
        // whenever it fits there alone; V with it if both fit, else in scratch
        const bool w_smem = (size_t)ncol * ldw32 * sizeof(float) <= (size_t)SM_WORK;
        float* Wf = w_smem ? (float*)work : (float*)(scr + J.lay.jw_off);
        float* Vf = need32 <= (size_t)SM_WORK ? (float*)work + (size_t)ncol * ldw32 : Vg;
        for (int idx = threadIdx.x; idx < ncol * len; idx += blockDim.x) {
          const int jj = idx / len, i = idx % len;
          Wf[(size_t)jj * ldw32 + i] = (float)(scl * (double)(trans ? C[(size_t)i * n + jj] : C[(size_t)jj * n + i]));
        }
        __syncthreads();
        sw32 = jacobi_cols_fast<float>(Wf, ldw32, Vf, ldv32, ncol, len, imin(maxsw, 30));
        if (Vf != Vg)
          for (int idx = threadIdx.x; idx < ncol * ldv32; idx += blockDim.x) __stcg(Vg + idx, Vf[idx]);
        __syncthreads();
      }
      if (threadIdx.x == 0) pc.acc[PH_SWEEPS32] += sw32;
      pc.lap(PH_J32);
    }
    const int start = path.wide ? SW_WIDE : logged ? sw32 : path.plain || sizeof(T) == 8 ? SW_PLAIN : SW_SCRATCH;
    if (!solo) cl_command(cc, 2, ncol, len, maxsw, m, n, k, delta, scl, start);
    int sw = 0;
    bool noconv = false;
    double xfl = 0.0;
    const int r = svd64_rows<T>(solo ? one : cc, J, L, k, m, n, scl, delta, maxsw, start, &sw, &noconv, &xfl, pc.on ? pc.acc : nullptr);
    pc.lap(PH_JACOBI);
    if (threadIdx.x == 0) { pc.acc[PH_SVD64_FLOPS] += svd_flops(m, n); pc.acc[PH_SVD64_EXEC] += xfl; }
    const RowsLayout R = rows_layout(ncol, len, solo ? 1 : cc.P, rows_stage(sizeof(T), start));
    const unsigned char* wa = (const unsigned char*)work;
    const double* sig = (const double*)(wa + R.sig);
    const int* perm = (const int*)(wa + R.perm);
    const double* tail = (const double*)(wa + R.tail);
    if (threadIdx.x == 0) {
      pc.acc[6] += sw; pc.acc[7] += 1.0;
      if (noconv) {
        flag(status, ST_NOCONV);
        if (atomicCAS(&status[1], 0, 1) == 0) {
          status[2] = blockIdx.x / cc.P; status[3] = k; status[4] = ncol; status[5] = len;
        }
      }
      if (r == 0) flag(status, ST_CAPACITY);
      else {
        if (J.discard && r < ncol) atomicAdd(J.discard, tail[2 + r]);
        J.dst.ranks[k] = r;
      }
      *sh.flops += svd_flops(m, n);
      if (lc && lc->counters) atomicAdd(&lc->counters[2], 1);
    }
    // singular values and order where the spectrum log reads them
    for (int j = threadIdx.x; j < ncol; j += blockDim.x) { sh.sig[j] = sig[j]; sh.perm[j] = perm[j]; }
    // the other CTAs wrote rows of the core and of U S at L2: read them back
    // past this SM's L1 before the leader's own loads use them
    if (r > 0) {
      for (int idx = threadIdx.x; idx < r * n; idx += blockDim.x) out[idx] = __ldcg(out + idx);
      for (int idx = threadIdx.x; idx < m * r; idx += blockDim.x) US[idx] = __ldcg(US + idx);
    }
    __syncthreads();
    return r;
  }
  for (int idx = threadIdx.x; idx < ncol * len; idx += blockDim.x) {
    const int jj = idx / len, i = idx % len;
    const double v = scl * (double)(trans ? C[(size_t)i * n + jj] : C[(size_t)jj * n + i]);
    if (in_smem) Wm[(size_t)jj * ldw + i] = v;
    else __stcg(Wm + (size_t)jj * ldw + i, v);
  }
  __syncthreads();
  pc.lap(PH_SVD_OUT);
  const double jac0 = pc.acc[PH_JACOBI];
  int sw;
  if (in_smem) {
    sw = jacobi_cols_fast<double>(Wm, ldw, Vm, ldv, ncol, len, maxsw);
  } else {
    cl_command(cc, 1, ncol, len, maxsw);
    sw = jacobi64_cluster(cc, Wm, ldw, Vm, ldv, ncol, len, maxsw);
  }
  pc.lap(PH_JACOBI);
  if (threadIdx.x == 0) { pc.acc[6] += sw; pc.acc[7] += 1.0; pc.acc[PH_SVD64_FLOPS] += svd_flops(m, n); }
  if (threadIdx.x == 0 && !in_smem) { pc.acc[8] += pc.acc[PH_JACOBI] - jac0; pc.acc[9] += 1.0; }
  if (sw >= maxsw && threadIdx.x == 0) {
    flag(status, ST_NOCONV);
    if (atomicCAS(&status[1], 0, 1) == 0) {
      status[2] = blockIdx.x / cc.P; status[3] = k; status[4] = ncol; status[5] = len;
    }
  }
  auto ldW = [&](size_t i) -> double { return in_smem ? Wm[i] : __ldcg(Wm + i); };
  auto ldV = [&](size_t i) -> double { return in_smem ? Vm[i] : __ldcg(Vm + i); };
  for (int jj = threadIdx.x; jj < ncol; jj += blockDim.x) {
    double a = 0.0;
    for (int i = 0; i < len; ++i) { const double w = ldW((size_t)jj * ldw + i); a += w * w; }
    const double sv = sqrt(a) / scl;
    if (!(sv >= 0.0) || isinf(sv)) { sh.sig[jj] = -1.0; flag(status, ST_NAN); }   // orders last
    else sh.sig[jj] = sv;
  }
  __syncthreads();
  for (int jj = threadIdx.x; jj < ncol; jj += blockDim.x) {
    int rank = 0;
    const double sj = sh.sig[jj];
    for (int o = 0; o < ncol; ++o) {
      const double so = sh.sig[o];
      rank += (so > sj) || (so == sj && o < jj);
    }
    sh.perm[rank] = jj;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const int rmax = imin(J.chi, ncol);
    double tail2 = 0.0;
    int rr = rmax;
    for (int p = ncol - 1; p >= 1; --p) {
      const double sv = sh.sig[sh.perm[p]];
      tail2 += sv * sv;
      sh.tau[2 + p] = tail2;
    }
    for (int q = 1; q <= rmax; ++q) {
      const double t2 = (q < ncol) ? sh.tau[2 + q] : 0.0;
      if (sqrt(t2) <= delta) { rr = q; break; }
    }
    if (rr > bond_cap(L, J.dst.cap, k)) { *sh.bad = 1; rr = bond_cap(L, J.dst.cap, k); }
    *sh.rank = rr;
    if (J.discard && rr < ncol) atomicAdd(J.discard, sh.tau[2 + rr]);
    *sh.flops += svd_flops(m, n);
    if (lc && lc->counters) atomicAdd(&lc->counters[2], 1);
  }
  __syncthreads();
  if (*sh.bad) { if (threadIdx.x == 0) flag(status, ST_CAPACITY); return 0; }
  const int r = *sh.rank;
  for (int idx = threadIdx.x; idx < r * n; idx += blockDim.x) {
    const int jr = idx / n, c = idx % n;
    const int pj = sh.perm[jr];
    double v;
    if (trans) {
      v = ldV((size_t)pj * ldv + c);
    } else {
      const double sg = sh.sig[pj] * scl;
      v = sg > 0.0 ? ldW((size_t)pj * ldw + c) / sg : (c == jr ? 1.0 : 0.0);
    }
    out[idx] = (T)v;
  }
  for (int idx = threadIdx.x; idx < m * r; idx += blockDim.x) {
    const int i = idx / r, jr = idx % r;
    const int pj = sh.perm[jr];
    US[idx] = (T)(trans ? ldW((size_t)pj * ldw + i) * (1.0 / scl) : ldV((size_t)pj * ldv + i) * sh.sig[pj]);
  }
  if (threadIdx.x == 0) J.dst.ranks[k] = r;
  __syncthreads();
  return r;
}

// Shared-memory bytes of svd32_site: W, then (once W is final) the kept rows of
// V^T and their Gram matrix beside it.
__host__ __device__ inline size_t svd32_vbytes(int r, int n) {
  return ((size_t)r * (n | 1) + (size_t)r * (r | 1)) * sizeof(float);
}

// Bytes of the copy of C that svd32_site's QR works on, its panel after it.
__host__ __device__ inline size_t svd32_qr_off(int m, int n) {
  return ((size_t)m * (n | 1) * sizeof(float) + 15) & ~(size_t)15;
}

// Whether svd32_site takes an m x n centre matrix: its vectors fit the register
// Jacobi, and W with the QR panel (m > n) fits the work area.
__host__ __device__ inline bool svd32_fits(int m, int n) {
  const int k = m < n ? m : n;
  if (!jacobi_reg_fits(k, n)) return false;
  if (m > n && (!qr_reg_fits(m, n) || svd32_qr_off(m, n) + qr_reg_bytes(m) > (size_t)SM_WORK)) return false;
  return (size_t)jacobi_reg_cols(k) * jacobi_reg_ld(n) * sizeof(float) <= (size_t)SM_WORK;
}

// Centre SVD of one right-to-left step in FP32, without accumulating the
// rotations: the Jacobi runs on the rows of C (n-vectors; of the R of C = QR when
// m > n, whose right singular vectors are C's), so its converged vectors are
// s_j v_j, their directions the kept rows of V^T, and U S = C V is one product.
// The kept rows are made orthonormal to FP32 rounding by one Newton-Schulz step
// (the Jacobi stops at |cos| <= 16 eps sqrt(n)), so C V V^T is an orthogonal
// projection of C itself: the error is that of the discarded part and of one
// product, not of the ~1000 rotations a column goes through.  Vectors below the
// Jacobi's floor (1e-12 of the scale) carry nothing: their columns of U S are zero.
// Leaves singular values and order in sh.sig / sh.perm; returns the kept rank,
// or 0 after flagging an error.
__device__ __noinline__ int svd32_site(const RoundJob& J, int L, int k, const float* C, int m, int n, float* out,
                                       float* US, float* scr, float* work, const SiteShared& sh, int job,
                                       int* status, const LearnCtx* lc, PhaseClock& pc,
                                       double delta) {
  const int ncol = imin(m, n), ld = jacobi_reg_ld(n), ncp = jacobi_reg_cols(ncol);
  float* W = work;
  // exact power-of-two scale so that max |C| is in [1, 2)
  float amax = 0.f;
  for (int idx = threadIdx.x; idx < m * n; idx += blockDim.x) amax = fmaxf(amax, fabsf(C[idx]));
  for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
  if ((threadIdx.x & 31) == 0) sh.red[threadIdx.x >> 5] = (double)amax;
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) a = fmax(a, sh.red[w]);
    int e = 0;
    if (a > 0.0 && isfinite(a)) frexp(a, &e);
    sh.tau[1] = ldexp(1.0, 1 - e);
  }
  __syncthreads();
  const double scl = sh.tau[1];
  const float* X = C;
  if (m > n) {
    // R of C (n x n): the QR runs on a copy in the work area
    const int lda = n | 1;
    for (int idx = threadIdx.x; idx < m * n; idx += blockDim.x) work[(size_t)(idx / n) * lda + idx % n] = C[idx];
    __syncthreads();
    float* R = scr + J.lay.jv_off;
    float* V = (float*)((unsigned char*)work + svd32_qr_off(m, n));
    qr_reg(work, m, n, lda, nullptr, 0, R, n, V, V + (size_t)m * 16, scr + J.lay.qw_off, (float*)sh.sig);
    X = R;
  }
  for (int idx = threadIdx.x; idx < ncp * ld; idx += blockDim.x) {
    const int j = idx / ld, i = idx % ld;
    W[idx] = (j < ncol && i < n) ? (float)scl * X[(size_t)j * n + i] : 0.f;
  }
  __syncthreads();
  const int maxsw = J.max_sweeps > 0 ? J.max_sweeps : 60;
  pc.lap(PH_SVD_OUT);
  const int sw = jacobi_reg<false>(W, ncol, n, maxsw, nullptr);
  pc.lap(PH_JACOBI);
  if (threadIdx.x == 0) {
    pc.acc[6] += sw; pc.acc[7] += 1.0;
    if (sw >= maxsw) {
      flag(status, ST_NOCONV);
      if (atomicCAS(&status[1], 0, 1) == 0) {
        status[2] = job; status[3] = k; status[4] = ncol; status[5] = imax(m, n);
      }
    }
  }
  // the padded columns moved among the others: norms of all ncp; padding is zero like
  // any column of nothing, and what is not finite orders behind it (and is reported)
  {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int j = warp; j < ncp; j += nw) {
      float a = 0.f;
      for (int i = lane; i < ld; i += 32) { const float w = W[(size_t)j * ld + i]; a = fmaf(w, w, a); }
      for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
      if (lane == 0) {
        const double sv = (double)sqrtf(a) / scl;
        if (!(sv >= 0.0) || isinf(sv)) { sh.sig[j] = -1.0; flag(status, ST_NAN); }
        else sh.sig[j] = sv;
      }
    }
  }
  __syncthreads();
  for (int jj = threadIdx.x; jj < ncp; jj += blockDim.x) {
    int rank = 0;
    const double sj = sh.sig[jj];
    for (int o = 0; o < ncp; ++o) {
      const double so = sh.sig[o];
      rank += (so > sj) || (so == sj && o < jj);
    }
    sh.perm[rank] = jj;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const int rmax = imin(J.chi, ncol);
    double tail2 = 0.0;
    int rr = rmax;
    for (int p = ncol - 1; p >= 1; --p) {
      const double sv = sh.sig[sh.perm[p]];
      tail2 += sv * sv;
      sh.tau[2 + p] = tail2;
    }
    for (int q = 1; q <= rmax; ++q) {
      const double t2 = (q < ncol) ? sh.tau[2 + q] : 0.0;
      if (sqrt(t2) <= delta) { rr = q; break; }
    }
    if (rr > bond_cap(L, J.dst.cap, k)) { *sh.bad = 1; rr = bond_cap(L, J.dst.cap, k); }
    *sh.rank = rr;
    if (J.discard && rr < ncol) atomicAdd(J.discard, sh.tau[2 + rr]);
    *sh.flops += svd_flops(m, n);
    if (lc && lc->counters) atomicAdd(&lc->counters[2], 1);
  }
  __syncthreads();
  if (*sh.bad) { if (threadIdx.x == 0) flag(status, ST_CAPACITY); return 0; }
  const int r = *sh.rank;
  // kept directions, orthonormalised: V <- (3/2 I - 1/2 V V^T) V
  const size_t wbytes = (size_t)ncp * ld * sizeof(float);
  const bool vs = wbytes + svd32_vbytes(r, n) <= (size_t)SM_WORK;
  const int ldv = vs ? (n | 1) : n, ldg = r | 1;
  float* V = vs ? work + (size_t)ncp * ld : out;
  float* G = vs ? V + (size_t)r * ldv : scr + J.lay.jv_off;
  for (int idx = threadIdx.x; idx < r * n; idx += blockDim.x) {
    const int jr = idx / n, c = idx % n, pj = sh.perm[jr];
    const float sg = (float)(sh.sig[pj] * scl);
    V[(size_t)jr * ldv + c] = sg > 0.f ? W[(size_t)pj * ld + c] / sg : (c == jr ? 1.f : 0.f);
  }
  __syncthreads();
  cta_gemm_nt<float>(r, r, n, V, ldv, V, ldv, G, vs ? ldg : r);
  for (int idx = threadIdx.x; idx < r * r; idx += blockDim.x) {
    const int i = idx / r, j = idx % r;
    const bool live = sh.sig[sh.perm[i]] * scl > 1e-12 && sh.sig[sh.perm[j]] * scl > 1e-12;
    float* g = G + (size_t)i * (vs ? ldg : r) + j;
    *g = (i == j ? 1.f : 0.f) + (live ? 0.5f * ((i == j ? 1.f : 0.f) - *g) : 0.f);
  }
  __syncthreads();
  // V is read as a whole before it is replaced: the product goes to the W area
  cta_gemm<float>(r, n, r, G, vs ? ldg : r, V, ldv, W, n, false);
  for (int idx = threadIdx.x; idx < r * n; idx += blockDim.x) {
    const float v = W[idx];
    out[idx] = v;
    if (vs) V[(size_t)(idx / n) * ldv + idx % n] = v;
  }
  __syncthreads();
  cta_gemm_nt<float>(m, r, n, C, n, V, ldv, US, r);
  for (int idx = threadIdx.x; idx < m * r; idx += blockDim.x)
    if (sh.sig[sh.perm[idx % r]] * scl <= 1e-12) US[idx] = 0.f;
  if (threadIdx.x == 0) J.dst.ranks[k] = r;
  __syncthreads();
  return r;
}

// The rounding job as run by the leader CTA of its cluster (the whole job
// when the cluster has one CTA).
template <typename T>
__device__ void round_job_body(const RoundJob& J, int L_arg, int n_bits_arg, const T* __restrict__ masks_arg,
                               const double* __restrict__ scal_arg, int* __restrict__ status,
                               double* __restrict__ ctr, const LearnCtx* __restrict__ lc, ClusterCtx& cc) {
  // per-job chain length, mask table and scalars (jobs of several simulations,
  // possibly of different lattice sizes, in one launch)
  const int L = J.L > 0 ? J.L : L_arg;
  const int n_bits = J.n_bits > 0 ? J.n_bits : n_bits_arg;
  const T* __restrict__ masks = J.masks ? (const T*)J.masks : masks_arg;
  const double* __restrict__ scal = J.scal ? J.scal : scal_arg;
  extern __shared__ __align__(16) unsigned char smem[];
  int* s_rt = (int*)smem;                            // [TN_MAXT][TN_MAXL+1] term bonds
  int* s_ro = s_rt + TN_MAXT * (TN_MAXL + 1);        // row offsets at each bond
  int* s_wo = s_ro + TN_MAXT * (TN_MAXL + 1);        // per-term offsets in W buffer
  int* s_R = s_wo + TN_MAXT;                         // wide bonds
  int* s_q = s_R + TN_MAXL + 1;                      // QR sweep bonds
  int* s_perm = s_q + TN_MAXL + 1;                   // [MAXK]
  double* s_red = (double*)(smem + SM_RED);
  double* s_tau = (double*)(smem + SM_TAU);
  double* s_sig = (double*)(smem + SM_SIG);
  T* s_wv = (T*)(smem + SM_WV);
  T* work = (T*)(smem + SM_SMALL);
  __shared__ double s_coef[TN_MAXT];
  __shared__ double s_phase[PH_COUNT];
  __shared__ double s_flops;                          // algorithmic FLOPs (thread 0)
  __shared__ int s_bad, s_rank;

  const int nt = J.nterms;
  T* scr = (T*)J.scratch;
  double& flops = s_flops;
  PhaseClock pc(ctr != nullptr, s_phase);
  if (threadIdx.x == 0) { s_bad = 0; s_flops = 0.0; }
  __syncthreads();
  // ---- bonds of every term and of the wide sum
  for (int idx = threadIdx.x; idx < nt * (L + 1); idx += blockDim.x) {
    const int t = idx / (L + 1), k = idx % (L + 1);
    const Term& tm = J.t[t];
    int rb = term_bond(tm, n_bits, k);
    if (tm.kind != T_ONES) {
      if (tm.x.ranks[k] > bond_cap(L, tm.x.cap, k) || tm.x.ranks[k] < 1) s_bad = 1;
      if (tm.kind == T_KRON && (tm.y.ranks[k] > bond_cap(L, tm.y.cap, k) || tm.y.ranks[k] < 1)) s_bad = 1;
    }
    s_rt[t * (TN_MAXL + 1) + k] = rb;
  }
  for (int t = threadIdx.x; t < nt; t += blockDim.x) {
    double c = J.t[t].coef;
    if (J.t[t].coef_slot >= 0) c *= scal[J.t[t].coef_slot];
    s_coef[t] = c;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 0; k <= L; ++k) {
      int acc = 0;
      for (int t = 0; t < nt; ++t) {
        s_ro[t * (TN_MAXL + 1) + k] = (k == 0 || k == L) ? 0 : acc;
        acc += s_rt[t * (TN_MAXL + 1) + k];
      }
      s_R[k] = (k == 0 || k == L) ? 1 : acc;
      if (s_R[k] > J.rw[k]) s_bad = 1;
    }
  }
  __syncthreads();
  if (s_bad) { if (threadIdx.x == 0) flag(status, ST_CAPACITY); return; }

  // ---- materialise a single term without rounding
  if (J.materialize_only) {
    const Term& tm = J.t[0];
    for (int k = 0; k < L; ++k) {
      const int r0 = s_rt[k], r1 = s_rt[k + 1];
      if (r0 > bond_cap(L, J.dst.cap, k) || r1 > bond_cap(L, J.dst.cap, k + 1)) {
        if (threadIdx.x == 0) flag(status, ST_CAPACITY);
        return;
      }
      T* out = (T*)J.dst.base + core_offset(L, J.dst.cap, k);
      const T cf = (T)(k == 0 ? s_coef[0] : 1.0);
      for (int idx = threadIdx.x; idx < r0 * 2 * r1; idx += blockDim.x) {
        int i = idx / (2 * r1), s = (idx / r1) % 2, jj = idx % r1;
        out[idx] = cf * term_elem<T>(tm, L, n_bits, k, i, s, jj, masks);
      }
    }
    for (int k = threadIdx.x; k <= L; k += blockDim.x) J.dst.ranks[k] = s_rt[k];
    return;
  }

  // ---- left-orthogonalising sweep over the wide sum
  T* Rc = scr + J.lay.r_off;                // carried R factor, rc x R_k (ld R_k)
  if (threadIdx.x == 0) { Rc[0] = (T)1; s_q[0] = 1; }
  __syncthreads();
  int rc = 1;
  for (int k = 0; k < L; ++k) {
    const int Rk = s_R[k], Rk1 = s_R[k + 1];
    // (a) term blocks of core k into W (global scratch)
    T* W = scr + J.lay.w_off;
    if (threadIdx.x == 0) {
      int o = 0;
      for (int t = 0; t < nt; ++t) {
        s_wo[t] = o;
        o += s_rt[t * (TN_MAXL + 1) + k] * 2 * s_rt[t * (TN_MAXL + 1) + k + 1];
      }
    }
    __syncthreads();
    for (int t = 0; t < nt; ++t) {
      const int r0 = s_rt[t * (TN_MAXL + 1) + k], r1 = s_rt[t * (TN_MAXL + 1) + k + 1];
      const T cf = (T)(k == 0 ? s_coef[t] : 1.0);
      T* Wt = W + s_wo[t];
      for (int idx = threadIdx.x; idx < r0 * 2 * r1; idx += blockDim.x) {
        int i = idx / (2 * r1), s = (idx / r1) % 2, jj = idx % r1;
        Wt[idx] = cf * term_elem<T>(J.t[t], L, n_bits, k, i, s, jj, masks);
      }
    }
    __syncthreads();
    pc.lap(PH_TERMS);
    // (b) M = Rc * blockdiag(W): rows (r, s), row length Rk1, leading dim ld
    const int mrows = 2 * rc;
    int ld = Rk1 | 1;
    // FP32: the register QR, with its panel beside M in the work area
    const bool reg_qr = sizeof(T) == 4 && qr_reg_fits(mrows, Rk1) && qr_reg_bytes(mrows) <= (size_t)SM_WORK;
    const size_t msz = ((size_t)mrows * ld * sizeof(T) + 15) & ~(size_t)15;
    bool in_smem = msz + (reg_qr ? qr_reg_bytes(mrows) : 0) <= (size_t)SM_WORK;
    if (!in_smem) ld = Rk1;
    T* M = in_smem ? work : scr + J.lay.m_off;
    const bool last = (k == L - 1);
    if (last)
      for (int idx = threadIdx.x; idx < mrows * ld; idx += blockDim.x) M[idx] = (T)0;
    __syncthreads();
    for (int t = 0; t < nt; ++t) {
      const int r0 = s_rt[t * (TN_MAXL + 1) + k], r1 = s_rt[t * (TN_MAXL + 1) + k + 1];
      const int co = s_ro[t * (TN_MAXL + 1) + k + 1], ro = s_ro[t * (TN_MAXL + 1) + k];
      const T* Wt = W + s_wo[t];
      for (int s = 0; s < 2; ++s)
        cta_gemm<T>(rc, r1, r0, Rc + ro, Rk, Wt + s * r1, 2 * r1, M + (size_t)s * ld + co, 2 * ld, last);
      if (threadIdx.x == 0) flops += 4.0 * rc * r0 * r1;
    }
    pc.lap(PH_GEMM_M);
    T* Qk = scr + J.lay.q_off[k];
    if (last) {
      for (int idx = threadIdx.x; idx < mrows; idx += blockDim.x) Qk[idx] = M[(size_t)idx * ld];
      __syncthreads();
      break;
    }
    // (c) QR of M (mrows x Rk1) -> Q_k (ld rq), new carried R (rq x Rk1, ld Rk1)
    const int rq = imin(mrows, Rk1);
    if (rq > MAXK || Rk1 > MAXK) { if (threadIdx.x == 0) flag(status, ST_CAPACITY); return; }
    T* vb = scr + J.lay.qw_off;
    bool qr_done = false;
    if constexpr (sizeof(T) == 4) {
      if (reg_qr) {
        float* V = (float*)((unsigned char*)work + (in_smem ? msz : 0));
        qr_reg(M, mrows, Rk1, ld, Qk, rq, Rc, Rk1, V, V + (size_t)mrows * 16, vb, (float*)s_sig);
        qr_done = true;
      }
    }
    if (!qr_done)
      householder_qr_blk<T>(M, mrows, Rk1, ld, Qk, rq, Rc, Rk1, s_tau, s_wv, s_red, vb, vb + (size_t)mrows * QB);
    if (threadIdx.x == 0) flops += qr_flops(mrows, Rk1);
    pc.lap(PH_QR);
    rc = rq;
    if (threadIdx.x == 0) s_q[k + 1] = rq;
    __syncthreads();
    (void)Rk;
  }
  if (threadIdx.x == 0) s_q[L] = 1;
  __syncthreads();

  // ---- right-to-left truncated SVD sweep
  T* C = scr + J.lay.c_off;
  {
    const int q = s_q[L - 1];
    const T* Ql = scr + J.lay.q_off[L - 1];
    double part = 0.0;
    for (int idx = threadIdx.x; idx < 2 * q; idx += blockDim.x) {
      double v = (double)Ql[idx];
      part += v * v;
      C[idx] = Ql[idx];
    }
    double nrm2 = block_sum(part, s_red);
    if (!isfinite(nrm2)) { if (threadIdx.x == 0) flag(status, ST_NAN); }
    if (threadIdx.x == 0) s_tau[0] = J.eps * sqrt(nrm2) / sqrt((double)(L - 1));
    __syncthreads();
  }
  const double delta = s_tau[0];
  __syncthreads();
  int rnext = 1;
  for (int k = L - 1; k >= 1; --k) {
    const int m = s_q[k], n = 2 * rnext;
    T* out = (T*)J.dst.base + core_offset(L, J.dst.cap, k);
    T* US = scr + J.lay.us_off;
    int r = 0;
    bool done = false;             // randomized truncation accepted
    bool full64 = false;           // full SVD taken by svd64_site or svd32_site
    // ---- randomized truncation at a target rank, certified (learned-rank path)
    int tgt = 0;
    if (J.rsvd_mode && lc != nullptr && lc->omega != nullptr) {
      if (J.rsvd_mode == 1) {
        tgt = J.targets ? J.targets[k] : J.rsvd_k;
      } else if (J.rsvd_mode == 3 && J.log != nullptr && J.log->valid[k]) {
        tgt = J.log->label[k];                     // previous step's kept rank
      } else if (J.rsvd_mode == 2 && lc->mlp != nullptr && J.log != nullptr && J.log->valid[k]) {
        const float stepf = lc->step ? fminf((float)(*lc->step) / 1000.f, 1.f) : 0.f;
        tgt = mlp_predict_rank(lc->mlp, J.log->spec[k], (float)k / (float)L, stepf, J.chi,
                               (float*)s_sig);
      }
    }
    tgt = imin(tgt, J.chi);
    const int fullmin = imin(m, n);
    // at least TN_SPEC samples, so that the logged spectrum has every value the model reads
    const int lsamp = imin(imax(tgt + (lc ? lc->oversample : 0), TN_SPEC), fullmin);
    // Y (m x l, and n x l in the power steps) must fit the shared work area;
    // B and V (l x n, l x l) go there too when they fit, else to global scratch
    const bool fits = (size_t)imax(m, n) * (lsamp | 1) * sizeof(T) <= (size_t)SM_WORK;
    const bool bv_smem = ((size_t)lsamp * jacobi_ld<T>(n) + (size_t)lsamp * jacobi_ld<T>(lsamp)) * sizeof(T) <=
                         (size_t)SM_WORK;
    if (tgt > 0 && lsamp < fullmin && fits && n <= lc->omega_rows && lsamp <= lc->omega_ld) {
      const int l = lsamp;
      const int ldy = l | 1, ldw = jacobi_ld<T>(n), ldv = jacobi_ld<T>(l);
      T* Ysm = work;
      const T* Om = (const T*)lc->omega;
      // Y = C Omega (m x l), in shared memory
      cta_gemm<T>(m, l, n, C, n, Om, lc->omega_ld, Ysm, ldy, false);
      T* Qy = scr + J.lay.jw_off;                  // m x l
      T* Rtmp = scr + J.lay.jv_off;                // l x l (discarded)
      // power steps: Y <- C orth(C^T orth(Y)), re-orthonormalised for stability
      for (int it = 0; it < lc->power; ++it) {
        T* Z = scr + J.lay.rz_off;                 // n x l
        householder_qr_par<T>(Ysm, m, l, ldy, Qy, l, Rtmp, l, s_tau, s_wv, s_red);
        cta_gemm_tn<T>(n, l, m, C, n, Qy, l, Ysm, ldy);
        householder_qr_par<T>(Ysm, n, l, ldy, Z, l, Rtmp, l, s_tau, s_wv, s_red);
        cta_gemm<T>(m, l, n, C, n, Z, l, Ysm, ldy, false);
        if (threadIdx.x == 0) flops += 4.0 * m * n * l + qr_flops(m, l) + qr_flops(n, l);
      }
      householder_qr_par<T>(Ysm, m, l, ldy, Qy, l, Rtmp, l, s_tau, s_wv, s_red);
      // B = Qy^T C (l x n), row j = Jacobi column j; in shared memory, or in the
      // power-step and R regions of the scratch (both free by now)
      T* Wm = bv_smem ? work : scr + J.lay.rz_off;
      T* Vm = bv_smem ? work + (size_t)l * ldw : Rtmp;
      cta_gemm_tn<T>(l, n, m, Qy, l, C, n, Wm, ldw);
      // residual ||C - Qy B||^2 and ||C||^2 (FP64 sums)
      double pr = 0.0, pc2 = 0.0;
      for (int idx = threadIdx.x; idx < m * n; idx += blockDim.x) {
        const int i = idx / n, c = idx % n;
        const T* qrow = Qy + (size_t)i * l;
        T acc = C[idx];
        for (int q = 0; q < l; ++q) acc -= qrow[q] * Wm[(size_t)q * ldw + c];
        pr += (double)acc * (double)acc;
        pc2 += (double)C[idx] * (double)C[idx];
      }
      const double resid2 = block_sum(pr, s_red);
      const double c2 = block_sum(pc2, s_red);
      // scale B to max |entry| in [1, 2)
      T amax = (T)0;
      for (int idx = threadIdx.x; idx < l * n; idx += blockDim.x)
        amax = fmax(amax, fabs(Wm[(size_t)(idx / n) * ldw + idx % n]));
      for (int o = 16; o > 0; o >>= 1) amax = fmax(amax, __shfl_xor_sync(0xffffffffu, amax, o));
      if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = (double)amax;
      __syncthreads();
      if (threadIdx.x == 0) {
        double a = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) a = fmax(a, s_red[w]);
        int e = 0;
        if (a > 0.0 && isfinite(a)) frexp(a, &e);
        s_tau[1] = ldexp(1.0, 1 - e);
      }
      __syncthreads();
      const double scl = s_tau[1];
      for (int idx = threadIdx.x; idx < l * n; idx += blockDim.x)
        Wm[(size_t)(idx / n) * ldw + idx % n] *= (T)scl;
      __syncthreads();
      const int sw = jacobi_cols_fast<T>(Wm, ldw, Vm, ldv, l, n, 60);
      for (int jj = threadIdx.x; jj < l; jj += blockDim.x) {
        T a = (T)0;
        const T* w = Wm + (size_t)jj * ldw;
        for (int i = 0; i < n; ++i) a += w[i] * w[i];
        const double sv = (double)sqrt(a) / scl;
        if (!(sv >= 0.0) || isinf(sv)) { s_sig[jj] = -1.0; flag(status, ST_NAN); }   // orders last
        else s_sig[jj] = sv;
      }
      __syncthreads();
      for (int jj = threadIdx.x; jj < l; jj += blockDim.x) {
        int rank = 0;
        const double sj = s_sig[jj];
        for (int o = 0; o < l; ++o) rank += (s_sig[o] > sj) || (s_sig[o] == sj && o < jj);
        s_perm[rank] = jj;
      }
      __syncthreads();
      if (threadIdx.x == 0) {
        const int rmax = imin(J.chi, l);
        double tail2 = 0.0;
        s_tau[2 + l] = 0.0;
        for (int p = l - 1; p >= 0; --p) {
          const double sv = s_sig[s_perm[p]];
          tail2 += sv * sv;
          s_tau[2 + p] = tail2;
        }
        int rr = rmax;
        for (int q = 1; q <= rmax; ++q)
          if (sqrt(resid2 + s_tau[2 + q]) <= delta) { rr = q; break; }
        const double err2 = resid2 + s_tau[2 + rr];
        const int full_cap = imin(J.chi, imin(m, n));
        const bool rule_ok = sqrt(err2) <= delta || rr == full_cap || rr == J.chi;
        // accept: measured error within the tolerance, or (at the chi cap) the
        // residual bound proves err^2 <= opt^2 / (1 - eta) (Ky Fan on C^T C = B^T B + E^T E)
        const double floor2 = (double)lc->floor_rel * (double)lc->floor_rel * c2;
        const bool cert = sqrt(err2) <= delta || resid2 <= fmax((double)lc->eta * err2, floor2);
        const bool ok = rule_ok && cert && sw < 60 && rr <= bond_cap(L, J.dst.cap, k);
        s_rank = ok ? rr : 0;
        if (ok && J.discard) atomicAdd(J.discard, err2);
        if (lc->counters) atomicAdd(&lc->counters[ok ? 0 : 1], 1);
        flops += 2.0 * m * n * l * 3 + qr_flops(m, l) + svd_flops(l, n);
      }
      __syncthreads();
      if (s_rank > 0) {
        r = s_rank;
        for (int idx = threadIdx.x; idx < r * n; idx += blockDim.x) {
          const int jr = idx / n, c = idx % n;
          const int pj = s_perm[jr];
          const T sg = (T)(s_sig[pj] * scl);
          out[idx] = sg > (T)0 ? Wm[(size_t)pj * ldw + c] / sg : (T)(c == jr ? 1 : 0);
        }
        for (int idx = threadIdx.x; idx < m * r; idx += blockDim.x) {
          const int i = idx / r, jr = idx % r;
          const int pj = s_perm[jr];
          const T* qrow = Qy + (size_t)i * l;
          const T* vcol = Vm + (size_t)pj * ldv;
          T acc = (T)0;
          for (int q = 0; q < l; ++q) acc += qrow[q] * vcol[q];
          US[idx] = acc * (T)s_sig[pj];
        }
        done = true;
        if (threadIdx.x == 0) J.dst.ranks[k] = r;
      }
      __syncthreads();
      pc.lap(PH_JACOBI);
    }
    // ---- full SVD (reference path, and fallback of the randomized one)
    const int ncol = imin(m, n), len = imax(m, n);
    if (!done && (J.svd64 || (sizeof(T) == 8 && cc.P > 1))) {
      if (ncol > MAXK) { if (threadIdx.x == 0) flag(status, ST_CAPACITY); return; }
      const SiteShared sh{s_red, s_tau, s_sig, s_perm, &s_bad, &s_rank, &s_flops};
      r = svd64_site<T>(J, L, k, C, m, n, out, US, scr, work, sh, cc, status, lc, pc, delta);
      if (r == 0) return;
      full64 = true;
    }
    if constexpr (sizeof(T) == 4) {
      if (!done && !full64 && svd32_fits(m, n)) {
        const SiteShared sh{s_red, s_tau, s_sig, s_perm, &s_bad, &s_rank, &s_flops};
        r = svd32_site(J, L, k, C, m, n, out, US, scr, work, sh, blockIdx.x / cc.P, status, lc, pc, delta);
        if (r == 0) return;
        full64 = true;
      }
    }
    if (!done && !full64) {
      if (ncol > MAXK) { if (threadIdx.x == 0) flag(status, ST_CAPACITY); return; }
      const bool trans = (n <= m);             // Jacobi on the columns of C
      // 16-byte row strides (vector loads in the Jacobi); shared memory if it
      // fits -- W alone when W and V do not fit together
      const int ldw = jacobi_ld<T>(len), ldv = jacobi_ld<T>(ncol);
      const size_t need = ((size_t)ncol * ldw + (size_t)ncol * ldv) * sizeof(T);
      const bool w_smem = (size_t)ncol * ldw * sizeof(T) <= (size_t)SM_WORK;
      T* Wm = w_smem ? work : scr + J.lay.jw_off;
      T* Vm = (need <= (size_t)SM_WORK) ? work + (size_t)ncol * ldw : scr + J.lay.jv_off;
      const int ldw_e = ldw;
      const int ldv_e = ldv;
      // scale by an exact power of two so that max |C| is in [1, 2): keeps the
      // Jacobi inner products far from under- and overflow; undone exactly below
      T amax = (T)0;
      for (int idx = threadIdx.x; idx < m * n; idx += blockDim.x) amax = fmax(amax, fabs(C[idx]));
      for (int o = 16; o > 0; o >>= 1) amax = fmax(amax, __shfl_xor_sync(0xffffffffu, amax, o));
      if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = (double)amax;
      __syncthreads();
      if (threadIdx.x == 0) {
        double a = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) a = fmax(a, s_red[w]);
        int e = 0;
        if (a > 0.0 && isfinite(a)) frexp(a, &e);
        s_tau[1] = ldexp(1.0, 1 - e);     // scale
      }
      __syncthreads();
      const double scl = s_tau[1];
      const T tscl = (T)scl;
      for (int idx = threadIdx.x; idx < ncol * len; idx += blockDim.x) {
        const int jj = idx / len, i = idx % len;
        Wm[(size_t)jj * ldw_e + i] = tscl * (trans ? C[(size_t)i * n + jj] : C[(size_t)jj * n + i]);
      }
      __syncthreads();
      const int maxsw = J.max_sweeps > 0 ? J.max_sweeps : 60;
      pc.lap(PH_SVD_OUT);
      const double jac0 = pc.acc[PH_JACOBI];
      int sw = jacobi_cols_fast<T>(Wm, ldw_e, Vm, ldv_e, ncol, len, maxsw);
      pc.lap(PH_JACOBI);
      if (threadIdx.x == 0) { pc.acc[6] += sw; pc.acc[7] += 1.0; }   // sweeps, SVD count
      if (threadIdx.x == 0 && need > (size_t)SM_WORK) {               // matrices in global memory
        pc.acc[8] += pc.acc[PH_JACOBI] - jac0;
        pc.acc[9] += 1.0;
      }
      if (sw >= maxsw && threadIdx.x == 0) {
        flag(status, ST_NOCONV);
        if (atomicCAS(&status[1], 0, 1) == 0) {     // first failure: where and how big
          status[2] = blockIdx.x / cc.P; status[3] = k; status[4] = ncol; status[5] = len;
        }
      }
      for (int jj = threadIdx.x; jj < ncol; jj += blockDim.x) {
        T a = (T)0;
        const T* w = Wm + (size_t)jj * ldw_e;
        for (int i = 0; i < len; ++i) a += w[i] * w[i];
        const double sv = (double)sqrt(a) / scl;   // singular value of the unscaled C
        if (!(sv >= 0.0) || isinf(sv)) { s_sig[jj] = -1.0; flag(status, ST_NAN); }   // orders last
        else s_sig[jj] = sv;
      }
      __syncthreads();
      for (int jj = threadIdx.x; jj < ncol; jj += blockDim.x) {
        int rank = 0;
        const double sj = s_sig[jj];
        for (int o = 0; o < ncol; ++o) {
          const double so = s_sig[o];
          rank += (so > sj) || (so == sj && o < jj);
        }
        s_perm[rank] = jj;
      }
      __syncthreads();
      if (threadIdx.x == 0) {
        // smallest r in [1, min(chi, ncol)] with discarded tail <= delta (FP64 tail)
        const int rmax = imin(J.chi, ncol);
        double tail2 = 0.0;
        int rr = rmax;
        for (int p = ncol - 1; p >= 1; --p) {
          const double sv = s_sig[s_perm[p]];
          tail2 += sv * sv;
          s_tau[2 + p] = tail2;                  // tail starting at position p
        }
        for (int q = 1; q <= rmax; ++q) {
          const double t2 = (q < ncol) ? s_tau[2 + q] : 0.0;
          if (sqrt(t2) <= delta) { rr = q; break; }
        }
        if (rr > bond_cap(L, J.dst.cap, k)) { s_bad = 1; rr = bond_cap(L, J.dst.cap, k); }
        s_rank = rr;
        if (J.discard && rr < ncol) atomicAdd(J.discard, s_tau[2 + rr]);   // squared discarded tail
        flops += svd_flops(m, n);
        if (lc && lc->counters) atomicAdd(&lc->counters[2], 1);
      }
      __syncthreads();
      if (s_bad) { if (threadIdx.x == 0) flag(status, ST_CAPACITY); return; }
      r = s_rank;
      // outputs: core k = V^T[:r] (r x n) into dst; US (m x r) into scratch
      for (int idx = threadIdx.x; idx < r * n; idx += blockDim.x) {
        const int jr = idx / n, c = idx % n;
        const int pj = s_perm[jr];
        T v;
        if (trans) {
          v = Vm[(size_t)pj * ldv_e + c];
        } else {
          const T sg = (T)(s_sig[pj] * scl);       // norm of the scaled column
          v = sg > (T)0 ? Wm[(size_t)pj * ldw_e + c] / sg : (T)(c == jr ? 1 : 0);
        }
        out[idx] = v;
      }
      for (int idx = threadIdx.x; idx < m * r; idx += blockDim.x) {
        const int i = idx / r, jr = idx % r;
        const int pj = s_perm[jr];
        US[idx] = trans ? Wm[(size_t)pj * ldw_e + i] * (T)(1.0 / scl)
                        : Vm[(size_t)pj * ldv_e + i] * (T)s_sig[pj];
      }
      if (threadIdx.x == 0) J.dst.ranks[k] = r;
      __syncthreads();
    }
    // ---- sign gauge of the kept singular pairs: each row of V^T gets a
    // positive inner product with the probe weights frac((c+1) g) + 1/4,
    // g = 0.618..., a generic positive vector (rows with tied entries are
    // common in structured fields).  Contracted results do not depend on the
    // gauge; the randomized sample of the next step does.
    __syncthreads();
    {
      const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
      for (int jr = warp; jr < r; jr += nw) {
        T* row = out + (size_t)jr * n;
        double dot = 0.0;
        for (int c = lane; c < n; c += 32) {
          const double x = (double)(c + 1) * 0.6180339887498949;
          dot += (double)row[c] * (x - floor(x) + 0.25);
        }
        for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
        __syncwarp();
        if (dot < 0.0) {
          for (int c = lane; c < n; c += 32) row[c] = -row[c];
          for (int i = lane; i < m; i += 32) US[(size_t)i * r + jr] = -US[(size_t)i * r + jr];
        }
      }
    }
    __syncthreads();
    // ---- spectrum log: (features of the previous step, rank kept now)
    if (J.log != nullptr && lc != nullptr) {
      const int nsv = done ? imin(lsamp, TN_SPEC) : imin(ncol, TN_SPEC);
      if (threadIdx.x == 0 && lc->dataset != nullptr && J.log->valid[k]) {
        const int slot = atomicAdd(lc->dataset_count, 1);
        if (slot < lc->dataset_cap) {
          float* row = lc->dataset + (size_t)slot * (MLP_IN + 1);
          for (int q = 0; q < TN_SPEC; ++q) row[q] = J.log->spec[k][q];
          row[16] = (float)k / (float)L;
          row[17] = lc->step ? fminf((float)(*lc->step) / 1000.f, 1.f) : 0.f;
          row[18] = (float)r / (float)J.chi;
        }
      }
      __syncthreads();
      if (threadIdx.x < TN_SPEC) {
        const double s0 = s_sig[s_perm[0]];
        const double sv = threadIdx.x < nsv ? s_sig[s_perm[threadIdx.x]] : 0.0;
        J.log->spec[k][threadIdx.x] = (s0 > 0.0 && sv > 0.0) ? (float)log10(fmax(sv / s0, 1e-20)) : -20.f;
      }
      if (threadIdx.x == 0) { J.log->label[k] = r; J.log->valid[k] = 1; }
      __syncthreads();
    }
    // C' = Q_{k-1} (2 q_{k-1} x m) * US (m x r)
    const int rows = 2 * s_q[k - 1];
    const T* Qp = scr + J.lay.q_off[k - 1];
    pc.lap(PH_SVD_OUT);
    cta_gemm<T>(rows, r, m, Qp, m, US, r, C, r, false);
    if (threadIdx.x == 0) flops += 2.0 * rows * m * r;
    pc.lap(PH_GEMM_C);
    rnext = r;
  }
  // core 0 = C (1 x 2 x r_1)
  {
    T* out = (T*)J.dst.base;
    for (int idx = threadIdx.x; idx < 2 * rnext; idx += blockDim.x) out[idx] = C[idx];
    if (threadIdx.x == 0) {
      J.dst.ranks[0] = 1;
      J.dst.ranks[L] = 1;
      if (ctr) {
        atomicAdd(&ctr[C_ROUND], flops);
        for (int p = 0; p < PH_COUNT; ++p) atomicAdd(&ctr[C_COUNT + p], pc.acc[p]);
      }
    }
  }
}

// Worker CTA (rank > 0 of a cluster): joins the leader's FP64 Jacobi runs
// until the leader sends the exit command or a wait runs out.
template <typename T>
__device__ void round_worker(const RoundJob& J, int L_arg, ClusterCtx& cc) {
  T* scr = (T*)J.scratch;
  double* Wm = (double*)(scr + J.lay.jw64_off);
  double* Vm = (double*)(scr + J.lay.jv64_off);
  const int L = J.L > 0 ? J.L : L_arg;
  for (;;) {
    if (!cl_sync(cc)) break;
    const volatile ClusterCmd* cmd = (const volatile ClusterCmd*)&cc.sh->cmd;
    const int op = cmd->op, ncol = cmd->ncol, len = cmd->len, maxsw = cmd->maxsw;
    const int m = cmd->m, n = cmd->n, k = cmd->k, sw32 = cmd->sw32;
    const double delta = cmd->delta, scl = cmd->scl;
    __syncthreads();
    if (op == 1) {
      jacobi64_cluster(cc, Wm, jacobi_ld<double>(len), Vm, jacobi_ld<double>(ncol), ncol, len, maxsw);
    } else if (op == 2) {
      int sw = 0;
      bool noconv = false;
      svd64_rows<T>(cc, J, L, k, m, n, scl, delta, maxsw, sw32, &sw, &noconv);
    } else {
      break;
    }
  }
}

// ---------------------------------------------------------------- eigenvectors of a Gram matrix
// The dominant eigenvectors U (m x r, row-major) of the symmetric positive
// semi-definite G (m x m, its upper triangle) for the TT-SVD of a dense field, by
// the centre SVD of the FP64 roundings (G = V diag V^T, V its right vectors) on one
// cluster.  r: the smallest rank whose discarded eigenvalues sum to at most
// max(delta2, the round-off level of the Gram matrix), capped at min(chi, m, ncols).
//
// A single CTA's FP64 Jacobi has two multiply-adds a clock: 25 k cycles a round of 48
// pairs of 96, 10 ms a site.  The cluster's FP32 sweeps in registers and
// refinement by products need ~0.3 ms.
__global__ void __launch_bounds__(RT) gram_eig_kernel(const RoundJob* __restrict__ job, const double* __restrict__ G, int m,
                                                      double* __restrict__ U, int chi, double delta2, int ncols_cap,
                                                      int* r_out, int* status) {
  __shared__ ClusterShared s_cl;
  __shared__ double s_phase[PH_COUNT];
  __shared__ double s_flops;
  __shared__ int s_bad, s_rank;
  extern __shared__ __align__(16) unsigned char smem[];
  ClusterCtx cc;
  const RoundJob& J = *job;
  cl_init(cc, &s_cl, status, J.wait_ns > 0 ? J.wait_ns : 5000000000LL);
  if (cc.rank == 0) {
    double* scr = (double*)J.scratch;
    double* C = scr + J.lay.c_off;
    double* out = (double*)J.dst.base + core_offset(J.L, J.dst.cap, 1);
    const SiteShared sh{(double*)(smem + SM_RED), (double*)(smem + SM_TAU), (double*)(smem + SM_SIG),
                        (int*)smem, &s_bad, &s_rank, &s_flops};
    PhaseClock pc(false, s_phase);
    if (threadIdx.x == 0) { s_bad = 0; s_flops = 0.0; }
    bool bad = false;
    for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
      const int i = e / m, j = e % m;
      const double v = j >= i ? G[e] : G[(size_t)j * m + i];
      C[e] = v;
      bad |= !isfinite(v);
    }
    bad = __syncthreads_or(bad);
    // every non-zero singular value kept; the rank rule of the eigenvalues is below
    const int kept = bad ? 0
                         : svd64_site<double>(J, J.L, 1, C, m, m, out, scr + J.lay.us_off, scr,
                                              (double*)(smem + SM_SMALL), sh, cc, status, nullptr, pc, 0.0);
    if (bad && threadIdx.x == 0) flag(status, ST_NAN);
    __syncthreads();
    if (threadIdx.x == 0) {
      int r = 1;
      if (kept > 0) {
        const int rmax = imin(chi, imin(m, ncols_cap));
        const double* lam = sh.sig;
        const int* perm = sh.perm;
        // eigenvalues below the Gram matrix's round-off level carry no information:
        // that level is the smallest resolvable tail
        const double floor2 = 64.0 * 2.220446049250313e-16 * (double)m * lam[perm[0]];
        const double thr = delta2 > floor2 ? delta2 : floor2;
        double tail = 0.0;
        r = rmax;
        for (int p = m - 1; p >= 1; --p) {
          tail += lam[perm[p]];
          if (!(tail <= thr)) break;
          if (p <= rmax) r = p;
        }
      }
      s_rank = r;
      *r_out = r;
    }
    __syncthreads();
    const int r = s_rank;
    // (a zero singular value's vector is never within r unless G is zero)
    for (int e = threadIdx.x; e < m * r; e += blockDim.x) {
      const int i = e / r, j = e % r;
      U[e] = j < kept ? out[(size_t)j * m + i] : (i == j ? 1.0 : 0.0);
    }
    cl_command(cc, 0, 0, 0, 0);
  } else {
    round_worker<double>(J, J.L, cc);
  }
  cl_exit(cc);
}

// Scratch of the eigenproblems of one TT-SVD (m <= mmax) as a job of one site.
size_t plan_gram_eig(RoundJob& j, int mmax) {
  j = RoundJob{};
  j.L = 3;
  j.n_bits = 1;
  j.chi = mmax;
  j.refine = REFINE_TOP;
  j.dst.cap = mmax;
  size_t off = 0;
  auto al = [&](size_t n) { const size_t o = off; off += (n + 31) & ~(size_t)31; return o; };
  const size_t ld = jacobi_ld<double>(mmax), n = mmax;
  j.lay.c_off = al(n * n);
  j.lay.us_off = al(n * n);
  j.lay.jw64_off = j.lay.jw_off = al(n * ld);
  j.lay.jv64_off = j.lay.jv_off = al(n * ld);
  j.lay.log_off = al(jacobi_reg_log_sweep(imin(mmax, 128)) * JR_LOG_SWEEPS);
  j.lay.j32_off = al((n * jacobi_ld<float>(mmax) + 1) / 2);
  j.lay.vb64_off = al(n * ld + n + CL_MAX * 4);
  j.lay.wide_off = jacobi_reg_fits(mmax, mmax) ? 0 : al((jacobi_wide_floats(mmax, mmax) + 1) / 2);
  j.lay.q_off[0] = al(mps_size(3, mmax));                  // the vectors, as the job's dst
  j.lay.q_off[1] = al(4);                                  // its bonds (ints)
  return j.lay.total = off;
}

// scratch: the doubles that plan_gram_eig returned.  j is copied to the device after this.
void place_gram_eig(RoundJob& j, double* scratch) {
  j.scratch = scratch;
  j.dst.base = scratch + j.lay.q_off[0];
  j.dst.ranks = (int*)(scratch + j.lay.q_off[1]);
}

cudaError_t launch_gram_eig(const RoundJob* d_job, const double* G, int m, double* U, int chi, double delta2,
                            int ncols_cap, int* r_out, int* status, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(gram_eig_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)round_smem_bytes());
  if (e == cudaSuccess) e = cudaFuncSetAttribute(gram_eig_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(RT, 1, 1);
  cfg.dynamicSmemBytes = round_smem_bytes();
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  // the widest cluster that this device can hold (below ~32 columns the exchanges
  // among 16 CTAs would cost more than the work)
  int P = m < 8 ? 1 : m < 32 ? 4 : CL_MAX;
  for (; P > 1; P /= 2) {
    at[0].val.clusterDim.x = P;
    cfg.gridDim = dim3(P, 1, 1);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, gram_eig_kernel, &cfg) == cudaSuccess && n > 0) break;
    cudaGetLastError();
  }
  at[0].val.clusterDim.x = P;
  cfg.gridDim = dim3(P, 1, 1);
  return cudaLaunchKernelEx(&cfg, gram_eig_kernel, d_job, G, m, U, chi, delta2, ncols_cap, r_out, status);
}

template <typename T>
__global__ void __launch_bounds__(RT) round_kernel(const RoundJob* __restrict__ jobs, int L_arg,
                                                   int n_bits_arg, const T* __restrict__ masks_arg,
                                                   const double* __restrict__ scal_arg,
                                                   int* __restrict__ status,
                                                   double* __restrict__ ctr,
                                                   const LearnCtx* __restrict__ lc) {
  __shared__ ClusterShared s_cl;
  ClusterCtx cc;
  const RoundJob& J = jobs[blockIdx.x / cl_size()];
  cl_init(cc, &s_cl, status, J.wait_ns > 0 ? J.wait_ns : 5000000000LL);
  if (cc.rank == 0) {
    round_job_body<T>(J, L_arg, n_bits_arg, masks_arg, scal_arg, status, ctr, lc, cc);
    cl_command(cc, 0, 0, 0, 0);
  } else {
    round_worker<T>(J, L_arg, cc);
  }
  cl_exit(cc);
}

template <typename T>
void launch_round(const RoundJob* d_jobs, int njobs, int L, int n_bits, const T* d_masks,
                  const double* d_scal, int* d_status, cudaStream_t st, double* d_ctr,
                  const LearnCtx* d_learn, int cluster) {
  if (njobs <= 0) return;
  static bool attr_set = false;
  if (!attr_set) {
    cudaFuncSetAttribute(round_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)round_smem_bytes());
    cudaFuncSetAttribute(round_kernel<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    attr_set = true;
  }
  if (cluster <= 1) {
    round_kernel<T><<<njobs, RT, round_smem_bytes(), st>>>(d_jobs, L, n_bits, d_masks, d_scal,
                                                           d_status, d_ctr, d_learn);
    return;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(njobs * cluster, 1, 1);
  cfg.blockDim = dim3(RT, 1, 1);
  cfg.dynamicSmemBytes = round_smem_bytes();
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cluster;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, round_kernel<T>, d_jobs, L, n_bits, d_masks, d_scal, d_status, d_ctr, d_learn);
}

// Resident clusters of P CTAs (1 <= P <= 16) of the rounding kernel on the
// current device; the table is queried once per device.
template <typename T>
int round_cluster_resident(int P) {
  static int cached_dev = -1;
  static int max_active[CL_MAX + 1];
  if (P < 1 || P > CL_MAX) return 0;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (dev != cached_dev) {
    cudaFuncSetAttribute(round_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)round_smem_bytes());
    cudaFuncSetAttribute(round_kernel<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    for (int q = 1; q <= CL_MAX; ++q) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(q, 1, 1);
      cfg.blockDim = dim3(RT, 1, 1);
      cfg.dynamicSmemBytes = round_smem_bytes();
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = q;
      at[0].val.clusterDim.y = 1;
      at[0].val.clusterDim.z = 1;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, round_kernel<T>, &cfg) != cudaSuccess) n = 0;
      max_active[q] = n;
    }
    cudaGetLastError();
    cached_dev = dev;
  }
  return max_active[P];
}

template <typename T>
int round_cluster_size(int njobs, int cap) {
  // the largest cluster at which every job of the launch is resident at once
  // (the FP64 Jacobi scales with the SMs of its cluster)
  for (int P = imin(cap, CL_MAX); P >= 2; --P)
    if (round_cluster_resident<T>(P) >= njobs) return P;
  return 1;
}

template void launch_round<float>(const RoundJob*, int, int, int, const float*, const double*,
                                  int*, cudaStream_t, double*, const LearnCtx*, int);
template void launch_round<double>(const RoundJob*, int, int, int, const double*,
                                   const double*, int*, cudaStream_t, double*, const LearnCtx*, int);
template int round_cluster_size<float>(int, int);
template int round_cluster_size<double>(int, int);
template int round_cluster_resident<float>(int);
template int round_cluster_resident<double>(int);

}  // namespace tn
