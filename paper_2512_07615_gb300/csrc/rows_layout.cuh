// Work area of the FP64 centre SVDs with the rows of the Jacobi matrices split over the
// CTAs of a cluster, and which way such an SVD takes: host and device, so that the
// sizes can be checked without a GPU.
#pragma once

#include "internal.cuh"
#include "jacobi_reg.cuh"
#include "jacobi_wide.cuh"
#include "refine64.cuh"

namespace tn {

static constexpr int SM_SMALL = 41 * 1024;          // bookkeeping part of smem
static constexpr int SM_WORK = 176 * 1024;          // work area in smem

// What is staged before the first exchange of the sweeps: nothing; rows of V and X for
// W = X V (what a refinement hands over); or those and the block of V0^T V0 of the
// Newton-Schulz step (FP32 data).
enum : int { RS_NONE = 0, RS_XV = 1, RS_NS = 2 };

// Layout (bytes, same in every CTA of the cluster) of svd64_rows: the CTA's rows of W
// and of V (FP64), the column norms, each pair's rotation and flag, the exchange
// buffers of the pair inner products and of the column norms, and the singular values,
// order and tails the rank rule reads.  What is staged shares the exchange buffers'
// space (it is read before the first exchange of the sweeps).
struct RowsLayout {
  int lw, lv, npairs, kc;
  size_t wl, vl, nrm, pcw, psw, pf, gl, xb, nbuf, gb, st, xs, st_end, sig, perm, tail, total;
};
__host__ __device__ inline RowsLayout rows_layout(int ncol, int len, int P, int stage) {
  RowsLayout R;
  R.lw = (len + P - 1) / P;
  R.lv = (ncol + P - 1) / P;
  R.npairs = (ncol + 1) / 2;
  R.kc = imax(1, imin(32, 2048 / imax(ncol, 1)));      // staged rows of V per chunk (<= 16 KB)
  size_t o = 0;
  auto rnd16 = [](size_t bytes) { return (bytes + 15) & ~(size_t)15; };
  auto take = [&](size_t bytes) { size_t r = o; o += rnd16(bytes); return r; };
  R.wl = take((size_t)ncol * R.lw * 8);
  R.vl = take((size_t)ncol * R.lv * 8);
  R.nrm = take((size_t)ncol * 8);
  R.pcw = take((size_t)R.npairs * 8);
  R.psw = take((size_t)R.npairs * 8);
  R.pf = take((size_t)R.npairs * 4);
  R.gl = take((size_t)imax(R.npairs, ncol) * 8);
  // shared region: exchange buffers | staging
  const size_t xch = rnd16((size_t)2 * R.npairs * P * 8) + rnd16((size_t)ncol * P * 8);
  const size_t g = stage == RS_NS ? rnd16((size_t)ncol * R.lv * 8) : 0;
  const size_t v = stage == RS_NONE ? 0 : rnd16((size_t)ncol * R.kc * 8);
  const size_t x = stage == RS_NONE ? 0 : rnd16((size_t)R.lw * R.kc * 8);
  const size_t stg = g + v + x;
  const size_t base = take(xch > stg ? xch : stg);
  R.xb = base;
  R.nbuf = base + rnd16((size_t)2 * R.npairs * P * 8);
  R.gb = base;
  R.st = base + g;
  R.xs = R.st + v;
  R.st_end = R.xs + x;
  R.sig = take((size_t)ncol * 8);
  R.perm = take((size_t)ncol * 4);
  R.tail = take((size_t)(ncol + 2) * 8);
  R.total = o;
  return R;
}

// How an SVD starts: >= 0: logged FP32 sweeps in registers, then the refinement; SW_WIDE:
// FP32 sweeps over the cluster, then the refinement; SW_SCRATCH (FP32 data): FP32 sweeps
// whose V is in the job's scratch; SW_PLAIN: FP64 sweeps from V = I.
enum : int { SW_SCRATCH = -1, SW_PLAIN = -2, SW_WIDE = -3 };
__host__ __device__ inline int rows_stage(int eb, int sw32) {
  return eb == 4 ? RS_NS : sw32 >= 0 || sw32 == SW_WIDE ? RS_XV : RS_NONE;
}

// Centre matrices whose sweeps the leader runs alone, as a cluster of one: the exchanges of a
// round (~3 k of its 9 k cycles) cost more than the other CTAs' FP64 units bring for a
// few columns, and below ~16 columns the refinement of FP64 data costs more than
// the sweeps.  One FP64 step of a 16^3 channel 42.8 -> 36.8 ms, 16^3 wall terms of 18 jobs 7.74 ->
// 7.04, 32^3 ones 14.5 -> 14.7 (three medians of 15 each, 0.3 % apart).  Ten channel steps with up
// to 12 columns 57.9 ms, 16 56.6, 24 the same, 32 worse for the roundings.  FP32 data
// are refined from RF_MIN columns on (16 columns alone: 128^3 sums 55 -> 61 ms).
static constexpr int SOLO_LEN = 128;
__host__ __device__ constexpr int solo_cols(int eb) { return eb == 8 ? 16 : RF_MIN - 1; }

// The way of an SVD of ncol columns of len entries (ncol <= len) of elements of eb bytes on
// a cluster of P > 1 CTAs; refine: the job has the refinement's scratch.
struct Svd64Path {
  bool solo;               // the leader's FP64 sweeps alone
  bool rows;               // rows split over the cluster (else the matrices in global memory)
  bool reg, wide;          // FP32 sweeps and refinement: in a CTA's registers, over the cluster
  bool plain;              // FP64 sweeps from V = I
};
__host__ __device__ inline Svd64Path svd64_path(int ncol, int len, int P, int eb, bool refine) {
  Svd64Path p;
  p.solo = ncol <= solo_cols(eb) && len <= SOLO_LEN;
  p.plain = p.solo || ncol < RF_MIN;
  p.rows = !p.solo && rows_layout(ncol, len, P, rows_stage(eb, SW_PLAIN)).total <= (size_t)SM_WORK;
  // the sweeps may have to finish what the refinement starts: its staging has to fit too
  const bool ref = p.rows && !p.plain && refine && rf_bytes(ncol, len, P) <= (size_t)SM_WORK &&
                   rows_layout(ncol, len, P, rows_stage(eb, SW_WIDE)).total <= (size_t)SM_WORK;
  p.reg = ref && jacobi_reg_fits(ncol, len);
  p.wide = ref && !p.reg && jacobi_wide_fits(ncol, len, P);
  return p;
}

}  // namespace tn
