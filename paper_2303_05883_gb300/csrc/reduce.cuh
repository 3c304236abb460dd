// Deterministic grid reductions fused into the producing kernel, and the
// device-side BiCGStab scalar updates they feed.
//
// Each block reduces its per-thread partial sums (FP64) with a fixed
// shuffle tree, writes one partial per block, and the last block to finish
// (atomic ticket, no waiting) sums all partials in a fixed order and runs a
// finalizer.  The result is bit-reproducible for a given launch shape, which
// is what makes a solve give the same answer alone and in a mix of requests.
//
// What bounds it is latency on the FP64 pipe (2 lanes a clock): a launch with
// three dot products took 7.6 us where the same launch without took 2.4, 27 us
// with twelve right-hand sides.  Hence the merged warp sums, one value a lane
// over the partials, a warp for each right-hand side, and nothing at all once
// every solve has ended.  Solves without and with these: 8^4 4.94 -> 3.51 ms
// (one division a quotient; two, as the range of the quotients needs, add 0.05),
// 32^3 x 64 173 -> 167 ms, Moebius 16^3 x 32 x 16 202 -> 198 ms.
#pragma once

#include "common.cuh"

namespace bridge {

enum FinMode {
  FIN_NONE = 0,
  FIN_STORE = 1,
  FIN_ALPHA = 2,
  FIN_OMEGA = 3,
  FIN_RHO = 4,
  FIN_INIT = 5,
  FIN_CG_INIT = 6,   // s[0] = |b|^2 of the CG system
  FIN_CG_ALPHA = 7,  // s[0] = |D p|^2
  FIN_CG_BETA = 8    // s[0] = |r|^2 after the update
};

struct RedArgs {
  double* partials = nullptr;       // [nrhs][nblk][4]
  unsigned int* counter = nullptr;  // one ticket counter per launch site, reset by the last block
  BiCGScalars* sc = nullptr;        // per right-hand side (may be null)
  CGScalars* cg = nullptr;          // per right-hand side, CG finalizers (may be null)
  double* result = nullptr;         // [nrhs][4] for FIN_STORE
  int fin = FIN_NONE;               // FinMode
  int check_done = 0;               // blocks of a right-hand side whose solve has ended skip their work
};

// Complex helpers on the scalar struct (FP64, one thread).
struct zc {
  double r, i;
};
__device__ __forceinline__ zc zmul(zc a, zc b) { return {a.r * b.r - a.i * b.i, a.r * b.i + a.i * b.r}; }
// Two divisions, not one reciprocal: |b|^2 goes down to where 1 / |b|^2 is
// infinite and the quotients are not (|b|^2 < 5.6e-309).
__device__ __forceinline__ zc zdiv(zc a, zc b) {
  const double d = b.r * b.r + b.i * b.i;
  return {(a.r * b.r + a.i * b.i) / d, (a.i * b.r - a.r * b.i) / d};
}
__device__ __forceinline__ double zabs2(zc a) { return a.r * a.r + a.i * a.i; }

// BiCGStab (van der Vorst 1992; the solver of Sec. 3) scalar recurrences.
__device__ inline void finalize(const RedArgs& ra, int rhs, const double s[4]) {
  BiCGScalars* q = ra.sc ? ra.sc + rhs : nullptr;
  switch (ra.fin) {
    case FIN_STORE:
#pragma unroll
      for (int k = 0; k < 4; ++k) ra.result[rhs * 4 + k] = s[k];
      break;
    case FIN_INIT: {  // s[0] = |b|^2 ; x = 0, r = rhat = p = b
      q->b2 = s[0];
      q->r2 = s[0];
      q->rhat2 = s[0];
      q->rho_r = s[0];
      q->rho_i = 0.0;
      q->alpha_r = q->omega_r = 1.0;
      q->alpha_i = q->omega_i = 0.0;
      q->beta_r = q->beta_i = 0.0;
      q->iter = 0;
      q->tol2 = q->tol2 * s[0];  // tol^2 was staged in tol2 by the host
      q->done = (s[0] == 0.0 || s[0] <= q->tol2) ? CONVERGED : RUNNING;
      break;
    }
    case FIN_ALPHA: {  // s = <rhat, v>
      if (q->done) break;
      zc rv = {s[0], s[1]};
      if (!(zabs2(rv) > 0.0) || !isfinite(s[0]) || !isfinite(s[1])) {
        q->done = BREAKDOWN;
        break;
      }
      zc a = zdiv(zc{q->rho_r, q->rho_i}, rv);
      q->alpha_r = a.r;
      q->alpha_i = a.i;
      break;
    }
    case FIN_OMEGA: {  // s = <t, s>, |t|^2
      if (q->done) break;
      if (s[2] > 0.0) {
        q->omega_r = s[0] / s[2];
        q->omega_i = s[1] / s[2];
      } else {
        q->omega_r = q->omega_i = 0.0;
      }
      break;
    }
    case FIN_RHO: {  // s = <rhat, r>, |r|^2 after x, r were updated
      if (q->done) break;
      q->iter += 1;
      q->r2 = s[2];
      zc rho_new = {s[0], s[1]};
      if (!isfinite(s[2])) {
        q->done = BREAKDOWN;
      } else if (s[2] <= q->tol2) {
        q->done = CONVERGED;
      } else if (q->omega_r == 0.0 && q->omega_i == 0.0) {
        q->done = BREAKDOWN;
      } else if (zabs2(rho_new) < 1e-60 * q->rhat2 * s[2]) {
        q->done = BREAKDOWN;
      } else {
        // (rho_new / rho) (alpha / omega), the two quotients in parallel
        zc b = zmul(zdiv(rho_new, zc{q->rho_r, q->rho_i}), zdiv(zc{q->alpha_r, q->alpha_i}, zc{q->omega_r, q->omega_i}));
        q->beta_r = b.r;
        q->beta_i = b.i;
        q->rho_r = rho_new.r;
        q->rho_i = rho_new.i;
        if (q->iter >= q->max_iter) q->done = MAXITER;
      }
      break;
    }
    case FIN_CG_INIT: {  // r = p = b, x = 0
      CGScalars* g = ra.cg + rhs;
      g->b2 = s[0];
      g->rr = s[0];
      g->alpha = g->beta = 0.0;
      g->iter = 0;
      g->tol2 = g->tol2 * s[0];
      g->done = !isfinite(s[0]) ? BREAKDOWN : (s[0] == 0.0 || s[0] <= g->tol2) ? CONVERGED : RUNNING;
      break;
    }
    case FIN_CG_ALPHA: {
      CGScalars* g = ra.cg + rhs;
      if (g->done) break;
      g->pq = s[0];
      if (!(s[0] > 0.0) || !isfinite(s[0]))
        g->done = BREAKDOWN;
      else
        g->alpha = g->rr / s[0];
      break;
    }
    case FIN_CG_BETA: {
      CGScalars* g = ra.cg + rhs;
      if (g->done) break;
      g->iter += 1;
      if (!isfinite(s[0])) {
        g->done = BREAKDOWN;
      } else {
        g->beta = s[0] / g->rr;
        g->rr = s[0];
        if (s[0] <= g->tol2)
          g->done = CONVERGED;
        else if (g->iter >= g->max_iter)
          g->done = MAXITER;
      }
      break;
    }
    default:
      break;
  }
}

// Sums of NV values over the 32 lanes of a warp, in a fixed order; value k ends
// in lane k * 32 / W, W = NV rounded up to a power of two.  Each exchange halves
// the values a lane carries before it halves the lanes: 6 additions for three
// values (5 for two) instead of 15 (10).  An FP64 addition holds a quarter of
// the SM's FP64 pipe for 64 clocks whatever lanes it is for, so these counts are
// the length of a reduction's tail.
template <int NV>
__device__ __forceinline__ double warp_sum(const double v[NV]) {
  const int lane = threadIdx.x & 31;
  double a;
  int off = 16;
  if (NV == 1) {
    a = v[0];
  } else if (NV == 2) {
    const bool hi = lane & 16;
    const double got = __shfl_xor_sync(0xffffffffu, hi ? v[0] : v[1], 16);
    a = (hi ? v[1] : v[0]) + got;
    off = 8;
  } else {
    const bool hi = lane & 16;
    // low half: values 0, 1; high half: value 2 (and 3)
    const double v3 = NV > 3 ? v[NV - 1] : 0.0;
    const double b0 = (hi ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, hi ? v[0] : v[2], 16);
    const double b1 = (hi ? v3 : v[1]) + __shfl_xor_sync(0xffffffffu, hi ? v[1] : v3, 16);
    const bool odd = lane & 8;
    a = (odd ? b1 : b0) + __shfl_xor_sync(0xffffffffu, odd ? b0 : b1, 8);
    off = 4;
  }
  for (; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
  return a;
}
template <int NV>
__host__ __device__ constexpr int warp_sum_lanes() { return NV == 1 ? 32 : NV == 2 ? 16 : 8; }

// Sum v[0..NV) over the block, value k into thread k (fixed order); needs all
// threads of the block.
template <int NV>
__device__ __forceinline__ double block_sum_spread(const double v[NV], double (*sh)[4]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  const double a = warp_sum<NV>(v);
  constexpr int W = warp_sum_lanes<NV>();
  __syncthreads();
  if (lane % W == 0 && lane / W < NV) sh[warp][lane / W] = a;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x < NV)
    for (int w = 0; w < nw; ++w) t += sh[w][threadIdx.x];
  return t;
}

// The same with all sums in thread 0's v.
template <int NV>
__device__ __forceinline__ void block_sum(double v[NV], double (*sh)[4]) {
  const double t = block_sum_spread<NV>(v, sh);
  if (threadIdx.x < 32)
#pragma unroll
    for (int k = 0; k < NV; ++k) v[k] = __shfl_sync(0xffffffffu, t, k);
}

// Block partial of one right-hand side -> its slot in ra.partials, written
// before thread 0 goes on.  Must be reached by every thread of the block.
template <int NV>
__device__ __forceinline__ void block_partial(const RedArgs& ra, int rhs, int sb, int nblk, const double v[NV]) {
  __shared__ double sh[32][4];
  const double t = block_sum_spread<NV>(v, sh);
  if (threadIdx.x < 32) {
    if (threadIdx.x < NV) ra.partials[((long)rhs * nblk + sb) * 4 + threadIdx.x] = t;
    __syncwarp();
  }
}

// Lane l of a group of `threads` sums value l % G of the partials l / G, l / G +
// threads / G, ... (G = NV rounded up to a power of two: one value a lane); eight
// loads in flight before their additions, which are in a fixed order.
template <int NV>
__host__ __device__ constexpr int partial_group() { return NV == 1 ? 1 : NV == 2 ? 2 : 4; }
template <int NV>
__device__ __forceinline__ double partials_sum(const double* p, int nblk, int l, int threads) {
  constexpr int G = partial_group<NV>();
  const int k = l % G, step = threads / G;
  double a = 0.0;
  if (k < NV)
    for (int b = l / G; b < nblk; b += 8 * step) {
      double t[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) t[u] = b + u * step < nblk ? __ldcg(p + 4 * (b + u * step) + k) : 0.0;
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (b + u * step < nblk) a += t[u];
    }
  return a;
}

// After this block's partials are written (block_partial, or its writers and a
// barrier): thread 0 takes a ticket behind a fence, which covers what the
// barrier ordered before it; the last block of the grid sums every right-hand
// side's partials in a fixed order and runs the finalizer -- the whole block
// for one right-hand side with many partials, else a warp for each right-hand
// side.  Must be reached by every thread of every block.
template <int NV>
__device__ void grid_finish(const RedArgs& ra, int nblk, int nrhs) {
  __shared__ double sh[32][4];
  __shared__ int is_last;
  if (threadIdx.x == 0) {
    __threadfence();
    is_last = (atomicAdd(ra.counter, 1u) == gridDim.x - 1);
  }
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (nrhs == 1 && nblk > 32 && nw > 1) {
    double a = partials_sum<NV>(ra.partials, nblk, threadIdx.x, nw * 32);
#pragma unroll
    for (int off = partial_group<NV>(); off < 32; off <<= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
    if (lane < NV) sh[warp][lane] = a;
    __syncthreads();
    if (warp == 0) {
      a = 0.0;
      if (lane < NV)
        for (int w = 0; w < nw; ++w) a += sh[w][lane];
      double s[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) s[k] = k < NV ? __shfl_sync(0xffffffffu, a, k) : 0.0;
      if (lane == 0) finalize(ra, 0, s);
    }
  } else {
    for (int r = warp; r < nrhs; r += nw) {
      double a = partials_sum<NV>(ra.partials + (long)r * nblk * 4, nblk, lane, 32);
#pragma unroll
      for (int off = partial_group<NV>(); off < 32; off <<= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
      double s[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) s[k] = k < NV ? __shfl_sync(0xffffffffu, a, k) : 0.0;
      if (lane == 0) finalize(ra, r, s);
    }
  }
  if (threadIdx.x == 0) *ra.counter = 0u;
}

// Block partial -> global partial; the last block reduces and finalizes.
// Must be reached by every thread of every block.
template <int NV>
__device__ void reduce_finalize(const RedArgs& ra, int rhs, int sb, int nblk, int nrhs, const double v[NV]) {
  block_partial<NV>(ra, rhs, sb, nblk, v);
  grid_finish<NV>(ra, nblk, nrhs);
}

// Whether every right-hand side's solve has ended: then a launch queued behind
// the end returns without reducing anything.  All blocks of a launch agree (the
// flags change only in a launch's last block, after all others took a ticket).
__device__ __forceinline__ bool all_finished(const RedArgs& ra, int nrhs) {
  if (!ra.check_done) return false;
  for (int r = 0; r < nrhs; ++r)
    if ((ra.sc == nullptr || ra.sc[r].done == RUNNING) && (ra.cg == nullptr || ra.cg[r].done == RUNNING)) return false;
  return ra.sc != nullptr || ra.cg != nullptr;
}

}  // namespace bridge
