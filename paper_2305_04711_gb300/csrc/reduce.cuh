// reduce.cuh -- deterministic dot products of the Krylov iteration and the
// per-right-hand-side scalars that follow from them (see krylov.cu).
#pragma once

#include <stdint.h>

#include "cpm_internal.cuh"

constexpr int NQMAX = 4;   // dot products reduced by one kernel at most

// per right-hand side scalar slots
enum {
  S_RHO_OLD = 0, S_ALPHA, S_OMEGA, S_RHO, S_BETA, S_ACTIVE, S_RESTART, S_NRESTART, S_FN2, S_RN2, S_BROKE,
  S_BEST, S_STALL, S_STOPPED, S_RN2_0, S_ITERS, S_RH2, S_SEED, NSC
};

enum { ST_OUT = 0, ST_INIT, ST_ALPHA, ST_OMEGA, ST_XR };

struct Red {
  double *part;      // [G][NQMAX][nrhs] block partials
  unsigned *ticket;  // arrival counter (reset by the last block)
  double *sc;        // [nrhs][NSC]
  double *out;       // [NQMAX][nrhs] reduced dot products (ST_OUT / ST_INIT)
  int nrhs;
};

struct Conv {
  double tol;     // relative tolerance on the iterated system's residual
  double stall;   // iterations without the residual halving before giving up
  float mix;      // shadow = r o (1 + mix u) (shadow 0; mix 0: the classical rhat = r)
  int shadow;     // 0: rhat from r as above; 1: rhat = u, independent of r
  unsigned seed;  // of the hash u (kept as S_SEED from the initial residual on: captured iterations serve any)
};

namespace {

// a fixed hash u(i, c, seed) in [-1, 1]
__device__ __forceinline__ float hash_unit(int64_t i, int c, unsigned seed) {
  uint64_t k = (uint64_t)i * 0x9E3779B97F4A7C15ull + (uint64_t)c * 0xD1B54A32D192ED03ull +
               (uint64_t)seed * 0x94D049BB133111EBull;
  k ^= k >> 31; k *= 0xBF58476D1CE4E5B9ull; k ^= k >> 29;
  return (float)((k >> 40) & 0xFFFFFF) * (2.0f / 16777215.0f) - 1.0f;
}

// The shadow residual rhat of a (re)start, given the residual r there.
// rhat = r is the classical choice, but when r is supported on few rows (a
// right-hand side on the BC rows only) A r lives elsewhere and (rhat, A r) = 0:
// the first step breaks down.  A random rhat (shadow 1) meets every row; its
// (rhat, r) ~ |rhat| |r| / sqrt(N) is still far above the rounding of the dot
// products.  `seed` is the hash's seed plus the restarts so far, which select a fresh
// hash after a near-breakdown.
__device__ __forceinline__ float shadow_of(const Conv &cv, int64_t i, int c, float r, unsigned seed) {
  if (cv.shadow == 1) return hash_unit(i, c, seed);
  if (cv.mix == 0.0f) return r;
  return r * (1.0f + cv.mix * hash_unit(i, c, 0u));
}
__device__ __forceinline__ double shadow_of(const Conv &cv, int64_t i, int c, double r, unsigned seed) {
  if (cv.shadow == 1) return (double)hash_unit(i, c, seed);
  if (cv.mix == 0.0f) return r;
  return r * (1.0 + (double)cv.mix * (double)hash_unit(i, c, 0u));
}

// ---- deterministic block reduction -----------------------------------------
// Thread t of a block of B owns column c = t % nrhs and rows sub, sub + rows_per,
// ... of the block's share (sub = t / nrhs, rows_per = B / nrhs).
template <int NQ, int B>
__device__ __forceinline__ bool block_publish(const double (&acc)[NQ], const Red &R) {
  __shared__ double sh[NQ][B];
  __shared__ bool s_last;
  const int t = threadIdx.x, nrhs = R.nrhs;
  if (nrhs == 1) {
    // one warp per product adds the block's B values, 32 at a time.  Every FP64
    // instruction of a warp takes the SM's FP64 pipe for 16 clocks however many
    // lanes it has, so shuffles in all of a block's warps (5 each) cost a small
    // problem more than its elements did.
#pragma unroll
    for (int q = 0; q < NQ; ++q) sh[q][t] = acc[q];
    __syncthreads();
    const int w = t >> 5, lane = t & 31;
    if (w < NQ) {
      double s0 = 0.0, s1 = 0.0;
#pragma unroll
      for (int k = 0; k < B / 32; k += 2) { s0 += sh[w][k * 32 + lane]; s1 += sh[w][k * 32 + 32 + lane]; }
      s0 += s1;
#pragma unroll
      for (int off = 16; off; off >>= 1) s0 += __shfl_xor_sync(0xffffffffu, s0, off);
      if (lane == 0) R.part[(int64_t)blockIdx.x * NQMAX + w] = s0;
    }
  } else if (nrhs < 32 && (32 % nrhs) == 0) {
    // lanes with equal column combine by xor shuffles, then the warps in order
    double v[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) v[q] = acc[q];
    for (int off = 16; off >= nrhs; off >>= 1)
#pragma unroll
      for (int q = 0; q < NQ; ++q) v[q] += __shfl_xor_sync(0xffffffffu, v[q], off);
    const int lane = t & 31, w = t >> 5;
    if (lane < nrhs)
#pragma unroll
      for (int q = 0; q < NQ; ++q) sh[q][w * nrhs + lane] = v[q];
    __syncthreads();
    if (t < nrhs)
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        double s = 0.0;
        for (int k = 0; k < B / 32; ++k) s += sh[q][k * nrhs + t];
        R.part[((int64_t)blockIdx.x * NQMAX + q) * nrhs + t] = s;
      }
  } else {
    const int rows_per = B / nrhs;
#pragma unroll
    for (int q = 0; q < NQ; ++q) sh[q][t] = acc[q];
    __syncthreads();
    if (t < nrhs)
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        double s = 0.0;
        for (int k = 0; k < rows_per; ++k) s += sh[q][k * nrhs + t];
        R.part[((int64_t)blockIdx.x * NQMAX + q) * nrhs + t] = s;
      }
  }
  __threadfence();
  __syncthreads();
  if (t == 0) s_last = (atomicAdd(R.ticket, 1u) == gridDim.x - 1);
  __syncthreads();
  return s_last;
}

__device__ void stage_finish(int stage, const Red &R, const Conv &cv, int c, const double *d) {
  double *s = R.sc + c * NSC;
  if (stage == ST_OUT) return;
  if (stage == ST_INIT) {
    const double fn2 = d[1] > 0.0 ? d[1] : 1.0;
    s[S_FN2] = fn2;
    s[S_RN2] = d[0]; s[S_BEST] = d[0]; s[S_RN2_0] = d[0];
    // (the scale of the breakdown test: |rhat|^2; a later random shadow has the same)
    s[S_RH2] = (cv.shadow == 0 && cv.mix == 0.0f) ? d[0] : d[3];
    s[S_RHO] = d[2]; s[S_RHO_OLD] = 1.0; s[S_ALPHA] = 1.0; s[S_OMEGA] = 1.0; s[S_BETA] = 0.0;
    s[S_RESTART] = 0.0; s[S_NRESTART] = 0.0; s[S_BROKE] = 0.0; s[S_STALL] = 0.0; s[S_STOPPED] = 0.0;
    s[S_ITERS] = 0.0;
    s[S_SEED] = (double)cv.seed;
    const bool fin = isfinite(d[0]);
    s[S_ACTIVE] = (!fin || sqrt(d[0]) <= cv.tol * sqrt(fn2)) ? 0.0 : 1.0;
    if (!fin) s[S_STOPPED] = 1.0;
    return;
  }
  if (s[S_ACTIVE] == 0.0) return;
  if (stage == ST_ALPHA) {
    if (d[0] == 0.0 || !isfinite(d[0])) { s[S_BROKE] = 1.0; s[S_ACTIVE] = 0.0; return; }
    s[S_ALPHA] = s[S_RHO] / d[0];
    return;
  }
  if (stage == ST_OMEGA) {
    const double om = (d[1] > 0.0) ? d[0] / d[1] : 0.0;
    s[S_OMEGA] = om;
    if (om == 0.0 || !isfinite(om)) { s[S_BROKE] = 1.0; s[S_ACTIVE] = 0.0; }
    return;
  }
  // ST_XR, d = (r, r), (rhat, r), (rhat', r) with rhat' the shadow a restart would
  // take: residual bookkeeping, then rho and beta of the next iteration
  s[S_ITERS] += 1.0;
  const double rn2 = d[0];
  s[S_RN2] = rn2;
  if (!isfinite(rn2) || rn2 > 1e16 * s[S_BEST]) { s[S_STOPPED] = 1.0; s[S_ACTIVE] = 0.0; return; }
  if (sqrt(rn2) <= cv.tol * sqrt(s[S_FN2])) { s[S_ACTIVE] = 0.0; return; }
  if (rn2 < 0.25 * s[S_BEST]) { s[S_BEST] = rn2; s[S_STALL] = 0.0; }
  else {
    s[S_STALL] += 1.0;
    if (s[S_STALL] > cv.stall) { s[S_STOPPED] = 1.0; s[S_ACTIVE] = 0.0; return; }
  }
  double rho = d[1];
  s[S_RESTART] = 0.0;
  // |rho| <= 1e-28 |rhat| |r|, looked at closely only where the larger mean of the
  // two squares does not already rule it out (the square roots are long)
  if (!(fabs(rho) > 1e-28 * (s[S_RH2] + rn2)) &&
      (fabs(rho) <= 1e-28 * sqrt(s[S_RH2]) * sqrt(rn2) || rho == 0.0)) {
    // restart from a new shadow residual: p = r, rho = (rhat', r)
    const double fresh = (cv.shadow == 0 && cv.mix == 0.0f) ? rn2 : d[2];
    if (cv.shadow == 0 && cv.mix == 0.0f) s[S_RH2] = rn2;
    s[S_RESTART] = 1.0;
    s[S_NRESTART] += 1.0;
    if (s[S_NRESTART] > 20.0) { s[S_BROKE] = 1.0; s[S_ACTIVE] = 0.0; return; }
    rho = fresh;
    s[S_RHO] = 1.0; s[S_ALPHA] = 1.0; s[S_OMEGA] = 1.0;
  }
  s[S_BETA] = (rho / s[S_RHO]) * (s[S_ALPHA] / s[S_OMEGA]);
  s[S_RHO_OLD] = s[S_RHO];
  s[S_RHO] = rho;
}

// the last block: sum the partials in block order (a warp per (q, c), lanes
// strided over the blocks, then an xor-shuffle tree, identical in every lane)
template <int NQ, int B>
__device__ void finish_reduce(int stage, const Red &R, const Conv &cv) {
  __shared__ double sd[NQMAX][256];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5, nrhs = R.nrhs;
  const int G = gridDim.x;
  __threadfence();
  for (int pr = w; pr < NQ * nrhs; pr += B / 32) {
    const int q = pr / nrhs, c = pr - q * nrhs;
    double s = 0.0;
    for (int b = lane; b < G; b += 32) s += __ldcg(R.part + ((int64_t)b * NQMAX + q) * nrhs + c);
#pragma unroll
    for (int off = 16; off; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) sd[q][c] = s;
  }
  __syncthreads();
  if (t < nrhs) {
    double d[NQMAX] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int q = 0; q < NQ; ++q) d[q] = sd[q][t];
    if (stage == ST_OUT || stage == ST_INIT)
#pragma unroll
      for (int q = 0; q < NQ; ++q) R.out[q * nrhs + t] = d[q];
    stage_finish(stage, R, cv, t, d);
  }
  if (t == 0) *R.ticket = 0u;
}

}  // namespace

// dot products that a product v = A u of one right-hand side can take along where
// it writes v: stage ST_ALPHA (w, v); ST_OMEGA (v, u) and (v, v)
template <typename T>
struct FusedDot {
  Red R;
  Conv cv;
  int stage;
  const T *w;
  bool done;  // set by the product that took them
};
