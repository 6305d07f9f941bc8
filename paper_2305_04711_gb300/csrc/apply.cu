// apply.cu -- the matrix-free CPM operator on the device.
//
// Sec. 5.4 computes v = A u in four passes with stored E and L:
//   a = E u;  b = (L - diag L) a;  a = diag(L) u;  v = m u + n a + n b.
// Here E and L are never stored for the bulk of the rows: each PDE row keeps
// only the packed location of its interpolation stencil's base node and the
// fractional position t (FP64 and FP32 copies).  Two steps per product:
//   gather : a_i = (E u - u)_i for PDE rows (tile.cu up to 15 columns, cells.cu
//            from 16), rows near an interior boundary with the crossing-test
//            flips (Eq. 10) added as a sparse correction (small FP32 batches of
//            2D bands: a thread per row and column here, flips included);
//   combine: the FD stencil of the PDE rows and the BC rows
//            v_alpha = sum_beta B_alpha,beta u_beta,
// where a neighbour flipped to a BC DOF reads u of that DOF (E rows of BC DOFs
// are the identity).
#include <mutex>

#include "apply.cuh"
#include "cpm_internal.cuh"
#include "fixed.cuh"

namespace {

// ---- combine -----------------------------------------------------------------
// With a holding the extension defects cs sum_j w_j (u_j - u_k) (the gather's
// difference form), a PDE row is
//   v_i = R { m cs u_i + (n/h^2) [ sum_{k PDE} (a_k + cs u_k - cs u_i)
//             + sum_{k BC} (u_k - cs u_i) - n_missing cs u_i ] }.
// FP32 sums the terms as they stand.  In FP64 the dozen additions a row are 12 of
// the FP64 pipe's clocks per SM, which held the kernel at 82 % of that pipe (126 us
// on the sphere at h = 1/128); there the u and the a differences are summed as
// integers of one exponent each (fixed.cuh).  Neighbouring u within 6 binary
// orders are represented exactly, so sum (u_k - u_i) is exact on smooth fields
// and otherwise off by 2^-58 of the largest value, where each FP64 difference is
// rounded at 2^-53 of itself.
struct CombineArgs {
  int64_t NS, N;
  int nfd;
  const int32_t *nbr8;  // [NS][8] FD neighbour columns, flipped near curves
  const int32_t *bc_cnt, *bc_col;
};

template <typename T>
struct CombineScale {
  T m, c;    // R m cs, R n / h^2
  T cs;
};

__device__ __forceinline__ void load_nbrs(const int32_t *nbr8, int64_t i, int32_t (&nb)[6]) {
  const int4 n0 = __ldg(reinterpret_cast<const int4 *>(nbr8 + i * 8));
  const int2 n1 = __ldg(reinterpret_cast<const int2 *>(nbr8 + i * 8 + 4));
  nb[0] = n0.x; nb[1] = n0.y; nb[2] = n0.z; nb[3] = n0.w; nb[4] = n1.x; nb[5] = n1.y;
}

// one row, one column: u0 = u_i; uk, ak the values at the neighbours nb (anything
// where nb < 0, ak anything where the neighbour is a BC DOF).  ALL: all six are
// PDE DOFs, as in every row away from curves and from the band's edge
template <bool ALL>
__device__ __forceinline__ float combine_row(const CombineScale<float> &S, int NS, int nfd, const int32_t (&nb)[6],
                                             float u0, const float (&uk)[6], const float (&ak)[6]) {
  const float ui = S.cs * u0;
  float s = 0.0f;
  int present = 0;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    if (!ALL && nb[k] < 0) continue;
    ++present;
    s += (ALL || nb[k] < NS) ? ak[k] + (S.cs * uk[k] - ui) : uk[k] - ui;
  }
  if (ALL) return S.m * u0 + S.c * s;
  return S.m * u0 + S.c * (s - (float)(nfd - present) * ui);
}

__device__ __forceinline__ double combine_row_plain(const CombineScale<double> &S, int NS, int nfd,
                                                 const int32_t (&nb)[6], double u0, const double (&uk)[6],
                                                 const double (&ak)[6]) {
  const double ui = S.cs * u0;
  double s = 0.0;
  int present = 0;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    if (nb[k] < 0) continue;
    ++present;
    s += (nb[k] < NS) ? ak[k] + (S.cs * uk[k] - ui) : uk[k] - ui;
  }
  return S.m * u0 + S.c * (s - (nfd - present) * ui);
}

template <bool ALL>
__device__ __forceinline__ double combine_row(const CombineScale<double> &S, int NS, int nfd,
                                              const int32_t (&nb)[6], double u0, const double (&uk)[6],
                                              const double (&ak)[6]) {
  unsigned tu = fx_key(u0), ta = 0;
  int npde = 0, nbc = 0;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    if (ALL || (nb[k] >= 0 && nb[k] < NS)) {
      ++npde;
      tu = max(tu, fx_key(uk[k]));
      ta = max(ta, fx_key(ak[k]));
    }
    if (!ALL) nbc += nb[k] >= NS;
  }
  const int eu = (int)(tu >> 20), ea = (int)(ta >> 20);
  const int ecs = ((__double2hiint(S.cs) >> 20) & 0x7FF) + eu - 1081;
  if (fx_ok(tu) && fx_ok(ta) && (tu == 0u || (ecs >= 1 && ecs <= 2046))) {
    // 12 values below 2^59: no overflow
    long long su = 0, sa = 0;
    const long long x0 = fx_of(u0, eu, 6);
#pragma unroll
    for (int k = 0; k < 6; ++k)
      if (ALL || (nb[k] >= 0 && nb[k] < NS)) {
        su += fx_of(uk[k], eu, 6) - x0;
        sa += fx_of(ak[k], ea, 6);
      }
    double s = (ta == 0u) ? 0.0 : (double)sa * fx_scale(1.0, ea - 1081);
    if (tu != 0u) s = fma((double)su, fx_scale(S.cs, eu - 1081), s);
    if (!ALL && nbc) {
#pragma unroll
      for (int k = 0; k < 6; ++k)
        if (nb[k] >= NS) s += uk[k] - S.cs * u0;
    }
    const int miss = ALL ? 0 : nfd - npde - nbc;
    if (miss) s -= miss * (S.cs * u0);
    return fma(S.c, s, S.m * u0);
  }
  return combine_row_plain(S, NS, nfd, nb, u0, uk, ak);
}

template <typename T>
__device__ __forceinline__ T combine_element(const CombineArgs &A, const CombineScale<T> &S,
                                             const T *__restrict__ bc_val, const T *__restrict__ u,
                                             const T *__restrict__ a, int64_t i, int r, int64_t ld) {
  if (i < A.NS) {
    int32_t nb[6];
    load_nbrs(A.nbr8, i, nb);
    T uk[6], ak[6];
    const T u0 = __ldg(u + i * ld + r);
#pragma unroll
    for (int k = 0; k < 6; ++k) {  // absent ones read the row's own: all 13 loads start at once
      const int64_t c = (nb[k] >= 0) ? nb[k] : i, ca = (c < A.NS) ? c : i;
      uk[k] = __ldg(u + c * ld + r);
      ak[k] = __ldg(a + ca * ld + r);
    }
    return combine_row<false>(S, (int)A.NS, A.nfd, nb, u0, uk, ak);
  }
  const int64_t al = i - A.NS;
  const int cnt = __ldg(A.bc_cnt + al);
  T s = T(0);
  for (int e = 0; e < cnt; ++e) {
    const int32_t c = __ldg(A.bc_col + al * CPM_BC_STRIDE + e);
    s += __ldg(bc_val + al * CPM_BC_STRIDE + e) * (__ldg(u + (int64_t)c * ld + r) * ((c < A.NS) ? S.cs : T(1)));
  }
  return s;
}

// a few columns: one thread per element
template <typename T>
__global__ void __launch_bounds__(256, (sizeof(T) == 8) ? 6 : 8)
    combine_kernel(CombineArgs A, CombineScale<T> S, const T *__restrict__ bc_val, const T *__restrict__ u,
                   const T *__restrict__ a, T *__restrict__ v, int nrhs, int64_t ld) {
  CPM_ROWS_COLS_LOOP(A.N, nrhs, i, r) v[i * ld + r] = combine_element<T>(A, S, bc_val, u, a, i, r, ld);
}

// ---- gather of small 2D batches -------------------------------------------------
// a_i = cs (E u - u)_i with one thread per row and column, flipped entries included (the
// rows near curves read their explicit stencils): one launch where tiles or cells of
// rows and the flipped entries take two.
template <int NP>
__global__ void __launch_bounds__(256) gather_rows2d_kernel(ApplyArgs<float> A, float cs, const float *__restrict__ u,
                                                            float *__restrict__ a, int nrhs, int64_t ld) {
  const int64_t NS = A.v.NS;
  CPM_ROWS_COLS_LOOP(NS, nrhs, i, r) {
    const uint32_t rb = __ldg(A.rbase + i);
    const float ui = __ldg(u + i * ld + r);
    float acc = 0.0f;
    if (rb & CPM_SPECIAL_BIT) {
      const int64_t s = __ldg(A.spec_of + i);
      for (int e = 0; e < 16; ++e) {  // (the 4 x 4 entries of a 2D stencil; absent ones are -1)
        const int32_t c = __ldg(A.ecol + s * 64 + e);
        if (c < 0) continue;
        const float val = __ldg(u + (int64_t)c * ld + r) * ((c < NS) ? cs : 1.0f);
        acc += __ldg(A.ew + s * 64 + e) * (val - cs * ui);
      }
    } else {
      const int32_t b = (int32_t)(rb >> 9);
      const int l = (int)(rb & 511u), lx = l & 7, ly = (l >> 3) & 7;
      const int split = (lx + NP - 1 < 8) ? NP : 8 - lx;
      float wx[4], wy[4];
      cpm_lagrange<NP, float>(__ldg(A.t + 3 * i), wx);
      cpm_lagrange<NP, float>(__ldg(A.t + 3 * i + 1), wy);
#pragma unroll
      for (int cy = 0; cy < NP; ++cy) {
        int32_t s0, s1;
        if (!cpm_line_start<NP>(A.v, b, lx, ly, 0, cy, 0, s0, s1)) continue;  // (set-up excludes it)
        float line = 0.0f;
#pragma unroll
        for (int cx = 0; cx < NP; ++cx) {
          const int32_t j = (cx < split) ? s0 + cx : s1 + (cx - split);
          line += wx[cx] * (__ldg(u + (int64_t)j * ld + r) - ui);
        }
        acc += wy[cy] * line;
      }
      acc *= cs;
    }
    a[i * ld + r] = acc;
  }
}

// one column with the iteration's dot products of v: (w, v), or (v, u) and (v, v)
// (STAGE); reading v back for them was a launch and a pass over two vectors
template <typename T, int STAGE>
__global__ void __launch_bounds__(256, (sizeof(T) == 8) ? 6 : 8)
    combine_dot_kernel(CombineArgs A, CombineScale<T> S, const T *__restrict__ bc_val, const T *__restrict__ u,
                       const T *__restrict__ a, T *__restrict__ v, Red R, Conv cv, const T *__restrict__ w) {
  constexpr int NQ = (STAGE == ST_OMEGA) ? 2 : 1;
  double acc[NQ] = {};
  T run[NQ] = {};
  int k = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < A.N; i += (int64_t)gridDim.x * blockDim.x) {
    const T o = (STAGE == ST_OMEGA) ? u[i] : w[i];
    const T x = combine_element<T>(A, S, bc_val, u, a, i, 0, 1);
    v[i] = x;
    run[0] += x * o;
    if (NQ > 1) run[NQ - 1] += x * x;
    if (sizeof(T) == 4 && (++k & 15) == 0)  // FP32 runs of 16, the runs in FP64
#pragma unroll
      for (int q = 0; q < NQ; ++q) { acc[q] += (double)run[q]; run[q] = T(0); }
  }
#pragma unroll
  for (int q = 0; q < NQ; ++q) acc[q] += (double)run[q];
  if (block_publish<NQ, 256>(acc, R)) finish_reduce<NQ, 256>(STAGE, R, cv);
}

// ---- batched combine: one warp per row, lanes over right-hand sides ---------
// With many right-hand sides the FD stencil is the same for every column, so
// one warp reads it once per row and each lane carries RPL adjacent columns per
// group of 32 RPL: every neighbour is one coalesced load ([N][ld] layout, ld a
// multiple of RPL).
template <typename T, int RPL>
struct Vec;
template <> struct Vec<float, 1> { typedef float t; };
template <> struct Vec<float, 2> { typedef float2 t; };
template <> struct Vec<double, 1> { typedef double t; };
template <> struct Vec<double, 2> { typedef double2 t; };

template <typename T, int RPL>
__device__ __forceinline__ void ldv(const T *p, T out[RPL]) {
  typedef typename Vec<T, RPL>::t V;
  V v = __ldg(reinterpret_cast<const V *>(p));
  const T *q = reinterpret_cast<const T *>(&v);
#pragma unroll
  for (int k = 0; k < RPL; ++k) out[k] = q[k];
}

template <typename T, int RPL>
__device__ __forceinline__ void stv(T *p, const T in[RPL]) {
  typedef typename Vec<T, RPL>::t V;
  V v;
  T *q = reinterpret_cast<T *>(&v);
#pragma unroll
  for (int k = 0; k < RPL; ++k) q[k] = in[k];
  *reinterpret_cast<V *>(p) = v;
}

// A block takes `chunk` consecutive rows, its 8 warps 8 of them at a time, so
// that the y neighbours (8 rows away inside a brick) are still in L1.
template <typename T, int RPL>
__global__ void __launch_bounds__(256, (sizeof(T) == 8) ? 3 : 4) combine_batched_kernel(CombineArgs A, CombineScale<T> S,
                                                              const T *__restrict__ bc_val, const T *__restrict__ u,
                                                              const T *__restrict__ a, T *__restrict__ v, int nrhs,
                                                              unsigned ld, int chunk) {
  // (a 32-bit stride: one widening multiply-add per neighbour's address)
  const int lane = threadIdx.x & 31;
  const int NS = (int)A.NS, N = (int)A.N;
  for (int64_t c0 = (int64_t)blockIdx.x * chunk; c0 < N; c0 += (int64_t)gridDim.x * chunk) {
    const int c1 = (int)((c0 + chunk < N) ? c0 + chunk : N);
    for (int i = (int)c0 + (int)(threadIdx.x >> 5); i < c1; i += 8) {
      int32_t nb[6];
      bool all = false;  // (the same in the whole warp)
      if (i < NS) {
        load_nbrs(A.nbr8, i, nb);
        all = min(min(min(nb[0], nb[1]), min(nb[2], nb[3])), min(nb[4], nb[5])) >= 0 &&
              max(max(max(nb[0], nb[1]), max(nb[2], nb[3])), max(nb[4], nb[5])) < NS;
      }
      for (int col = lane * RPL; col < nrhs; col += 32 * RPL) {
        T out[RPL];
        if (all) {
          T u0[RPL], uk[6][RPL], ak[6][RPL];
          ldv<T, RPL>(u + (uint64_t)(unsigned)i * ld + col, u0);
#pragma unroll
          for (int q = 0; q < 6; ++q) {
            const uint64_t o = (uint64_t)(unsigned)nb[q] * ld + col;
            ldv<T, RPL>(u + o, uk[q]);
            ldv<T, RPL>(a + o, ak[q]);
          }
#pragma unroll
          for (int k = 0; k < RPL; ++k) {
            T x[6], y[6];
#pragma unroll
            for (int q = 0; q < 6; ++q) { x[q] = uk[q][k]; y[q] = ak[q][k]; }
            out[k] = combine_row<true>(S, NS, A.nfd, nb, u0[k], x, y);
          }
        } else if (i < NS) {
          T u0[RPL], uk[6][RPL], ak[6][RPL];
          ldv<T, RPL>(u + (uint64_t)(unsigned)i * ld + col, u0);
#pragma unroll
          for (int q = 0; q < 6; ++q) {  // absent ones read the row's own: all 13 loads start at once
            const int c = (nb[q] >= 0) ? nb[q] : i, ca = (c < NS) ? c : i;
            ldv<T, RPL>(u + (uint64_t)(unsigned)c * ld + col, uk[q]);
            ldv<T, RPL>(a + (uint64_t)(unsigned)ca * ld + col, ak[q]);
          }
#pragma unroll
          for (int k = 0; k < RPL; ++k) {
            T x[6], y[6];
#pragma unroll
            for (int q = 0; q < 6; ++q) { x[q] = uk[q][k]; y[q] = ak[q][k]; }
            out[k] = combine_row<false>(S, NS, A.nfd, nb, u0[k], x, y);
          }
        } else {
          const int64_t al = i - NS;
          const int cnt = __ldg(A.bc_cnt + al);
#pragma unroll
          for (int k = 0; k < RPL; ++k) out[k] = T(0);
          for (int e = 0; e < cnt; ++e) {
            const int32_t cc = __ldg(A.bc_col + al * CPM_BC_STRIDE + e);
            const T w = __ldg(bc_val + al * CPM_BC_STRIDE + e) * ((cc < NS) ? S.cs : T(1));
            T val[RPL];
            ldv<T, RPL>(u + (uint64_t)(unsigned)cc * ld + col, val);
#pragma unroll
            for (int k = 0; k < RPL; ++k) out[k] += w * val[k];
          }
        }
        stv<T, RPL>(v + (uint64_t)(unsigned)i * ld + col, out);
      }
    }
  }
}

template <typename T>
void combine_args(const cpm_ctx *c, T m, T n, T rowscale, T cs, CombineArgs *A, CombineScale<T> *S, const T **bc_val) {
  *A = CombineArgs{c->NS, c->NS + c->NC, 2 * c->dim, c->d_nbr8, c->d_bc_cnt, c->d_bc_col};
  const double inv_h = 1.0 / c->h;
  *S = CombineScale<T>{(T)((double)rowscale * (double)m * (double)cs),
                       (T)((double)rowscale * (double)n * (inv_h * inv_h)), cs};
  if constexpr (sizeof(T) == 8) *bc_val = reinterpret_cast<const T *>(c->d_bc_val);
  else *bc_val = reinterpret_cast<const T *>(c->d_bc_val32);
}

template <typename T>
void launch_combine(const cpm_ctx *c, T m, T n, T rowscale, T cs, const T *u, const T *a, T *v, int nrhs, int64_t ld,
                    cudaStream_t st, FusedDot<T> *dot) {
  CombineArgs A;
  CombineScale<T> S;
  const T *bv;
  combine_args<T>(c, m, n, rowscale, cs, &A, &S, &bv);
  if (dot && nrhs == 1 && ld == 1) {
    // (the partials hold 4 blocks per SM)
    const unsigned g = (unsigned)std::min<int64_t>((A.N + 255) / 256, (int64_t)c->nsm * 4);
    if (dot->stage == ST_ALPHA)
      combine_dot_kernel<T, ST_ALPHA><<<g, 256, 0, st>>>(A, S, bv, u, a, v, dot->R, dot->cv, dot->w);
    else
      combine_dot_kernel<T, ST_OMEGA><<<g, 256, 0, st>>>(A, S, bv, u, a, v, dot->R, dot->cv, dot->w);
    dot->done = true;
    return;
  }
  combine_kernel<T><<<cpm_grid(A.N * nrhs, 256), 256, 0, st>>>(A, S, bv, u, a, v, nrhs, ld);
}

// batched product: E u for all PDE rows through the cell-bucketed gather
// (cells.cu), then the warp-per-row combine
template <typename T, int RPL>
int launch_batched(const cpm_ctx *c, T m, T n, T rowscale, T cs, const T *u, T *a, T *v, int nrhs, int64_t ld,
                   cudaStream_t st) {
  CombineArgs A;
  CombineScale<T> S;
  const T *bv;
  combine_args<T>(c, m, n, rowscale, cs, &A, &S, &bv);
  // 8 warps per block; by default 8 blocks per SM
  const int64_t warps = (int64_t)c->nsm * (c->tune.combine_warps_per_sm > 0 ? c->tune.combine_warps_per_sm : 64);
  // 64 rows a block; on bands that have fewer than four such blocks an SM, down to 8:
  // a warp's rows follow one another, and 64 left half of the SMs without any (16 columns
  // on the circle at h = 0.01, FP32 20.9 -> 14.4 us a product, FP64 30.8 -> 20.6)
  int chunk = 64;
  while (chunk > 8 && (A.N + chunk - 1) / chunk < 4 * (int64_t)c->nsm) chunk >>= 1;
  unsigned g = (unsigned)std::min<int64_t>((A.N + chunk - 1) / chunk, warps / 8);
  if (g < 1) g = 1;
  const int launched = 1 + cpm_launch_gather_cells<T>(c, cs, u, a, nrhs, ld, st, true, RPL);
  combine_batched_kernel<T, RPL><<<g, 256, 0, st>>>(A, S, bv, u, a, v, nrhs, (unsigned)ld, chunk);
  return launched;
}

__global__ void rhs_kernel(BandView v, const CurveDev *curves, const int32_t *bc_curve, const int32_t *side,
                           const int32_t *type, const double *param, const double *s, const double *g,
                           const double *samples, double *f, int nrhs, int64_t ld) {
  const int64_t N = v.NS + v.NC;
  CPM_ROWS_COLS_LOOP(N, nrhs, i, r) {
    if (i < v.NS) {
      f[i * ld + r] = s ? s[i * ld + r] : 0.0;
      continue;
    }
    int64_t al = i - v.NS;
    const CurveDev &cv = curves[bc_curve[al]];
    double gv = 0.0;
    if (g) {
      gv = g[al * ld + r];
    } else if (samples) {
      int ns = cv.n_samples;
      double sp = param[al] / 6.283185307179586476925286766559 * ns;
      double fl = floor(sp);
      int i0 = ((int)fl) % ns;
      if (i0 < 0) i0 += ns;
      int i1 = (i0 + 1) % ns;
      double fr = sp - fl;
      int64_t o = cv.sample_off;
      double plus = (1.0 - fr) * samples[(o + i0) * ld + r] + fr * samples[(o + i1) * ld + r];
      if (cv.two_sided) {
        double minus = (1.0 - fr) * samples[(o + ns + i0) * ld + r] + fr * samples[(o + ns + i1) * ld + r];
        int sd = side[al];
        gv = (sd > 0) ? minus : (sd < 0) ? plus : 0.5 * (plus + minus);
      } else {
        gv = plus;
      }
    }
    f[i * ld + r] = cpm_bc_data_scale(type[al]) * gv;
  }
}

// dL/dsamples = B^T (c_alpha lambda_alpha): one block per (sample, rhs), a fixed
// order reduction over the BC DOFs of the sample's curve (deterministic)
__global__ void boundary_grad_kernel(BandView v, const CurveDev *curves, int ncurves, const int32_t *curve_first,
                                     const int32_t *side, const int32_t *type, const double *param,
                                     const double *lam, double *out, int64_t nsamples_total, int nrhs,
                                     int64_t ld) {
  __shared__ double red[256];
  for (int64_t q = blockIdx.x; q < nsamples_total * nrhs; q += gridDim.x) {
    int64_t sidx = q / nrhs;
    int r = (int)(q - sidx * nrhs);
    int k = 0;
    while (k + 1 < ncurves && curves[k + 1].sample_off <= sidx) ++k;
    const CurveDev &cv = curves[k];
    int ns = cv.n_samples;
    int64_t loc = sidx - cv.sample_off;
    int blockside = (cv.two_sided && loc >= ns) ? -1 : +1;  // plus block first, then minus block
    int kk = (int)(loc % ns);
    double acc = 0.0;
    for (int64_t al = curve_first[k] + threadIdx.x; al < curve_first[k + 1]; al += blockDim.x) {
      double sp = param[al] / 6.283185307179586476925286766559 * ns;
      double fl = floor(sp);
      int i0 = ((int)fl) % ns;
      if (i0 < 0) i0 += ns;
      int i1 = (i0 + 1) % ns;
      double fr = sp - fl;
      double wblk = 1.0;
      if (cv.two_sided) {
        int sd = side[al];
        // a BC DOF whose cp_S is on the plus side takes the minus-side samples
        if (sd > 0) wblk = (blockside < 0) ? 1.0 : 0.0;
        else if (sd < 0) wblk = (blockside > 0) ? 1.0 : 0.0;
        else wblk = 0.5;
      }
      double w = 0.0;
      if (i0 == kk) w += 1.0 - fr;
      if (i1 == kk) w += fr;
      const double c = cpm_bc_data_scale(type[al]);
      acc += wblk * w * c * lam[(v.NS + al) * ld + r];
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
      if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
      __syncthreads();
    }
    if (threadIdx.x == 0) out[sidx * ld + r] = red[0];
    __syncthreads();
  }
}

}  // namespace

template <typename T>
ApplyArgs<T> cpm_apply_args(const cpm_ctx *c) {
  ApplyArgs<T> A;
  A.v = c->view();
  A.rbase = c->d_rbase;
  A.rself = c->d_rself;
  A.spec_of = c->d_spec_of;
  A.ecol = c->d_spec_ecol;
  A.fcol = c->d_spec_fcol;
  A.nbr8 = c->d_nbr8;
  A.bc_cnt = c->d_bc_cnt;
  A.bc_col = c->d_bc_col;
  if constexpr (sizeof(T) == 8) {
    A.t = reinterpret_cast<const T *>(c->d_t64);
    A.ew = reinterpret_cast<const T *>(c->d_spec_ew);
    A.bc_val = reinterpret_cast<const T *>(c->d_bc_val);
  } else {
    A.t = reinterpret_cast<const T *>(c->d_t32);
    A.ew = reinterpret_cast<const T *>(c->d_spec_ew32);
    A.bc_val = reinterpret_cast<const T *>(c->d_bc_val32);
  }
  return A;
}

template ApplyArgs<double> cpm_apply_args<double>(const cpm_ctx *);
template ApplyArgs<float> cpm_apply_args<float>(const cpm_ctx *);

// the kernels of one product v = R A C u with the intermediate a ([N_S][ld]);
// returns the number of launches
template <typename T>
static int launch_product(cpm_ctx *c, T m, T n, T rowscale, T cs, const T *u, T *a, T *v, int nrhs, int64_t ld,
                          cudaStream_t st, FusedDot<T> *dot) {
  // from 16 columns on a warp holds a cell for a group of columns; two adjacent
  // columns per lane need an even column count and 2-element alignment
  const bool aligned2 = (ld % 2 == 0) && ((reinterpret_cast<uintptr_t>(u) | reinterpret_cast<uintptr_t>(v) |
                                           reinterpret_cast<uintptr_t>(a)) % (2 * sizeof(T)) == 0);
  if constexpr (sizeof(T) == 4) {
    // Small 2D batches are bound by their launches: below a quarter (16 columns on: half)
    // of a million elements a thread per row and column takes two of them where tiles or
    // cells take three (circle, cubic, us a product, rows / tiles or cells: h = 0.01,
    // 2 columns 10.3 / 12.3, 15 columns 12.3 / 20.6, 33 15.3 / 26.7, 65 18.5 / 31.3; h = 0.001,
    // 5 columns 18.6 / 19.6, 8 columns, above the line, 23.6 / 18.5).  Widths that fill the
    // warps of the cell gather evenly stay there (16 columns 16.5 / 14.4).
    const bool even_batch = nrhs >= 16 && (nrhs <= 32 || (nrhs <= 64 && nrhs % 2 == 0 && aligned2));
    if (c->dim == 2 && nrhs > 1 && !even_batch && c->NS * nrhs <= (nrhs < 16 ? 262144 : 524288)) {
      const ApplyArgs<T> A = cpm_apply_args<T>(c);
      const unsigned g = cpm_grid(c->NS * nrhs, 256);
      if (c->p == 2) gather_rows2d_kernel<3><<<g, 256, 0, st>>>(A, cs, u, a, nrhs, ld);
      else gather_rows2d_kernel<4><<<g, 256, 0, st>>>(A, cs, u, a, nrhs, ld);
      launch_combine<T>(c, m, n, rowscale, cs, u, a, v, nrhs, ld, st, dot);
      return 2;
    }
  }
  if (nrhs > 32 && nrhs % 2 == 0 && aligned2)
    return launch_batched<T, 2>(c, m, n, rowscale, cs, u, a, v, nrhs, ld, st);
  if (nrhs >= 16) return launch_batched<T, 1>(c, m, n, rowscale, cs, u, a, v, nrhs, ld, st);
  int launched = 0;
  if (nrhs == 1 && c->ncells > 0 && c->tune.single_mode != 0) {
    ApplyArgs<T> A = cpm_apply_args<T>(c);
    if (c->tune.single_mode == 2) {
      launched = cpm_launch_fused1<T>(c, A, m, n, rowscale, cs, u, a, v, st);
      if (launched) return launched;
    } else {
      cpm_launch_gather1<T>(c, A, cs, u, a, st);
      launched = 1 + cpm_launch_correct_few<T>(c, cs, u, a, 1, ld, st);
    }
  }
  if (launched == 0) launched = cpm_launch_gather_tile<T>(c, cs, u, a, nrhs, ld, st, true);
  launch_combine<T>(c, m, n, rowscale, cs, u, a, v, nrhs, ld, st, dot);
  return launched + 1;
}

// v = R A C u using the context's reserved scratch for a (no allocation): R
// scales the PDE rows of the result by `rowscale` and C the PDE entries of the
// input by `colscale` (1 and 1 for the plain product); BC rows and BC entries
// are left alone.  Both forms use the difference form of the gather, which
// keeps the rounding of smooth fields relative to local differences.
template <typename T>
cpm_status cpm_apply_rc_T(cpm_ctx *c, double m, double n, double rowscale, double colscale, const T *u, T *v,
                          int nrhs, int64_t ld, cudaStream_t st, FusedDot<T> *dot) {
  if (sizeof(T) * (size_t)c->NS * (size_t)ld > c->a_scratch.bytes) return CPM_ERR_CAPACITY;
  T *a = reinterpret_cast<T *>(c->a_scratch.p);
  cpm_prof_begin(c, st);
  const int launched = launch_product<T>(c, (T)m, (T)n, (T)rowscale, (T)colscale, u, a, v, nrhs, ld, st, dot);
  cpm_prof_end(c, st, c->NS * (int64_t)nrhs);
  cpm_count_launches(c, launched);
  CPM_CUDA_TRY(cudaGetLastError());
  return CPM_OK;
}
template cpm_status cpm_apply_rc_T<double>(cpm_ctx *, double, double, double, double, const double *, double *, int,
                                           int64_t, cudaStream_t, FusedDot<double> *);
template cpm_status cpm_apply_rc_T<float>(cpm_ctx *, double, double, double, double, const float *, float *, int,
                                          int64_t, cudaStream_t, FusedDot<float> *);

template <typename T>
cpm_status cpm_apply_T(cpm_ctx *c, double m, double n, const T *u, T *v, int nrhs, int64_t ld, cudaStream_t st) {
  return cpm_apply_rc_T<T>(c, m, n, 1.0, 1.0, u, v, nrhs, ld, st);
}
template cpm_status cpm_apply_T<double>(cpm_ctx *, double, double, const double *, double *, int, int64_t,
                                        cudaStream_t);
template cpm_status cpm_apply_T<float>(cpm_ctx *, double, double, const float *, float *, int, int64_t,
                                       cudaStream_t);

void cpm_prof_begin(cpm_ctx *c, cudaStream_t st) {
  if (!c->prof.on) return;
  Profiler &p = c->prof;
  if (p.used + 2 > p.ev.size()) {
    for (int k = 0; k < 64; ++k) {
      cudaEvent_t e;
      if (cudaEventCreate(&e) != cudaSuccess) { (void)cudaGetLastError(); p.on = false; return; }
      p.ev.push_back(e);
    }
  }
  cudaEventRecord(p.ev[p.used], st);
}

void cpm_prof_end(cpm_ctx *c, cudaStream_t st, int64_t row_rhs) {
  if (!c->prof.on) return;
  Profiler &p = c->prof;
  cudaEventRecord(p.ev[p.used + 1], st);
  p.used += 2;
  p.applies += 1;
  p.row_rhs += row_rhs;
}

cpm_status cpm_internal_extend(cpm_ctx *c, const double *u, double *a, int nrhs, int64_t ld, cudaStream_t st) {
  cpm_count_launches(c, nrhs < 16 ? cpm_launch_gather_tile<double>(c, 1.0, u, a, nrhs, ld, st, false)
                                  : cpm_launch_gather_cells<double>(c, 1.0, u, a, nrhs, ld, st, false, 1));
  CPM_CUDA_TRY(cudaGetLastError());
  return CPM_OK;
}

cpm_status cpm_internal_rhs(cpm_ctx *c, const double *s, const double *g, const double *samples, double *f, int nrhs,
                            int64_t ld, cudaStream_t st) {
  int64_t N = c->NS + c->NC;
  rhs_kernel<<<cpm_grid(N * nrhs, 256), 256, 0, st>>>(c->view(), c->d_curves, c->d_bc_curve, c->d_side, c->d_bc_type,
                                                      c->d_param, s,
                                                      g, samples, f, nrhs, ld);
  CPM_CUDA_TRY(cudaGetLastError());
  return CPM_OK;
}

cpm_status cpm_internal_boundary_grad(cpm_ctx *c, const double *lam, double *out, int nrhs, int64_t ld,
                                      cudaStream_t st) {
  if (c->nsamples_total == 0) return CPM_OK;
  // c->d_curve_first: first BC DOF of each curve (BC DOFs are ordered by curve),
  // built with the boundary
  unsigned grid = (unsigned)std::min<int64_t>(c->nsamples_total * nrhs, (int64_t)c->nsm * 32);
  boundary_grad_kernel<<<grid, 256, 0, st>>>(c->view(), c->d_curves, c->ncurves, c->d_curve_first, c->d_side,
                                             c->d_bc_type, c->d_param, lam, out, c->nsamples_total, nrhs, ld);
  cpm_count_launches(c, 1);
  CPM_CUDA_TRY(cudaGetLastError());
  return CPM_OK;
}

// ---- operator product with a static scratch (no allocation) -----------------
// The E u intermediate lives in a fixed module array instead of the context's
// lazily grown scratch, so this path calls no allocator.  Nothing in the array
// has to start at zero: every element the combine reads was written earlier in
// the same call.  One array per device serves every context and stream, so
// calls that overlap in time on one device race on it.
namespace {
constexpr size_t kNoAllocScratchBytes = size_t(16) << 20;  // 16 MiB
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];
constexpr int kNoAllocMaxDevices = 64;
std::mutex g_noalloc_mu;
void *g_noalloc_ptr[kNoAllocMaxDevices] = {};

// device address of the array for the current device, looked up on the first
// call for that device
cpm_status noalloc_scratch(void **out) {
  int dev = -1;
  CPM_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kNoAllocMaxDevices) return CPM_ERR_CAPACITY;
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (!g_noalloc_ptr[dev]) {
    void *p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return cpm_internal_cuda_err(e);
    g_noalloc_ptr[dev] = p;
  }
  *out = g_noalloc_ptr[dev];
  return CPM_OK;
}
}  // namespace

size_t cpm_noalloc_scratch_bytes() { return kNoAllocScratchBytes; }

template <typename T>
cpm_status cpm_apply_noalloc_T(cpm_ctx *c, double m, double n, const T *u, T *v, int nrhs, int64_t ld,
                               cudaStream_t st) {
  if (sizeof(T) * (size_t)c->NS * (size_t)ld > kNoAllocScratchBytes) return CPM_ERR_CAPACITY;
  void *p = nullptr;
  cpm_status rc = noalloc_scratch(&p);
  if (rc) return rc;
  // the same kernels as cpm_apply
  const int launched = launch_product<T>(c, (T)m, (T)n, T(1), T(1), u, reinterpret_cast<T *>(p), v, nrhs, ld, st,
                                         nullptr);
  cpm_count_launches(c, launched);
  CPM_CUDA_TRY(cudaGetLastError());
  return CPM_OK;
}
template cpm_status cpm_apply_noalloc_T<double>(cpm_ctx *, double, double, const double *, double *, int, int64_t,
                                                cudaStream_t);
template cpm_status cpm_apply_noalloc_T<float>(cpm_ctx *, double, double, const float *, float *, int, int64_t,
                                               cudaStream_t);
