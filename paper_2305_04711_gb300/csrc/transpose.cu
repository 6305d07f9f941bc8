// transpose.cu -- v = R A^T u, the adjoint operator, as gathers (no atomics).
//
// With s = n / h^2 and d = m + n (-2 dim / h^2), a PDE row i of A reads
//   (A u)_i = d u_i + s sum_k a~_{c(i,k)},   a~_c = (E u)_c (c < N_S),  a~_alpha = u_alpha,
// where c(i,k) is the k-th FD neighbour of row i after the crossing-test flips
// (Eqs. 10-11) and (E u)_c = sum_e w_{c,e} u_{col(c,e)}; a BC row is
// (A u)_alpha = sum_e B_{alpha,e} u_{bcol(alpha,e)} (Sec. 4.3).  The transpose is
//   b_c   = s sum_{i : c(i,k) = c} lambda_i                      (PDE DOFs c)
//   y_j   = d lambda_j + sum_{c, e : col(c,e) = j} w_{c,e} b_c
//           + s sum_{i : c(i,k) = j >= N_S} lambda_i + sum_{alpha, e : bcol = j} B lambda_alpha.
// Kernel 1 forms b from the geometric FD neighbours of c, keeping those whose
// own neighbour slot pointing back at c was not flipped.  E^T b is gathered at
// each node from the (up to 4^dim) stencil cells whose node set contains it: for
// one right-hand side from a block of 64 sums per cell that another kernel forms
// first, for batches from every row of those cells (the cell buckets of cells.cu).
// To that comes the sparse remainder -- flipped FD entries, flipped E entries (moved from node j to
// its twin) and BC-row entries -- from a per-column list built at set-up.
#include <algorithm>

#include "apply.cuh"
#include "cpm_internal.cuh"
#include "fixed.cuh"
#include "util.cuh"

namespace {

// packed location (brick << 9 | local) of a node given relative to brick b
// (offsets within one brick step); -1 when that brick is not in the band
__device__ __forceinline__ int64_t loc_of(const BandView &v, int32_t b, int lx, int ly, int lz) {
  const int dx = lx >> 3, dy = ly >> 3, dz = lz >> 3;
  if (dx | dy | dz) {
    b = __ldg(v.bnbr + (int64_t)b * 27 + 13 + dx + 3 * dy + 9 * dz);
    if (b < 0) return -1;
  }
  return ((int64_t)b << 9) | (int64_t)((lz & 7) * 64 + (ly & 7) * 8 + (lx & 7));
}

// the 1-D Lagrange factors of the PDE rows along each axis, in cell order ([NS][12]: x,
// y, z, 4 slots each, zeros past the np1 stencil nodes)
__global__ void w1d_kernel(int64_t NS, int dim, int np1, const double *tc64, double *w64, float *w32) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < NS; i += (int64_t)gridDim.x * blockDim.x) {
    for (int a = 0; a < 3; ++a) {
      double w[4] = {1.0, 0.0, 0.0, 0.0};
      if (a < dim) cpm_lagrange_rt<double>(np1, tc64[3 * i + a], w);
      for (int k = 0; k < 4; ++k) {
        w64[i * 12 + 4 * a + k] = w[k];
        w32[i * 12 + 4 * a + k] = (float)w[k];
      }
    }
  }
}

__global__ void cellid_kernel(const uint32_t *cell_key, int64_t ncells, int32_t *cellid) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < ncells; k += (int64_t)gridDim.x * blockDim.x)
    cellid[cell_key[k]] = (int32_t)k;
}

// ---- the sparse remainder, one list per column -------------------------------
// entry kinds: 0 flipped FD entry (y_target += s lambda_src), 1 flipped E entry
// (y_target += val b_src), 2 BC-row entry (y_target += val lambda_src)
struct TEntrySrc {
  const int32_t *spec_row; const int32_t *fcol; int64_t nspec;
  const int32_t *corr_row; const int32_t *corr_start; const int32_t *corr_node; const int32_t *corr_col;
  const double *corr_w; int64_t ncorr;
  const int32_t *bc_cnt; const int32_t *bc_col; const double *bc_val;
  int64_t NS, NC;
};

// pass 0 counts entries per target; pass 1 writes them at cursor positions
__global__ void tlist_kernel(TEntrySrc S, int pass, int32_t *count, int32_t *cursor, int32_t *t_src, int32_t *t_kind,
                             double *t_val) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t tid0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  auto put = [&](int32_t target, int kind, int32_t src, double val) {
    if (pass == 0) {
      atomicAdd(count + target, 1);
    } else {
      int32_t p = atomicAdd(cursor + target, 1);
      t_src[p] = src;
      t_kind[p] = kind;
      t_val[p] = val;
    }
  };
  for (int64_t s = tid0; s < S.nspec; s += stride) {
    const int32_t i = S.spec_row[s];
    for (int k = 0; k < 6; ++k) {
      const int32_t cc = S.fcol[s * 6 + k];
      if (cc >= S.NS) put(cc, 0, i, 1.0);
    }
  }
  for (int64_t q = tid0; q < S.ncorr; q += stride) {
    const int32_t r = S.corr_row[q];
    for (int32_t e = S.corr_start[q]; e < S.corr_start[q + 1]; ++e) {
      put(S.corr_col[e], 1, r, S.corr_w[e]);
      put(S.corr_node[e], 1, r, -S.corr_w[e]);
    }
  }
  for (int64_t a = tid0; a < S.NC; a += stride) {
    const int64_t o = a * CPM_BC_STRIDE;
    for (int e = 0; e < S.bc_cnt[a]; ++e) put(S.bc_col[o + e], 2, (int32_t)(S.NS + a), S.bc_val[o + e]);
  }
}

// deterministic order inside each column list: by (kind, source)
__global__ void tlist_sort_kernel(const int32_t *ptr, int64_t N, int32_t *t_src, int32_t *t_kind, double *t_val,
                                  float *t_val32) {
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < N; j += (int64_t)gridDim.x * blockDim.x) {
    const int32_t o = ptr[j], e1 = ptr[j + 1];
    for (int32_t a = o + 1; a < e1; ++a) {
      const int32_t s = t_src[a], k = t_kind[a];
      const double v = t_val[a];
      const int64_t key = ((int64_t)k << 32) | (uint32_t)s;
      int32_t b = a - 1;
      while (b >= o && (((int64_t)t_kind[b] << 32) | (uint32_t)t_src[b]) > key) {
        t_src[b + 1] = t_src[b]; t_kind[b + 1] = t_kind[b]; t_val[b + 1] = t_val[b];
        --b;
      }
      t_src[b + 1] = s; t_kind[b + 1] = k; t_val[b + 1] = v;
    }
    for (int32_t a = o; a < e1; ++a) t_val32[a] = (float)t_val[a];
  }
}

// columns with remainder entries, and every BC column (which has nothing else)
__global__ void tcol_flag_kernel(const int32_t *ptr, int64_t NS, int64_t N, int32_t *flag) {
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < N; j += (int64_t)gridDim.x * blockDim.x)
    flag[j] = j >= NS || ptr[j + 1] > ptr[j];
}
__global__ void tcol_fill_kernel(const int32_t *flag, const int32_t *pos, int64_t N, int32_t *cols) {
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < N; j += (int64_t)gridDim.x * blockDim.x)
    if (flag[j]) cols[pos[j]] = (int32_t)j;
}

template <typename T>
struct TArgs {
  BandView v;
  const uint32_t *rself;
  const T *w1d;  // [NS][12] per-axis Lagrange factors, in cell order
  const int32_t *nbr8;
  const int32_t *cellid;
  const int32_t *cell_start;
  const int32_t *cell_rows;
  const int32_t *T_ptr;
  const int32_t *T_src;
  const int32_t *T_kind;
  const T *T_val;
};

// b_c = s * sum of lambda over the rows whose unflipped FD slot points at c
// (cs: right diagonal factor on the PDE entries of lambda, as in the forward
// product: the kernels then apply A^T C)
template <typename T>
__global__ void __launch_bounds__(256) tb_kernel(TArgs<T> A, T s, const T *__restrict__ lam, T *__restrict__ bv,
                                                 int nrhs, int64_t ld, int64_t ldb) {
  const int nfd = 2 * A.v.dim;
  CPM_ROWS_COLS_LOOP(A.v.NS, nrhs, c, r) {
    const uint32_t rs = __ldg(A.rself + c);
    const int32_t b = (int32_t)(rs >> 9);
    const int l = (int)(rs & 511u);
    const int lx = l & 7, ly = (l >> 3) & 7, lz = l >> 6;
    T acc = T(0);
    for (int d = 0; d < nfd; ++d) {
      const int ax = d >> 1, sg = (d & 1) ? 1 : -1;
      const int32_t i = cpm_node_index(A.v, b, lx + (ax == 0 ? sg : 0), ly + (ax == 1 ? sg : 0),
                                       lz + (ax == 2 ? sg : 0));
      if (i < 0) continue;
      // row i's slot in the opposite direction points back at c unless flipped
      if (__ldg(A.nbr8 + (int64_t)i * 8 + (d ^ 1)) == (int32_t)c) acc += __ldg(lam + (int64_t)i * ld + r);
    }
    bv[c * ldb + r] = s * acc;
  }
}

// ---- column by column -------------------------------------------------------
// Per stencil cell the block of its E^T b contributions,
//   blk[cz*16 + cy*4 + cx] = sum over the cell's rows of w_x[cx] w_y[cy] w_z[cz] b_row,
// one warp per cell, two nodes per lane.  In FP64 the block is summed in integers
// (fixed.cuh): b relative to the cell's largest |b|, w_z b and w_y w_z b rounded to
// 57 bits, the last factor in three multiply-adds; the block is stored as integers
// below 2^57 of the cell's own exponent, so that the node gather adds them as
// integers too (up to 64 of them).  One thread per cell with 64 FP64 sums in
// registers took 872 us on the sphere at h = 1/128, the FP64 node gather 326 us.
constexpr int TCW = 8;           // warps per block
constexpr int TCR = 8;           // rows whose weights are staged together
constexpr int E_NONE = -100000;  // exponent of a block of zeros
constexpr int E_PLAIN = 100000;  // block of doubles (values outside the integer range)

struct TCellArgs {
  const int32_t *cstart, *crows;
  int64_t ncells;
  const double *tc64;
  const float *w1d32;
};

template <int DIM, int NP>
__global__ void __launch_bounds__(TCW * 32)
    tcell_fx_kernel(TCellArgs A, const double *__restrict__ bv, long long *__restrict__ blk, int32_t *__restrict__ bexp) {
  constexpr int SLOTS = (DIM == 3) ? 64 : 16;
  __shared__ __align__(16) int2 s_w[TCW][TCR][3][4];
  __shared__ int2 s_b[TCW][TCR];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  // the lane's nodes: x = x0, x0 + 1 of line cy, cz
  const int x0 = (lane & 1) * 2, cy = (lane >> 1) & 3, cz = (DIM == 3) ? lane >> 3 : 0;
  const bool mine = 2 * lane < SLOTS;
  const int ax = lane >> 3, j0 = lane & 7;
  for (int64_t cid = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; cid < A.ncells; cid += nwarps) {
    const int32_t r0 = __ldg(A.cstart + cid), r1 = __ldg(A.cstart + cid + 1);
    unsigned top = 0;
    for (int32_t q = r0 + lane; q < r1; q += 32) top = max(top, fx_key(__ldg(bv + __ldg(A.crows + q))));
    top = __reduce_max_sync(0xffffffffu, top);
    const int em = (int)(top >> 20);
    // |b| < 2^61 and an axis multiplies by at most 6 / 16 (|w| <= 1), so a row adds less
    // than 2^58.2 (2D) or 2^56.8 (3D) to a sum: 16 or 64 rows of one sign stay below
    // 2^62.9 in 64 bits, and every doubling of the rows takes a bit from the operands
    constexpr int FULL = (DIM == 3) ? 6 : 4;
    const int K = 8 - max(0, 32 - __clz((r1 - r0 - 1) >> FULL));
    // (the exponent limits leave room for the scale factors of the node gather)
    const bool ok = top == 0u || (em >= 300 && em < 2040 && K >= 0);
    long long a0 = 0, a1 = 0;
    if (top != 0u && ok) {
      for (int32_t c0 = r0; c0 < r1; c0 += TCR) {
        const int k = min(TCR, r1 - c0);
        if (ax < 3) {
          int32_t wh[4] = {0, 0, 0, 0}, wl[4] = {0, 0, 0, 0};
          if (ax < DIM && j0 < k) fixed_weights<NP>(__ldg(A.tc64 + 3 * (int64_t)(c0 + j0) + ax), wh, wl);
#pragma unroll
          for (int q = 0; q < 4; ++q) s_w[w][j0][ax][q] = make_int2(wh[q], (q < NP) ? wl[q] : 0);
        } else if (j0 < k) {
          int2 o;
          halves(fx_of(__ldg(bv + __ldg(A.crows + c0 + j0)), em, K), o.x, o.y);
          s_b[w][j0] = o;
        }
        __syncwarp();
        for (int j = 0; j < k; ++j) {
          const int2 b = s_b[w][j], wy = s_w[w][j][1][cy];
          const int4 wx = *reinterpret_cast<const int4 *>(&s_w[w][j][0][x0]);
          int32_t qh = b.x, ql = b.y;
          if (DIM == 3) {
            const int2 wz = s_w[w][j][2][cz];
            halves(mad_wide(wz.x, qh, high_word(mad_wide(wz.x, ql, mad_wide(wz.y, qh, HALF)))), qh, ql);
          }
          halves(mad_wide(wy.x, qh, high_word(mad_wide(wy.x, ql, mad_wide(wy.y, qh, HALF)))), qh, ql);
          a0 = mad_wide(wx.x, qh, a0 + high_word(mad_wide(wx.x, ql, mad_wide(wx.y, qh, HALF))));
          a1 = mad_wide(wx.z, qh, a1 + high_word(mad_wide(wx.z, ql, mad_wide(wx.w, qh, HALF))));
        }
        __syncwarp();
      }
      // the block's largest sum moved to 57 bits
      const unsigned long long m0 = (unsigned long long)(a0 < 0 ? -a0 : a0), m1 = (unsigned long long)(a1 < 0 ? -a1 : a1);
      const int bits = (int)__reduce_max_sync(0xffffffffu, mine ? 64u - (unsigned)__clzll((long long)(m0 | m1)) : 0u);
      const int sh = 57 - bits;  // bits <= 63
      // (right shifts round: 64 sums truncated the same way would add up)
      const long long half = (sh < 0) ? 1ll << (-sh - 1) : 0;
      a0 = (sh >= 0) ? (long long)((unsigned long long)a0 << sh) : ((a0 + half) >> -sh);
      a1 = (sh >= 0) ? (long long)((unsigned long long)a1 << sh) : ((a1 + half) >> -sh);
      if (lane == 0) bexp[cid] = (bits == 0) ? E_NONE : em - 1075 - K - sh;
    } else {
      if (!ok) {  // plain FP64
        double p0 = 0.0, p1 = 0.0;
        for (int32_t q = r0; q < r1; ++q) {
          double wx[4] = {0, 0, 0, 0}, wy[4] = {0, 0, 0, 0}, wz[4] = {1, 0, 0, 0};
          const double *tq = A.tc64 + 3 * (int64_t)q, bb = __ldg(bv + __ldg(A.crows + q));
          cpm_lagrange<NP, double>(tq[0], wx);
          cpm_lagrange<NP, double>(tq[1], wy);
          if (DIM == 3) cpm_lagrange<NP, double>(tq[2], wz);
          double g = 0.0, h0 = 0.0, h1 = 0.0;
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            if (e == cy) g += wy[e];
            if (e == x0) h0 += wx[e];
            if (e == x0 + 1) h1 += wx[e];
          }
          double gz = 0.0;
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (e == cz) gz += wz[e];
          // nodes outside the stencil take nothing, also of infinities
          if (cy < NP && cz < NP && x0 < NP) p0 += ((h0 * g) * gz) * bb;
          if (cy < NP && cz < NP && x0 + 1 < NP) p1 += ((h1 * g) * gz) * bb;
        }
        a0 = __double_as_longlong(p0);
        a1 = __double_as_longlong(p1);
      }
      if (lane == 0) bexp[cid] = ok ? E_NONE : E_PLAIN;
    }
    if (mine) *reinterpret_cast<longlong2 *>(blk + cid * SLOTS + 2 * lane) = make_longlong2(a0, a1);
  }
}

template <int DIM, int NP>
__global__ void __launch_bounds__(TCW * 32)
    tcell_kernel(TCellArgs A, const float *__restrict__ bv, float *__restrict__ blk) {
  constexpr int SLOTS = (DIM == 3) ? 64 : 16;
  __shared__ __align__(16) float s_w[TCW][TCR][3][4];
  __shared__ float s_b[TCW][TCR];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int x0 = (lane & 1) * 2, cy = (lane >> 1) & 3, cz = (DIM == 3) ? lane >> 3 : 0;
  const int ax = lane >> 3, j0 = lane & 7;
  for (int64_t cid = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; cid < A.ncells; cid += nwarps) {
    const int32_t r0 = __ldg(A.cstart + cid), r1 = __ldg(A.cstart + cid + 1);
    float a0 = 0.0f, a1 = 0.0f;
    for (int32_t c0 = r0; c0 < r1; c0 += TCR) {
      const int k = min(TCR, r1 - c0);
      // (weights formed in FP64 and rounded once, as the batches take them: formed from
      // a fraction rounded to FP32, those near zero lose their relative accuracy)
      if (ax < 3) {
        float4 wt = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (j0 < k) wt = __ldg(reinterpret_cast<const float4 *>(A.w1d32 + (int64_t)(c0 + j0) * 12 + 4 * ax));
        *reinterpret_cast<float4 *>(s_w[w][j0][ax]) = wt;
      } else if (j0 < k) {
        s_b[w][j0] = __ldg(bv + __ldg(A.crows + c0 + j0));
      }
      __syncwarp();
      for (int j = 0; j < k; ++j) {
        float q = s_b[w][j];
        if (DIM == 3) q *= s_w[w][j][2][cz];
        q *= s_w[w][j][1][cy];
        const float2 wx = *reinterpret_cast<const float2 *>(&s_w[w][j][0][x0]);
        a0 += wx.x * q;
        a1 += wx.y * q;
      }
      __syncwarp();
    }
    if (2 * lane < SLOTS) *reinterpret_cast<float2 *>(blk + cid * SLOTS + 2 * lane) = make_float2(a0, a1);
  }
}

// the remainder of one right-hand side, eight lanes per column that has any: up to
// about a hundred entries near a curve, which one thread each walked as a chain of
// dependent loads long after the other columns were done
template <typename T>
__global__ void __launch_bounds__(256) t_rest_kernel(TArgs<T> A, const int32_t *__restrict__ cols, int64_t ncols, T s,
                                                     T rowscale, T cs, const T *__restrict__ lam,
                                                     const T *__restrict__ bv, T *__restrict__ y, int64_t ld) {
  const int sub = threadIdx.x & 7;
  const unsigned m = 0xFFu << (threadIdx.x & 24);
  const int64_t stride = ((int64_t)gridDim.x * blockDim.x) >> 3;
  for (int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 3; t < ncols; t += stride) {
    const int64_t j = __ldg(cols + t);
    const int32_t e1 = __ldg(A.T_ptr + j + 1);
    T acc = T(0);
    for (int32_t e = __ldg(A.T_ptr + j) + sub; e < e1; e += 8) {
      const int64_t src = __ldg(A.T_src + e);
      const int kind = __ldg(A.T_kind + e);
      const T w = (kind == 0) ? s * cs : __ldg(A.T_val + e);
      acc += w * (kind == 1 ? __ldg(bv + src) : __ldg(lam + src * ld));
    }
    acc += __shfl_xor_sync(m, acc, 1);
    acc += __shfl_xor_sync(m, acc, 2);
    acc += __shfl_xor_sync(m, acc, 4);
    if (sub == 0) y[j * ld] = (j < A.v.NS) ? y[j * ld] + rowscale * acc : acc;
  }
}

// The node gather for one right-hand side, one block per brick: the ids (and
// exponents) of the cells whose base node lies in the brick or up to NP - 1 nodes
// before it, 11 x 11 x 11, are staged once, so that a node finds its 64 cells at
// fixed distances in shared memory; on a band about 12 of them exist.
constexpr int TYT = 256;

template <typename T, int DIM, int NP>
__global__ void __launch_bounds__(TYT, 5)
    ty_brick_kernel(TArgs<T> A, const void *__restrict__ blk_, const int32_t *__restrict__ bexp, T dg, T rowscale,
                    T cs, const T *__restrict__ lam, T *__restrict__ y, int64_t ld) {
  constexpr int H = 7 + NP, HZ = (DIM == 3) ? H : 1;  // NP - 1 before, 8 of the brick
  constexpr int NZ = (DIM == 3) ? NP : 1;
  constexpr int SLOTS = (DIM == 3) ? 64 : 16;
  constexpr bool FX = (sizeof(T) == 8);
  __shared__ int32_t s_id[HZ * H * H];
  __shared__ int32_t s_e[FX ? HZ * H * H : 1];
  const int32_t b = (int32_t)blockIdx.x;
  for (int e = threadIdx.x; e < HZ * H * H; e += TYT) {
    const int hx = e % H - (NP - 1), hy = (e / H) % H - (NP - 1), hz = (DIM == 3) ? e / (H * H) - (NP - 1) : 0;
    const int64_t loc = loc_of(A.v, b, hx, hy, hz);
    const int32_t id = (loc < 0) ? -1 : __ldg(A.cellid + loc);
    s_id[e] = id;
    if (FX) s_e[e] = (id < 0) ? E_NONE : __ldg(bexp + id);
  }
  __syncthreads();
  const int32_t n1 = __ldg(A.v.bstart + b + 1);
  for (int32_t j = __ldg(A.v.bstart + b) + (int32_t)threadIdx.x; j < n1; j += TYT) {
    const int l = (int)(__ldg(A.rself + j) & 511u);
    const int at = (((DIM == 3) ? (l >> 6) + NP - 1 : 0) * H + ((l >> 3) & 7) + NP - 1) * H + (l & 7) + NP - 1;
    // which of the node's cells exist (bit cz 16 + cy 4 + cx), then four at a time, so
    // that their blocks are read together
    unsigned long long have = 0;
    int top = E_NONE;
    bool plain = false;
#pragma unroll
    for (int cz = 0; cz < NZ; ++cz)
#pragma unroll
      for (int cy = 0; cy < NP; ++cy)
#pragma unroll
        for (int cx = 0; cx < NP; ++cx) {
          const int o = at - (cz * H + cy) * H - cx;
          bool yes;
          if constexpr (FX) {
            const int e = s_e[o];
            yes = e != E_NONE;
            plain = plain || e == E_PLAIN;
            if (e != E_PLAIN) top = max(top, e);
          } else {
            yes = s_id[o] >= 0;
          }
          if (yes) have |= 1ull << (cz * 16 + cy * 4 + cx);
        }
    // (FP32 starts from the diagonal, which the blocks mostly cancel: partial sums, and
    // with them the rounding, shrink on the way)
    T sum = FX ? T(0) : (dg * cs) * __ldg(lam + (int64_t)j * ld);
    long long acc = 0;
    while (have) {
      int slot[4], e[4];
      int64_t src[4];
      bool on[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        on[k] = have != 0;
        slot[k] = on[k] ? __ffsll((long long)have) - 1 : slot[0];
        have &= have - 1;
        const int o = at - ((slot[k] >> 4) * H + ((slot[k] >> 2) & 3)) * H - (slot[k] & 3);
        src[k] = (int64_t)s_id[o] * SLOTS + slot[k];
        e[k] = FX ? s_e[o] : 0;
      }
      if constexpr (FX) {
        const long long *blk = reinterpret_cast<const long long *>(blk_);
        long long z[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) z[k] = __ldg(blk + src[k]);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if (on[k] && e[k] != E_PLAIN) {
            const int sh = min(top - e[k], 62);
            acc += (z[k] + ((1ll << sh) >> 1)) >> sh;
          } else if (on[k]) {
            sum += __longlong_as_double(z[k]);
          }
        }
      } else {
        const T *blk = reinterpret_cast<const T *>(blk_);
        T z[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) z[k] = __ldg(blk + src[k]);
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (on[k]) sum += z[k];
      }
    }
    if constexpr (FX) {
      constexpr double back = (DIM == 3) ? 4096.0 / 216.0 : 256.0 / 36.0;  // every axis multiplied by 6 / 16
      if (top != E_NONE) sum = scaled_sum(fx_scale(back, top), acc, plain ? sum : 0.0);
      sum += (dg * cs) * __ldg(lam + j * ld);
    }
    y[j * ld] = rowscale * sum;
  }
}

// ---- batches ---------------------------------------------------------------------
// y = R (d lambda_S + E^T b + remainder).  FP32 takes the stencil's extent at compile
// time and reads the cell ids of a node's x line together, which depend on nothing else:
// 3 columns on the circle at h = 0.001 40.5 -> 33.3 us, on the sphere at h = 1/20 125 -> 115.
// FP64 (NP 0: extent at run time) is held by its pipe, and gets 2 to 5 %
// slower by it.
template <typename T, int DIM, int NP>
__global__ void __launch_bounds__(256) ty_kernel(TArgs<T> A, T dg, T s, T rowscale, T cs, const T *__restrict__ lam,
                                                 const T *__restrict__ bv, T *__restrict__ y, int nrhs, int64_t ld) {
  const int64_t NS = A.v.NS, N = NS + A.v.NC;
  CPM_ROWS_COLS_LOOP(N, nrhs, j, r) {
    T acc = T(0);
    if (j < NS) {
      acc = (dg * cs) * __ldg(lam + j * ld + r);
      const uint32_t rs = __ldg(A.rself + j);
      const int32_t b = (int32_t)(rs >> 9);
      const int l = (int)(rs & 511u);
      const int lx = l & 7, ly = (l >> 3) & 7, lz = l >> 6;
      const auto add_cell = [&](int32_t cell, int cx, int cy, int cz) {
        const int32_t q1 = __ldg(A.cell_start + cell + 1);
        for (int32_t q = __ldg(A.cell_start + cell); q < q1; ++q) {
          const int64_t row = __ldg(A.cell_rows + q);
          const T *wr = A.w1d + (int64_t)q * 12;
          const T w = __ldg(wr + cx) * __ldg(wr + 4 + cy) * __ldg(wr + 8 + cz);
          acc += w * __ldg(bv + row * ld + r);
        }
      };
      if constexpr (NP > 0) {
#pragma unroll 1
        for (int cz = 0; cz < ((DIM == 3) ? NP : 1); ++cz)
#pragma unroll 1
          for (int cy = 0; cy < NP; ++cy) {
            int32_t cell[NP];
#pragma unroll
            for (int cx = 0; cx < NP; ++cx) {
              const int64_t key = loc_of(A.v, b, lx - cx, ly - cy, lz - cz);
              cell[cx] = (key < 0) ? -1 : __ldg(A.cellid + key);
            }
#pragma unroll
            for (int cx = 0; cx < NP; ++cx)
              if (cell[cx] >= 0) add_cell(cell[cx], cx, cy, cz);
          }
      } else {
        const int np1 = A.v.np1, nz = (A.v.dim == 3) ? np1 : 1;
        for (int cz = 0; cz < nz; ++cz)
          for (int cy = 0; cy < np1; ++cy)
            for (int cx = 0; cx < np1; ++cx) {
              const int64_t key = loc_of(A.v, b, lx - cx, ly - cy, lz - cz);
              if (key < 0) continue;
              const int32_t cell = __ldg(A.cellid + key);
              if (cell >= 0) add_cell(cell, cx, cy, cz);
            }
      }
    }
    const int32_t e1 = __ldg(A.T_ptr + j + 1);
    for (int32_t e = __ldg(A.T_ptr + j); e < e1; ++e) {
      const int64_t src = __ldg(A.T_src + e);
      const int kind = __ldg(A.T_kind + e);
      if (kind == 0) acc += (s * cs) * __ldg(lam + src * ld + r);
      else if (kind == 1) acc += __ldg(A.T_val + e) * __ldg(bv + src * ld + r);
      else acc += __ldg(A.T_val + e) * __ldg(lam + src * ld + r);
    }
    y[j * ld + r] = (j < NS) ? rowscale * acc : acc;
  }
}

}  // namespace

cpm_status cpm_build_transpose(cpm_ctx *c) {
  cudaStream_t st = c->stream;
  cudaFree(c->d_T_ptr); cudaFree(c->d_T_row); cudaFree(c->d_T_kind); cudaFree(c->d_T_val); cudaFree(c->d_T_val32);
  cudaFree(c->d_cellid); cudaFree(c->d_w1d64); cudaFree(c->d_w1d32); cudaFree(c->d_tblk); cudaFree(c->d_T_cols);
  c->d_T_cols = nullptr; c->nTcols = 0;
  c->d_w1d64 = nullptr; c->d_w1d32 = nullptr; c->d_tblk = nullptr;
  c->d_T_ptr = nullptr; c->d_T_row = nullptr; c->d_T_kind = nullptr; c->d_T_val = nullptr; c->d_T_val32 = nullptr;
  c->d_cellid = nullptr;
  c->transpose_ready = false;
  const int64_t N = c->NS + c->NC;
  const int64_t nkeys = c->nb * 512;
  int32_t *count = nullptr, *cursor = nullptr, *d_tot = nullptr;
  int32_t h_tot = 0;
  cpm_status rc = CPM_OK;
  TEntrySrc S{c->d_spec_row, c->d_spec_fcol, c->nspec, c->d_corr_row, c->d_corr_start, c->d_corr_node, c->d_corr_col,
              c->d_corr_w64, c->ncorr, c->d_bc_cnt, c->d_bc_col, c->d_bc_val, c->NS, c->NC};
  const unsigned gl = cpm_grid(std::max<int64_t>(std::max<int64_t>(c->nspec, c->ncorr), c->NC), 128);
#define TRY(x)                                             \
  do {                                                     \
    cudaError_t e_ = (x);                                  \
    if (e_) { rc = cpm_internal_cuda_err(e_); goto done; } \
  } while (0)
  TRY(cudaMalloc(&c->d_cellid, sizeof(int32_t) * std::max<int64_t>(nkeys, 1)));
  // blocks of the one right-hand side form, then the blocks' exponents
  TRY(cudaMalloc(&c->d_tblk, (sizeof(double) * 64 + sizeof(int32_t)) * std::max<int64_t>(c->ncells, 1)));
  TRY(cudaMemsetAsync(c->d_cellid, 0xFF, sizeof(int32_t) * std::max<int64_t>(nkeys, 1), st));
  TRY(cudaMalloc(&c->d_w1d64, sizeof(double) * 12 * std::max<int64_t>(c->NS, 1)));
  TRY(cudaMalloc(&c->d_w1d32, sizeof(float) * 12 * std::max<int64_t>(c->NS, 1)));
  w1d_kernel<<<cpm_grid(c->NS, 256), 256, 0, st>>>(c->NS, c->dim, c->p + 1, c->d_tc64, c->d_w1d64, c->d_w1d32);
  if (c->ncells > 0)
    cellid_kernel<<<cpm_grid(c->ncells, 256), 256, 0, st>>>(c->d_cell_key, c->ncells, c->d_cellid);
  TRY(cudaMalloc(&count, sizeof(int32_t) * (N + 1)));
  TRY(cudaMalloc(&cursor, sizeof(int32_t) * (N + 1)));
  TRY(cudaMalloc(&d_tot, sizeof(int32_t)));
  TRY(cudaMalloc(&c->d_T_ptr, sizeof(int32_t) * (N + 1)));
  TRY(cudaMemsetAsync(count, 0, sizeof(int32_t) * (N + 1), st));
  tlist_kernel<<<gl, 128, 0, st>>>(S, 0, count, nullptr, nullptr, nullptr, nullptr);
  TRY(cpm_exclusive_scan(count, c->d_T_ptr, N + 1, d_tot, st));
  TRY(cudaMemcpyAsync(&h_tot, d_tot, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
  TRY(cudaStreamSynchronize(st));
  c->nT = h_tot;
  TRY(cudaMalloc(&c->d_T_row, sizeof(int32_t) * std::max<int64_t>(c->nT, 1)));
  TRY(cudaMalloc(&c->d_T_kind, sizeof(int32_t) * std::max<int64_t>(c->nT, 1)));
  TRY(cudaMalloc(&c->d_T_val, sizeof(double) * std::max<int64_t>(c->nT, 1)));
  TRY(cudaMalloc(&c->d_T_val32, sizeof(float) * std::max<int64_t>(c->nT, 1)));
  TRY(cudaMemcpyAsync(cursor, c->d_T_ptr, sizeof(int32_t) * (N + 1), cudaMemcpyDeviceToDevice, st));
  if (c->nT > 0) {
    tlist_kernel<<<gl, 128, 0, st>>>(S, 1, nullptr, cursor, c->d_T_row, c->d_T_kind, c->d_T_val);
    tlist_sort_kernel<<<cpm_grid(N, 128), 128, 0, st>>>(c->d_T_ptr, N, c->d_T_row, c->d_T_kind, c->d_T_val,
                                                       c->d_T_val32);
  }
  // columns with entries (count and cursor are free again)
  tcol_flag_kernel<<<cpm_grid(N, 256), 256, 0, st>>>(c->d_T_ptr, c->NS, N, count);
  TRY(cpm_exclusive_scan(count, cursor, N, d_tot, st));
  TRY(cudaMemcpyAsync(&h_tot, d_tot, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
  TRY(cudaStreamSynchronize(st));
  c->nTcols = h_tot;
  TRY(cudaMalloc(&c->d_T_cols, sizeof(int32_t) * std::max<int64_t>(c->nTcols, 1)));
  tcol_fill_kernel<<<cpm_grid(N, 256), 256, 0, st>>>(count, cursor, N, c->d_T_cols);
  TRY(cudaGetLastError());
  TRY(cudaStreamSynchronize(st));
  c->transpose_ready = true;
done:
#undef TRY
  cudaFree(count); cudaFree(cursor); cudaFree(d_tot);
  return rc;
}

template <typename T>
cpm_status cpm_apply_transpose_rc_T(cpm_ctx *c, double m, double n, double rowscale, double colscale, const T *u,
                                    T *v, int nrhs, int64_t ld, cudaStream_t st, FusedDot<T> * /*dot*/) {
  if (!c->transpose_ready) return CPM_ERR_STATE;
  if (sizeof(T) * (size_t)c->NS * (size_t)ld > c->b_scratch.bytes) return CPM_ERR_CAPACITY;
  TArgs<T> A;
  A.v = c->view();
  A.rself = c->d_rself;
  A.nbr8 = c->d_nbr8;
  A.cellid = c->d_cellid;
  A.cell_start = c->d_cell_start;
  A.cell_rows = c->d_cell_rows;
  A.T_ptr = c->d_T_ptr;
  A.T_src = c->d_T_row;
  A.T_kind = c->d_T_kind;
  if constexpr (sizeof(T) == 8) {
    A.w1d = reinterpret_cast<const T *>(c->d_w1d64);
    A.T_val = reinterpret_cast<const T *>(c->d_T_val);
  } else {
    A.w1d = reinterpret_cast<const T *>(c->d_w1d32);
    A.T_val = reinterpret_cast<const T *>(c->d_T_val32);
  }
  T *bv = reinterpret_cast<T *>(c->b_scratch.p);
  const double inv_h2 = 1.0 / (c->h * c->h);
  const T s = T(n * inv_h2), dg = T(m + n * (-2.0 * c->dim * inv_h2));
  const int64_t N = c->NS + c->NC;
  cpm_prof_begin(c, st);
  int launched = 0;
  // One column, or a few of a 3D band, one by one: per-cell blocks of E^T b (one
  // column's are reserved at set-up), then the nodes by bricks.  All columns at once
  // revisit every row of a node's 64 (27) cells but share the walk, and a small band pays
  // four launches a column, so the rows must make up for them.  Measured, one by one / at
  // once in us:
  //   FP64 cubic      27k rows: 6 columns 308 / 399, 8 columns 411 / 353; 42k: 8 431 / 477
  //   FP64 quadratic  21k rows: 2 columns 78 / 103, 4 156 / 119; 42k: 4 156 / 167, 5 200 / 190;
  //                   84k: 7 341 / 399, 8 394 / 365; 167k: 8 513 / 657
  //   FP32 cubic      60k rows: 3 columns 118 / 142, 4 160 / 154; 106k: 4 186 / 209
  //   FP32 quadratic  84k rows: 2 columns 66 / 68, 3 99 / 78; 167k: 2 86 / 104, 4 173 / 143;
  //                   339k: 4 247 / 256
  // (8 columns walk aligned 64-byte segments, hence their own line).  More columns than
  // these gain only on bands of a million rows and lose below: FP64 16 columns 5.6 / 10.1 ms
  // at 1.04M rows, 64 columns 11.5 / 10.6 ms at 424k.
  int64_t rows_a_column;  // fewer rows than this for each column: all at once
  if (sizeof(T) == 8) rows_a_column = (c->p == 2) ? (nrhs < 8 ? 8500 : 13500) : (nrhs < 8 ? 3800 : 4500);
  else rows_a_column = (c->p == 2) ? 60000 : 25000;
  const bool few = c->dim == 3 && nrhs <= (sizeof(T) == 8 ? 8 : 4) && c->NS >= nrhs * rows_a_column;
  const bool by_column = c->d_tblk && c->ncells > 0 && (nrhs == 1 || few);
  if (by_column) {
    TCellArgs C{c->d_cell_start, c->d_cell_rows, c->ncells, c->d_tc64, c->d_w1d32};
    int32_t *bexp = reinterpret_cast<int32_t *>(c->d_tblk + 64 * c->ncells);
    const unsigned gc = (unsigned)std::min<int64_t>((c->ncells + TCW - 1) / TCW, (int64_t)c->nsm * 64);
    for (int r = 0; r < nrhs; ++r) {
      const T *ur = u + r;
      T *vr = v + r;
      tb_kernel<T><<<cpm_grid(c->NS, 256), 256, 0, st>>>(A, T(s * T(colscale)), ur, bv, 1, ld, 1);
#define CPM_TCELL(D, NP)                                                                                             \
  do {                                                                                                               \
    if constexpr (sizeof(T) == 8)                                                                                    \
      tcell_fx_kernel<D, NP><<<gc, TCW * 32, 0, st>>>(C, bv, reinterpret_cast<long long *>(c->d_tblk), bexp);        \
    else                                                                                                             \
      tcell_kernel<D, NP><<<gc, TCW * 32, 0, st>>>(C, bv, reinterpret_cast<float *>(c->d_tblk));                     \
    ty_brick_kernel<T, D, NP><<<(unsigned)c->nb, TYT, 0, st>>>(A, c->d_tblk, bexp, dg, T(rowscale), T(colscale), ur, \
                                                               vr, ld);                                              \
  } while (0)
      if (c->dim == 3) {
        if (c->p == 2) CPM_TCELL(3, 3); else CPM_TCELL(3, 4);
      } else {
        if (c->p == 2) CPM_TCELL(2, 3); else CPM_TCELL(2, 4);
      }
#undef CPM_TCELL
      launched += 3;
      if (c->nTcols > 0) {
        t_rest_kernel<T><<<cpm_grid(8 * c->nTcols, 256), 256, 0, st>>>(A, c->d_T_cols, c->nTcols, s, T(rowscale),
                                                                       T(colscale), ur, bv, vr, ld);
        ++launched;
      }
    }
  } else {
    tb_kernel<T><<<cpm_grid(c->NS * nrhs, 256), 256, 0, st>>>(A, T(s * T(colscale)), u, bv, nrhs, ld, ld);
#define CPM_TY(D, NP) \
  ty_kernel<T, D, NP><<<cpm_grid(N * nrhs, 256), 256, 0, st>>>(A, dg, s, T(rowscale), T(colscale), u, bv, v, nrhs, ld)
    if constexpr (sizeof(T) == 8) {
      CPM_TY(0, 0);
    } else if (c->dim == 3) {
      if (c->p == 2) CPM_TY(3, 3); else CPM_TY(3, 4);
    } else {
      if (c->p == 2) CPM_TY(2, 3); else CPM_TY(2, 4);
    }
#undef CPM_TY
    launched = 2;
  }
  cpm_prof_end(c, st, c->NS * (int64_t)nrhs);
  cpm_count_launches(c, launched);
  CPM_CUDA_TRY(cudaGetLastError());
  return CPM_OK;
}
template cpm_status cpm_apply_transpose_rc_T<double>(cpm_ctx *, double, double, double, double, const double *,
                                                     double *, int, int64_t, cudaStream_t, FusedDot<double> *);
template cpm_status cpm_apply_transpose_rc_T<float>(cpm_ctx *, double, double, double, double, const float *,
                                                    float *, int, int64_t, cudaStream_t, FusedDot<float> *);

template <typename T>
cpm_status cpm_apply_transpose_T(cpm_ctx *c, double m, double n, const T *u, T *v, int nrhs, int64_t ld,
                                 cudaStream_t st) {
  return cpm_apply_transpose_rc_T<T>(c, m, n, 1.0, 1.0, u, v, nrhs, ld, st);
}
template cpm_status cpm_apply_transpose_T<double>(cpm_ctx *, double, double, const double *, double *, int, int64_t,
                                                  cudaStream_t);
template cpm_status cpm_apply_transpose_T<float>(cpm_ctx *, double, double, const float *, float *, int, int64_t,
                                                 cudaStream_t);
