// cells.cu -- PDE rows bucketed by the base node ("cell") of their
// interpolation stencil, and the batched products built on the buckets.
//
// All rows whose closest points fall in the same grid cell share the same
// 4x4x4 stencil nodes (Eq. 1); only their weights differ.  On a narrow band
// several rows (about 2 r / h divided by the number of cells the surface
// crosses per normal line, ~5 in 3D) share each cell.  With many right-hand
// sides the extension E u is bound by moving node values, so one warp takes a
// whole cell: it holds the cell's node values for its columns in registers and
// applies the separable weights of every row of the cell to them.
//
// Rows near an interior boundary use the same cell gather; the entries their
// crossing test flipped (node j replaced by its BC twin, Sec. 4) are applied
// afterwards as a sparse correction w (u_twin - u_j) from a list built here.
//
// The buckets are built by a counting sort over the dense (brick, local) key
// space, with each bucket then ordered by row index, so the layout does not
// depend on the scheduling of the atomics.
#include <algorithm>

#include "apply.cuh"
#include "cpm_internal.cuh"
#include "fixed.cuh"
#include "util.cuh"

namespace {

__global__ void cell_count_kernel(const uint32_t *rbase, int64_t NS, int32_t *count) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < NS; i += (int64_t)gridDim.x * blockDim.x)
    atomicAdd(count + (rbase[i] & ~CPM_SPECIAL_BIT), 1);
}

__global__ void cell_scatter_kernel(const uint32_t *rbase, int64_t NS, int32_t *cursor, int32_t *rows) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < NS; i += (int64_t)gridDim.x * blockDim.x) {
    int32_t p = atomicAdd(cursor + (rbase[i] & ~CPM_SPECIAL_BIT), 1);
    rows[p] = (int32_t)i;
  }
}

// per non-empty key: its cell id, start, and a deterministic (row-index) order
__global__ void cell_finish_kernel(const int32_t *count, const int32_t *offs, const int32_t *cellpos, int64_t nkeys,
                                   int32_t *rows, int32_t *cell_start, uint32_t *cell_key) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nkeys; k += (int64_t)gridDim.x * blockDim.x) {
    int32_t n = count[k];
    if (n == 0) continue;
    int32_t c = cellpos[k], o = offs[k];
    cell_start[c] = o;
    cell_key[c] = (uint32_t)k;
    // insertion sort of the bucket (a few to a few dozen rows)
    for (int32_t a = o + 1; a < o + n; ++a) {
      int32_t v = rows[a], b = a - 1;
      while (b >= o && rows[b] > v) { rows[b + 1] = rows[b]; --b; }
      rows[b + 1] = v;
    }
  }
}

__global__ void flag_nonzero_kernel(const int32_t *count, int64_t n, int32_t *flag) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
    flag[k] = count[k] != 0;
}

__global__ void set_i32_kernel(int32_t *p, int32_t v) { *p = v; }

// FD neighbour columns of every PDE row (x-, x+, y-, y+, z-, z+; -1 where
// absent; the flipped columns for rows near interior boundaries), padded to 8
__global__ void nbr8_kernel(BandView v, const uint32_t *rself, const uint32_t *rbase, const int32_t *spec_of,
                            const int32_t *fcol, int32_t *nbr8) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < v.NS; i += (int64_t)gridDim.x * blockDim.x) {
    int32_t o[8];
    if (rbase[i] & CPM_SPECIAL_BIT) {
      const int64_t sp = spec_of[i];
      for (int k = 0; k < 6; ++k) o[k] = fcol[sp * 6 + k];
    } else {
      const uint32_t rs = rself[i];
      const int32_t b = (int32_t)(rs >> 9);
      const int l = (int)(rs & 511u);
      const int lx = l & 7, ly = (l >> 3) & 7, lz = l >> 6;
      o[0] = cpm_node_index(v, b, lx - 1, ly, lz);
      o[1] = cpm_node_index(v, b, lx + 1, ly, lz);
      o[2] = cpm_node_index(v, b, lx, ly - 1, lz);
      o[3] = cpm_node_index(v, b, lx, ly + 1, lz);
      o[4] = (v.dim == 3) ? cpm_node_index(v, b, lx, ly, lz - 1) : -1;
      o[5] = (v.dim == 3) ? cpm_node_index(v, b, lx, ly, lz + 1) : -1;
    }
    o[6] = o[7] = -1;
    int4 *dst = reinterpret_cast<int4 *>(nbr8 + i * 8);
    dst[0] = make_int4(o[0], o[1], o[2], o[3]);
    dst[1] = make_int4(o[4], o[5], o[6], o[7]);
  }
}

// node of stencil entry e (x fastest) of the row with packed base rb
__device__ __forceinline__ int32_t entry_node(const BandView &v, uint32_t rb, int e) {
  const int32_t b = (int32_t)((rb & ~CPM_SPECIAL_BIT) >> 9);
  const int l = (int)(rb & 511u);
  return cpm_node_index(v, b, (l & 7) + (e & 3), ((l >> 3) & 7) + ((e >> 2) & 3), (l >> 6) + (e >> 4));
}

// number of flipped interpolation entries of each special row
__global__ void corr_count_kernel(BandView v, const int32_t *spec_row, int64_t nspec, const uint32_t *rbase,
                                  const int32_t *ecol, int32_t *cnt) {
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < nspec; s += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t rb = rbase[spec_row[s]];
    int n = 0;
    for (int e = 0; e < 64; ++e)
      if (cpm_in_stencil(e, v.np1, v.dim)) n += (ecol[s * 64 + e] != entry_node(v, rb, e));
    cnt[s] = n;
  }
}

__global__ void corr_fill_kernel(BandView v, const int32_t *spec_row, int64_t nspec, const uint32_t *rbase,
                                 const int32_t *ecol, const double *ew, const int32_t *cnt, const int32_t *offs,
                                 const int32_t *rowpos, int32_t *corr_row, int32_t *corr_start, int32_t *node,
                                 int32_t *col, double *w64, float *w32) {
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < nspec; s += (int64_t)gridDim.x * blockDim.x) {
    if (cnt[s] == 0) continue;
    const int32_t i = spec_row[s];
    const uint32_t rb = rbase[i];
    corr_row[rowpos[s]] = i;
    corr_start[rowpos[s]] = offs[s];
    int32_t o = offs[s];
    for (int e = 0; e < 64; ++e) {
      if (!cpm_in_stencil(e, v.np1, v.dim)) continue;
      const int32_t j = entry_node(v, rb, e), ce = ecol[s * 64 + e];
      if (ce == j) continue;
      node[o] = j;
      col[o] = ce;
      w64[o] = ew[s * 64 + e];
      w32[o] = (float)ew[s * 64 + e];
      ++o;
    }
  }
}

constexpr int CHUNK = 8;   // rows of a cell whose weights are staged together
constexpr int WARPS = 8;   // warps per block

struct CellArgs {
  const int32_t *cstart, *crows;
  const uint32_t *ckey;
  const int2 *lines;
  int64_t ncells;
};

template <typename T, int R>
struct VecT;
template <> struct VecT<float, 1> { typedef float t; };
template <> struct VecT<float, 2> { typedef float2 t; };
template <> struct VecT<double, 1> { typedef double t; };
template <> struct VecT<double, 2> { typedef double2 t; };

template <typename T, int R>
__device__ __forceinline__ void vld(const T *p, T out[R]) {
  typedef typename VecT<T, R>::t V;
  const V x = __ldg(reinterpret_cast<const V *>(p));
  const T *q = reinterpret_cast<const T *>(&x);
#pragma unroll
  for (int k = 0; k < R; ++k) out[k] = q[k];
}

template <typename T, int R>
__device__ __forceinline__ void vst(T *p, const T in[R]) {
  typedef typename VecT<T, R>::t V;
  V x;
  T *q = reinterpret_cast<T *>(&x);
#pragma unroll
  for (int k = 0; k < R; ++k) q[k] = in[k];
  *reinterpret_cast<V *>(p) = x;
}

// acc[r] += w d[r] and d[r] -= c[r] over a lane's R columns; two FP32 columns
// go through one packed instruction (FFMA2 / FADD2 of sm_100+), with the same
// rounding as the scalar FMA and add
__device__ __forceinline__ void axpy_w(float (&acc)[1], float w, const float (&d)[1]) { acc[0] += w * d[0]; }
__device__ __forceinline__ void axpy_w(float (&acc)[2], float2 w, const float (&d)[2]) {
  const float2 o = __ffma2_rn(w, make_float2(d[0], d[1]), make_float2(acc[0], acc[1]));
  acc[0] = o.x;
  acc[1] = o.y;
}
// a weight as the multiply-add above takes it: for two columns twice, so that it
// comes out of shared memory as the register pair the packed instruction wants
template <int R> struct Weight;
template <> struct Weight<1> { typedef float t; static __device__ __forceinline__ t of(float w) { return w; } };
template <> struct Weight<2> { typedef float2 t; static __device__ __forceinline__ t of(float w) { return make_float2(w, w); } };
template <typename T, int R>
__device__ __forceinline__ void sub_v(T (&d)[R], const T (&c)[R]) {
#pragma unroll
  for (int r = 0; r < R; ++r) d[r] -= c[r];
}
template <>
__device__ __forceinline__ void sub_v<float, 2>(float (&d)[2], const float (&c)[2]) {
  const float2 o = __fadd2_rn(make_float2(d[0], d[1]), make_float2(-c[0], -c[1]));
  d[0] = o.x;
  d[1] = o.y;
}

// what a cell's warp reads before its node values: the stencil line starts (lane
// ln < 16) and the brick-face split; the index of node x of line ln is
// x < split ? s0 + x : s1 + x - split
struct CellHead {
  int2 line;
  int split;
  int32_t r0, r1;
};

template <int NP>
__device__ __forceinline__ CellHead cell_head(const CellArgs &A, int64_t cid, int lane) {
  CellHead h;
  const int lx = (int)(__ldg(A.ckey + cid) & 7u);
  h.split = (lx + NP - 1 < 8) ? NP : 8 - lx;
  h.line = __ldg(A.lines + cid * 16 + (lane & 15));
  h.r0 = __ldg(A.cstart + cid);
  h.r1 = __ldg(A.cstart + cid + 1);
  return h;
}

// One warp per cell and group of 32 R columns, R adjacent ones per lane.  The lane
// takes the cell's nodes plane by plane (z), 16 values times R columns in registers,
// and applies w_x, w_y, w_z of up to CHUNK rows one after the other.  A weight that a
// warp reads from shared memory takes the LSU a wavefront whatever its width, so
// rows read the 9 weights of a plane and not 16 products of two and the third
// (850 -> 800 us of the 64-column product on the sphere at h = 1/128, whose
// multiply-adds take 230; 16 warps per SM then wait for L2 and for each other's
// 64 node rows of 256 B in L1).  The lines of the next cell are read while this one
// is worked on.
//
// The node values enter as differences to a value u_c of the cell and each row
// adds u_c - u_i, which equals sum_n w_n (u_n - u_i) for any u_c since sum_n w_n = 1;
// rounding then stays relative to local differences.  They are smallest around the
// middle of the stencil, where the rows' closest points lie: u_c is the mean of the
// cubic stencil's nodes 1 and 2 on its diagonal, or the quadratic's middle node.  With
// the first node for u_c the product's error against FP64 was, with 64 columns of smooth
// plus rough fields, 6.06e-8 (sphere h = 1/128, cubic) and 5.82e-8 (h = 1/64, quadratic),
// above the 5.86e-8 and 5.45e-8 of differences to each row's own u_i; it is 5.58e-8 and
// 4.78e-8 now (gather and combine 1322 -> 1338 us and 243 -> 241 us).
template <int DIM, int NP, int R>
__global__ void __launch_bounds__(WARPS * 32, 2)
    gather_cells_kernel(CellArgs A, const float *__restrict__ tc, float cs, const float *__restrict__ u,
                        float *__restrict__ a, int nrhs, unsigned ld) {
  constexpr int NZ = (DIM == 3) ? NP : 1;
  __shared__ __align__(16) float s_w[WARPS][CHUNK][3][4];
  __shared__ int32_t s_row[WARPS][CHUNK];
  __shared__ __align__(16) int32_t s_idx[WARPS][16 * 4];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int ngroups = (nrhs + 32 * R - 1) / (32 * R);
  const int64_t items = A.ncells * ngroups;
  if (warp >= items) return;
  int64_t cid = (ngroups == 1) ? warp : warp / ngroups;
  CellHead h = cell_head<NP>(A, cid, lane);
  const int ax = lane >> 3, j0 = lane & 7;
  for (int64_t it = warp; it < items; it += nwarps) {
    const int col = ((int)(it - cid * ngroups) * 32 + lane) * R;
    const bool on = col < nrhs;
    const float *ul = u + (on ? col : 0);  // lanes past the last column read the first ones (and store nothing)
    const int32_t r0 = h.r0, r1 = h.r1;
    if (lane < 16) {  // node x of line cz * 4 + cy at s_idx[line * 4 + x]
      int4 o;
      o.x = h.line.x;
      o.y = (1 < h.split) ? h.line.x + 1 : h.line.y + (1 - h.split);
      o.z = (2 < h.split) ? h.line.x + 2 : h.line.y + (2 - h.split);
      o.w = (3 < h.split) ? h.line.x + 3 : h.line.y + (3 - h.split);
      *reinterpret_cast<int4 *>(&s_idx[w][lane * 4]) = o;
    }
    const int64_t itn = it + nwarps;
    if (itn < items) {
      cid = (ngroups == 1) ? itn : itn / ngroups;
      h = cell_head<NP>(A, cid, lane);
    }
    for (int32_t c0 = r0; c0 < r1; c0 += CHUNK) {
      const int k = min(CHUNK, r1 - c0);
      const int32_t q = c0 + min(j0, k - 1);  // (rows past the last repeat it)
      if (ax < 3) {  // lane 8 axis + j forms the weights of one axis of row j
        float wt[4] = {1.0f, 0.0f, 0.0f, 0.0f};
        if (ax < DIM) cpm_lagrange<NP, float>(__ldg(tc + 3 * (int64_t)q + ax), wt);
        *reinterpret_cast<float4 *>(s_w[w][j0][ax]) = make_float4(wt[0], wt[1], wt[2], (NP == 4) ? wt[3] : 0.0f);
      } else {
        s_row[w][j0] = __ldg(A.crows + q);
      }
      __syncwarp();
      float part[CHUNK][R], uc[R];
#pragma unroll
      for (int j = 0; j < CHUNK; ++j)
#pragma unroll
        for (int r = 0; r < R; ++r) part[j][r] = 0.0f;
      vld<float, R>(ul + (uint64_t)(unsigned)s_idx[w][(DIM == 3) ? 21 : 5] * ld, uc);
      if (NP == 4) {
        float ud[R];
        vld<float, R>(ul + (uint64_t)(unsigned)s_idx[w][(DIM == 3) ? 42 : 10] * ld, ud);
#pragma unroll
        for (int r = 0; r < R; ++r) uc[r] = 0.5f * uc[r] + 0.5f * ud[r];
      }
#pragma unroll 1
      for (int cz = 0; cz < NZ; ++cz) {
        float d[NP][NP][R];
#pragma unroll
        for (int cy = 0; cy < NP; ++cy) {
          const int4 n4 = *reinterpret_cast<const int4 *>(&s_idx[w][(cz * 4 + cy) * 4]);
          const int32_t n[4] = {n4.x, n4.y, n4.z, n4.w};
#pragma unroll
          for (int cx = 0; cx < NP; ++cx) vld<float, R>(ul + (uint64_t)(unsigned)n[cx] * ld, d[cy][cx]);
        }
#pragma unroll
        for (int cy = 0; cy < NP; ++cy)
#pragma unroll
          for (int cx = 0; cx < NP; ++cx) sub_v<float, R>(d[cy][cx], uc);
#pragma unroll
        for (int j = 0; j < CHUNK; ++j)
          if (j < k) {
            const float4 x4 = *reinterpret_cast<const float4 *>(s_w[w][j][0]);
            const float4 y4 = *reinterpret_cast<const float4 *>(s_w[w][j][1]);
            const float wx[4] = {x4.x, x4.y, x4.z, x4.w}, wy[4] = {y4.x, y4.y, y4.z, y4.w};
            float S[R];
#pragma unroll
            for (int r = 0; r < R; ++r) S[r] = 0.0f;
#pragma unroll
            for (int cy = 0; cy < NP; ++cy) {
              float L[R];
#pragma unroll
              for (int r = 0; r < R; ++r) L[r] = 0.0f;
#pragma unroll
              for (int cx = 0; cx < NP; ++cx) axpy_w(L, Weight<R>::of(wx[cx]), d[cy][cx]);
              axpy_w(S, Weight<R>::of(wy[cy]), L);
            }
            axpy_w(part[j], Weight<R>::of(s_w[w][j][2][cz]), S);
          }
      }
      float ui[CHUNK][R];
#pragma unroll
      for (int j = 0; j < CHUNK; ++j) vld<float, R>(ul + (uint64_t)(unsigned)s_row[w][j] * ld, ui[j]);
      if (on)
#pragma unroll
        for (int j = 0; j < CHUNK; ++j)
          if (j < k) {
            float o[R];
#pragma unroll
            for (int r = 0; r < R; ++r) o[r] = cs * (part[j][r] + (uc[r] - ui[j][r]));
            vst<float, R>(a + (uint64_t)(unsigned)s_row[w][j] * ld + col, o);
          }
      __syncwarp();
    }
  }
}

// FP64: the sums of fixed.cuh, with an exponent per column and cell.  A warp
// takes 16 columns of a cell: its half-warps load every other node and put the
// node differences as integer halves into shared memory (8 KB a warp), then take
// every other row of the cell, so that both read the same shared-memory words in
// one broadcast.  64 nodes in the registers of a lane (254 of them) left 2 warps
// per scheduler, too few for the multiply-adds' latency: 3.6 ms on the torus at
// h = 1/64 with 64 columns (34M row columns), 5.8 ms in FP64 arithmetic.
constexpr int FXC = 16;  // columns per warp
constexpr int FXW = 4;   // warps per block

template <bool DIFF, int DIM, int NP>
__global__ void __launch_bounds__(FXW * 32, 5)
    gather_cells_fx_kernel(CellArgs A, const double *__restrict__ tc, double cs, const double *__restrict__ u,
                           double *__restrict__ a, int nrhs, unsigned ld) {
  constexpr int NZ = (DIM == 3) ? NP : 1;
  constexpr int SLOTS = 16 * NZ;  // node x of line cz * 4 + cy at (cz * 4 + cy) * 4 + x
  __shared__ __align__(16) int2 s_d[FXW][SLOTS][FXC];
  __shared__ __align__(16) int2 s_w[FXW][CHUNK][3][4];
  __shared__ int32_t s_row[FXW][CHUNK];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, half = lane >> 4, lc = lane & 15;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int ngroups = (nrhs + FXC - 1) / FXC;
  const int64_t items = A.ncells * ngroups;  // groups of a cell go to neighbouring warps
  for (int64_t it = warp; it < items; it += nwarps) {
    const int64_t cid = (ngroups == 1) ? it : it / ngroups;
    const int col = (int)(it - cid * ngroups) * FXC + lc;
    const bool on = col < nrhs;
    const CellHead h = cell_head<NP>(A, cid, lane);
    const int k0 = min(CHUNK, h.r1 - h.r0);
    // weights of the first rows while the node values are on their way
    const int ax0 = lane >> 3, j0 = lane & 7;
    double t0 = 1.0;
    if (ax0 < DIM && j0 < k0) t0 = __ldg(tc + 3 * (int64_t)(h.r0 + j0) + ax0);
    const double *uc_ = u + (on ? col : 0);
    double d[SLOTS / 2];
#pragma unroll
    for (int s = 0; s < SLOTS / 2; ++s) {
      // half-warp 0 takes x = 0, 2, half-warp 1 x = 1, 3 of each line
      const int ln = s >> 1, x = (s & 1) * 2 + half;
      d[s] = 0.0;
      if ((ln & 3) >= NP) continue;
      const int2 se = make_int2(__shfl_sync(0xffffffffu, h.line.x, ln), __shfl_sync(0xffffffffu, h.line.y, ln));
      const int32_t idx = (x < h.split) ? se.x + x : se.y + (x - h.split);
      if (x < NP) d[s] = __ldg(uc_ + (uint64_t)(unsigned)idx * ld);
    }
    const double uc = __shfl_sync(0xffffffffu, d[0], lc);
    unsigned top = 0;
#pragma unroll
    for (int s = 0; s < SLOTS / 2; ++s) {
      const int ln = s >> 1, x = (s & 1) * 2 + half;
      if ((ln & 3) >= NP) continue;
      d[s] = (x < NP) ? d[s] - uc : 0.0;
      top = max(top, fx_key(d[s]));
    }
    top = max(top, __shfl_xor_sync(0xffffffffu, top, 16));
    const double sc = fx_cell_scale<DIM>(top);
#pragma unroll
    for (int s = 0; s < SLOTS / 2; ++s) {
      const int ln = s >> 1, x = (s & 1) * 2 + half;
      if ((ln & 3) >= NP) continue;
      int2 o;
      halves(fx_of(d[s], (int)(top >> 20), 8), o.x, o.y);
      s_d[w][ln * 4 + x][lc] = o;
    }
    for (int32_t c0 = h.r0; c0 < h.r1; c0 += CHUNK) {
      const int k = min(CHUNK, h.r1 - c0);
      if (ax0 < 3) {  // lane 8 axis + j forms the weights of one axis of row j
        if (c0 != h.r0 && ax0 < DIM && j0 < k) t0 = __ldg(tc + 3 * (int64_t)(c0 + j0) + ax0);
        int32_t wh[4] = {0, 0, 0, 0}, wl[4] = {0, 0, 0, 0};
        if (ax0 < DIM) fixed_weights<NP>(t0, wh, wl);
#pragma unroll
        for (int q = 0; q < 4; ++q) s_w[w][j0][ax0][q] = make_int2(wh[q], wl[q]);
      }
      if (lane < k) s_row[w][lane] = __ldg(A.crows + c0 + lane);
      __syncwarp();
#pragma unroll 1
      for (int j = half; j < k; j += 2) {
        const int4 *wp = reinterpret_cast<const int4 *>(&s_w[w][j][0][0]);
        const int4 x0 = wp[0], x1 = wp[1], y0 = wp[2], y1 = wp[3];
        const int32_t yh_[4] = {y0.x, y0.z, y1.x, y1.z}, yl_[4] = {y0.y, y0.w, y1.y, y1.w};
        const int2(*dn)[FXC] = &s_d[w][0];
        const unsigned row = (unsigned)s_row[w][j];
        const double ui = (DIFF && on) ? __ldg(uc_ + (uint64_t)row * ld) : 0.0;
        long long zh = 0, zr = HALF;
#pragma unroll
        for (int cz = 0; cz < NZ; ++cz) {
          long long yh = 0, yr = HALF;
#pragma unroll
          for (int cy = 0; cy < NP; ++cy) {
            const int b = (cz * 4 + cy) * 4;
            long long xh = 0, xr = HALF;
            const int2 n0 = dn[b][lc], n1 = dn[b + 1][lc], n2 = dn[b + 2][lc];
            mac(xh, xr, x0.x, x0.y, n0.x, n0.y);
            mac(xh, xr, x0.z, x0.w, n1.x, n1.y);
            mac(xh, xr, x1.x, x1.y, n2.x, n2.y);
            if (NP == 4) {
              const int2 n3 = dn[b + 3][lc];
              mac(xh, xr, x1.z, x1.w, n3.x, n3.y);
            }
            int32_t lh, ll;
            halves(xh + high_word(xr), lh, ll);
            mac(yh, yr, yh_[cy], yl_[cy], lh, ll);
          }
          if constexpr (DIM == 3) {
            int32_t mh, ml;
            halves(yh + high_word(yr), mh, ml);
            const int2 wz = s_w[w][j][2][cz];
            mac(zh, zr, wz.x, wz.y, mh, ml);
          } else {
            zh = yh;
            zr = yr;
          }
        }
        if (on) {
          const double b = DIFF ? uc - ui : uc;
          double acc;
          if (sc > 0.0) acc = scaled_sum(sc, zh + high_word(zr), b);
          else acc = slow_row<DIM, NP>(tc + 3 * (int64_t)(c0 + j), A.lines + cid * 16, h.split, uc_, ld, uc) + b;
          if (cs != 1.0) acc *= cs;
          a[(uint64_t)row * ld + col] = acc;
        }
      }
      __syncwarp();
    }
  }
}

// a_i += sum over the row's flipped entries of w (u_twin - u_node): one warp
// per special row with flips, lanes over R adjacent columns
template <typename T, int R>
__global__ void __launch_bounds__(256) correct_kernel(const int32_t *__restrict__ crow,
                                                      const int32_t *__restrict__ cstart,
                                                      const int32_t *__restrict__ cnode,
                                                      const int32_t *__restrict__ ccol, const T *__restrict__ cw,
                                                      int64_t ncorr, T cs, const T *__restrict__ u,
                                                      T *__restrict__ a, int nrhs, int64_t ld_) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int ngroups = (nrhs + 32 * R - 1) / (32 * R);
  for (int64_t q = warp; q < ncorr; q += nwarps) {
    const int64_t row = __ldg(crow + q);
    const int32_t e0 = __ldg(cstart + q), e1 = __ldg(cstart + q + 1);
    for (int grp = 0; grp < ngroups; ++grp) {
      const int col = (grp * 32 + lane) * R;
      if (col >= nrhs) continue;
      T acc[R];
#pragma unroll
      for (int r = 0; r < R; ++r) acc[r] = T(0);
#pragma unroll 4
      for (int32_t e = e0; e < e1; ++e) {
        const T w = __ldg(cw + e);
        T ut[R], un[R];
        vld<T, R>(u + (int64_t)__ldg(ccol + e) * ld_ + col, ut);
        vld<T, R>(u + (int64_t)__ldg(cnode + e) * ld_ + col, un);
#pragma unroll
        for (int r = 0; r < R; ++r) acc[r] += w * (ut[r] - cs * un[r]);
      }
      T av[R];
      vld<T, R>(a + row * ld_ + col, av);
#pragma unroll
      for (int r = 0; r < R; ++r) av[r] += acc[r];
      vst<T, R>(a + row * ld_ + col, av);
    }
  }
}

// per cell the start of each of its stencil lines along x (slot cz * 4 + cy of
// 16; np1^2 used in 3D, np1 in 2D): s0 the DOF of the line's first node; s1 the
// DOF of its first node past the brick's x face where the line crosses it (-1
// otherwise)
__global__ void cell_lines_kernel(BandView v, const uint32_t *cell_key, int64_t ncells, int2 *lines) {
  const int np1 = v.np1;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < ncells * 16;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t cid = t >> 4;
    const int ln = (int)(t & 15);
    const int cy = ln & 3, cz = ln >> 2;
    int2 out = make_int2(-1, -1);
    if (cy < np1 && (v.dim == 3 ? cz < np1 : cz == 0)) {
      const uint32_t key = cell_key[cid];
      const int32_t b = (int32_t)(key >> 9);
      const int l = (int)(key & 511u);
      const int lx = l & 7, ly = (l >> 3) & 7, lz = l >> 6;
      out.x = cpm_node_index(v, b, lx, ly + cy, lz + cz);
      if (lx + np1 - 1 >= 8) out.y = cpm_node_index(v, b, 8, ly + cy, lz + cz);
    }
    lines[t] = out;
  }
}

// the rows' fractional stencil positions in cell order, so that a warp's rows
// read them as one contiguous run
__global__ void cell_frac_kernel(const int32_t *rows, int64_t NS, const double *t64, double *tc64, float *tc32) {
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < NS; q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = rows[q];
    for (int e = 0; e < 3; ++e) {
      const double t = t64[3 * i + e];
      tc64[3 * q + e] = t;
      tc32[3 * q + e] = (float)t;
    }
  }
}

__global__ void row_cell_kernel(const int32_t *cell_start, int64_t ncells, int32_t *row_cell) {
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < ncells; c += (int64_t)gridDim.x * blockDim.x)
    for (int32_t q = cell_start[c]; q < cell_start[c + 1]; ++q) row_cell[q] = (int32_t)c;
}

// single right-hand side: one thread per PDE row, rows taken in cell order so
// that the rows of a cell (same 64 nodes) run in neighbouring threads and share
// the cell's line table and node values in cache
template <typename T, bool DIFF, int DIM, int NP>
__global__ void __launch_bounds__(256) gather1_kernel(ApplyArgs<T> A, const int32_t *__restrict__ crows,
                                                      const int32_t *__restrict__ row_cell,
                                                      const uint32_t *__restrict__ ckey,
                                                      const int2 *__restrict__ lines, int64_t NS, T cs,
                                                      const T *__restrict__ u, T *__restrict__ a) {
  constexpr int NZ = (DIM == 3) ? NP : 1;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < NS; q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t row = __ldg(crows + q);
    const int32_t cid = __ldg(row_cell + q);
    const int lx = (int)(__ldg(ckey + cid) & 7u);
    const int split = (lx + NP - 1 < 8) ? NP : 8 - lx;
    const int2 *ln = lines + (int64_t)cid * 16;
    T wx[4], wy[4], wz[4];
    cpm_lagrange<NP, T>(__ldg(A.t + 3 * row), wx);
    cpm_lagrange<NP, T>(__ldg(A.t + 3 * row + 1), wy);
    if (DIM == 3) cpm_lagrange<NP, T>(__ldg(A.t + 3 * row + 2), wz);
    else { wz[0] = T(1); wz[1] = wz[2] = wz[3] = T(0); }
    const T uc = DIFF ? __ldg(u + __ldg(&ln[0].x)) : T(0);
    T acc = T(0);
#pragma unroll
    for (int cz = 0; cz < NZ; ++cz) {
      T pz = T(0);
#pragma unroll
      for (int cy = 0; cy < NP; ++cy) {
        const int2 se = __ldg(ln + cz * 4 + cy);
        T line = T(0);
#pragma unroll
        for (int cx = 0; cx < NP; ++cx) {
          const int32_t idx = (cx < split) ? (se.x + cx) : (se.y + (cx - split));
          line += wx[cx] * (__ldg(u + idx) - uc);
        }
        pz += wy[cy] * line;
      }
      acc += wz[cz] * pz;
    }
    if (DIFF) acc += uc - __ldg(u + row);
    a[row] = cs * acc;
  }
}

}  // namespace

void cpm_free_cells(cpm_ctx *c) {
  cpm_free_fused1(c);
  cudaFree(c->d_cell_start); cudaFree(c->d_cell_rows); cudaFree(c->d_cell_key); cudaFree(c->d_nbr8);
  cudaFree(c->d_corr_row); cudaFree(c->d_corr_start); cudaFree(c->d_corr_node); cudaFree(c->d_corr_col);
  cudaFree(c->d_corr_w64); cudaFree(c->d_corr_w32); cudaFree(c->d_cell_lines); cudaFree(c->d_row_cell);
  cudaFree(c->d_tc64); cudaFree(c->d_tc32);
  c->d_tc64 = nullptr; c->d_tc32 = nullptr;
  c->d_cell_lines = nullptr; c->d_row_cell = nullptr;
  c->d_cell_start = nullptr; c->d_cell_rows = nullptr; c->d_cell_key = nullptr; c->d_nbr8 = nullptr;
  c->d_corr_row = nullptr; c->d_corr_start = nullptr; c->d_corr_node = nullptr; c->d_corr_col = nullptr;
  c->d_corr_w64 = nullptr; c->d_corr_w32 = nullptr;
  c->ncells = 0; c->nbulk = 0; c->ncorr = 0; c->ncorr_ent = 0;
}

cpm_status cpm_build_cells(cpm_ctx *c) {
  cudaStream_t st = c->stream;
  cpm_free_cells(c);
  const int64_t nkeys = c->nb * 512;
  const int64_t nsp = std::max<int64_t>(c->nspec, 1);
  int32_t *count = nullptr, *offs = nullptr, *flag = nullptr, *cellpos = nullptr, *d_tot = nullptr;
  int32_t *ccnt = nullptr, *coffs = nullptr, *cflag = nullptr, *cpos = nullptr;
  int32_t h_tot = 0, h_cells = 0, h_ent = 0, h_rows = 0;
  cpm_status rc = CPM_OK;
#define TRY(x)                                             \
  do {                                                     \
    cudaError_t e_ = (x);                                  \
    if (e_) { rc = cpm_internal_cuda_err(e_); goto done; } \
  } while (0)
  TRY(cudaMalloc(&count, sizeof(int32_t) * nkeys));
  TRY(cudaMalloc(&offs, sizeof(int32_t) * nkeys));
  TRY(cudaMalloc(&flag, sizeof(int32_t) * nkeys));
  TRY(cudaMalloc(&cellpos, sizeof(int32_t) * nkeys));
  TRY(cudaMalloc(&d_tot, sizeof(int32_t)));
  TRY(cudaMemsetAsync(count, 0, sizeof(int32_t) * nkeys, st));
  cell_count_kernel<<<cpm_grid(c->NS, 256), 256, 0, st>>>(c->d_rbase, c->NS, count);
  TRY(cpm_exclusive_scan(count, offs, nkeys, d_tot, st));
  TRY(cudaMemcpyAsync(&h_tot, d_tot, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
  flag_nonzero_kernel<<<cpm_grid(nkeys, 256), 256, 0, st>>>(count, nkeys, flag);
  TRY(cpm_exclusive_scan(flag, cellpos, nkeys, d_tot, st));
  TRY(cudaMemcpyAsync(&h_cells, d_tot, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
  TRY(cudaStreamSynchronize(st));
  c->nbulk = h_tot;
  c->ncells = h_cells;
  TRY(cudaMalloc(&c->d_cell_rows, sizeof(int32_t) * std::max<int64_t>(c->nbulk, 1)));
  TRY(cudaMalloc(&c->d_cell_start, sizeof(int32_t) * (c->ncells + 1)));
  TRY(cudaMalloc(&c->d_cell_key, sizeof(uint32_t) * std::max<int64_t>(c->ncells, 1)));
  // scatter with a cursor copy of the offsets, then order each bucket
  TRY(cudaMemcpyAsync(flag, offs, sizeof(int32_t) * nkeys, cudaMemcpyDeviceToDevice, st));
  cell_scatter_kernel<<<cpm_grid(c->NS, 256), 256, 0, st>>>(c->d_rbase, c->NS, flag, c->d_cell_rows);
  cell_finish_kernel<<<cpm_grid(nkeys, 256), 256, 0, st>>>(count, offs, cellpos, nkeys, c->d_cell_rows,
                                                           c->d_cell_start, c->d_cell_key);
  set_i32_kernel<<<1, 1, 0, st>>>(c->d_cell_start + c->ncells, h_tot);
  TRY(cudaMalloc(&c->d_cell_lines, sizeof(int2) * 16 * std::max<int64_t>(c->ncells, 1)));
  TRY(cudaMalloc(&c->d_row_cell, sizeof(int32_t) * std::max<int64_t>(c->NS, 1)));
  TRY(cudaMalloc(&c->d_tc64, sizeof(double) * 3 * std::max<int64_t>(c->NS, 1)));
  TRY(cudaMalloc(&c->d_tc32, sizeof(float) * 3 * std::max<int64_t>(c->NS, 1)));
  cell_frac_kernel<<<cpm_grid(c->NS, 256), 256, 0, st>>>(c->d_cell_rows, c->NS, c->d_t64, c->d_tc64, c->d_tc32);
  if (c->ncells > 0) {
    cell_lines_kernel<<<cpm_grid(c->ncells * 16, 256), 256, 0, st>>>(c->view(), c->d_cell_key, c->ncells,
                                                                    reinterpret_cast<int2 *>(c->d_cell_lines));
    row_cell_kernel<<<cpm_grid(c->ncells, 256), 256, 0, st>>>(c->d_cell_start, c->ncells, c->d_row_cell);
  }
  TRY(cudaMalloc(&c->d_nbr8, sizeof(int32_t) * 8 * std::max<int64_t>(c->NS, 1)));
  nbr8_kernel<<<cpm_grid(c->NS, 256), 256, 0, st>>>(c->view(), c->d_rself, c->d_rbase, c->d_spec_of, c->d_spec_fcol,
                                                    c->d_nbr8);
  TRY(cudaGetLastError());
  // flipped interpolation entries of the special rows
  TRY(cudaMalloc(&ccnt, sizeof(int32_t) * nsp));
  TRY(cudaMalloc(&coffs, sizeof(int32_t) * nsp));
  TRY(cudaMalloc(&cflag, sizeof(int32_t) * nsp));
  TRY(cudaMalloc(&cpos, sizeof(int32_t) * nsp));
  if (c->nspec > 0) {
    corr_count_kernel<<<cpm_grid(c->nspec, 128), 128, 0, st>>>(c->view(), c->d_spec_row, c->nspec, c->d_rbase,
                                                               c->d_spec_ecol, ccnt);
    TRY(cpm_exclusive_scan(ccnt, coffs, c->nspec, d_tot, st));
    TRY(cudaMemcpyAsync(&h_ent, d_tot, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    flag_nonzero_kernel<<<cpm_grid(c->nspec, 256), 256, 0, st>>>(ccnt, c->nspec, cflag);
    TRY(cpm_exclusive_scan(cflag, cpos, c->nspec, d_tot, st));
    TRY(cudaMemcpyAsync(&h_rows, d_tot, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    TRY(cudaStreamSynchronize(st));
  }
  c->ncorr = h_rows;
  c->ncorr_ent = h_ent;
  TRY(cudaMalloc(&c->d_corr_row, sizeof(int32_t) * std::max<int64_t>(c->ncorr, 1)));
  TRY(cudaMalloc(&c->d_corr_start, sizeof(int32_t) * (c->ncorr + 1)));
  TRY(cudaMalloc(&c->d_corr_node, sizeof(int32_t) * std::max<int64_t>(c->ncorr_ent, 1)));
  TRY(cudaMalloc(&c->d_corr_col, sizeof(int32_t) * std::max<int64_t>(c->ncorr_ent, 1)));
  TRY(cudaMalloc(&c->d_corr_w64, sizeof(double) * std::max<int64_t>(c->ncorr_ent, 1)));
  TRY(cudaMalloc(&c->d_corr_w32, sizeof(float) * std::max<int64_t>(c->ncorr_ent, 1)));
  set_i32_kernel<<<1, 1, 0, st>>>(c->d_corr_start + c->ncorr, h_ent);
  if (c->ncorr > 0)
    corr_fill_kernel<<<cpm_grid(c->nspec, 128), 128, 0, st>>>(c->view(), c->d_spec_row, c->nspec, c->d_rbase,
                                                              c->d_spec_ecol, c->d_spec_ew, ccnt, coffs, cpos,
                                                              c->d_corr_row, c->d_corr_start, c->d_corr_node,
                                                              c->d_corr_col, c->d_corr_w64, c->d_corr_w32);
  TRY(cudaGetLastError());
  TRY(cudaStreamSynchronize(st));
  rc = cpm_build_fused1(c);
done:
#undef TRY
  cudaFree(count); cudaFree(offs); cudaFree(flag); cudaFree(cellpos); cudaFree(d_tot);
  cudaFree(ccnt); cudaFree(coffs); cudaFree(cflag); cudaFree(cpos);
  if (rc != CPM_OK) cpm_free_cells(c);
  return rc;
}

// the x passes that cpm_tune_info names; the gathers take z planes and have no use
// for them, recorded shapes stay valid
int cpm_cells_default_xh(int np1, bool fp64, int rpl) {
  return (np1 == 3) ? ((fp64 && rpl == 2) ? 3 : 1) : (fp64 ? (rpl == 2 ? 4 : 2) : 2);
}

// 4 blocks per SM (two rounds) with two columns per lane, 16 with one: 1324 / 1353 us
// of the 64-column product on the sphere at h = 1/128, 1202 / 1061 us of 24 columns (4 / 16)
int cpm_cells_default_blocks(int rpl) { return rpl == 2 ? 4 : 16; }

static CellArgs cell_args(const cpm_ctx *c) {
  return CellArgs{c->d_cell_start, c->d_cell_rows, c->d_cell_key, reinterpret_cast<const int2 *>(c->d_cell_lines),
                  c->ncells};
}

template <int DIM, int NP, int R>
static void launch_cells_k(const cpm_ctx *c, float cs, const float *u, float *a, int nrhs, int64_t ld,
                           cudaStream_t st) {
  const int per_sm = c->tune.cells_blocks_per_sm > 0 ? c->tune.cells_blocks_per_sm : cpm_cells_default_blocks(R);
  const int64_t items = c->ncells * ((nrhs + 32 * R - 1) / (32 * R));
  const unsigned g = (unsigned)std::min<int64_t>((items + WARPS - 1) / WARPS, (int64_t)c->nsm * per_sm);
  gather_cells_kernel<DIM, NP, R><<<g, WARPS * 32, 0, st>>>(cell_args(c), c->d_tc32, cs, u, a, nrhs, (unsigned)ld);
}

template <int R>
static void launch_cells(const cpm_ctx *c, float cs, const float *u, float *a, int nrhs, int64_t ld, cudaStream_t st) {
  if (c->dim == 3) {
    if (c->p == 2) launch_cells_k<3, 3, R>(c, cs, u, a, nrhs, ld, st);
    else launch_cells_k<3, 4, R>(c, cs, u, a, nrhs, ld, st);
  } else {
    if (c->p == 2) launch_cells_k<2, 3, R>(c, cs, u, a, nrhs, ld, st);
    else launch_cells_k<2, 4, R>(c, cs, u, a, nrhs, ld, st);
  }
}

template <bool DIFF>
static void launch_cells_fx(const cpm_ctx *c, double cs, const double *u, double *a, int nrhs, int64_t ld,
                            cudaStream_t st) {
  const int64_t items = c->ncells * ((nrhs + FXC - 1) / FXC);
  const unsigned g = (unsigned)std::min<int64_t>((items + FXW - 1) / FXW, (int64_t)c->nsm * 64);
  const CellArgs A = cell_args(c);
#define CPM_FX(D, NP) \
  gather_cells_fx_kernel<DIFF, D, NP><<<g, FXW * 32, 0, st>>>(A, c->d_tc64, cs, u, a, nrhs, (unsigned)ld)
  if (c->dim == 3) {
    if (c->p == 2) CPM_FX(3, 3); else CPM_FX(3, 4);
  } else {
    if (c->p == 2) CPM_FX(2, 3); else CPM_FX(2, 4);
  }
#undef CPM_FX
}

// the flipped entries of a batch
template <typename T, int R>
static int launch_correct(const cpm_ctx *c, T cs, const T *u, T *a, int nrhs, int64_t ld, cudaStream_t st) {
  if (c->ncorr == 0) return 0;
  const T *cw;
  if constexpr (sizeof(T) == 8) cw = reinterpret_cast<const T *>(c->d_corr_w64);
  else cw = reinterpret_cast<const T *>(c->d_corr_w32);
  unsigned gc = (unsigned)std::min<int64_t>((c->ncorr + 7) / 8, (int64_t)c->nsm * 16);
  correct_kernel<T, R><<<gc, 256, 0, st>>>(c->d_corr_row, c->d_corr_start, c->d_corr_node, c->d_corr_col, cw,
                                           c->ncorr, cs, u, a, nrhs, ld);
  return 1;
}

// FP32 takes the difference form only (no caller wants E u itself in FP32)
template <>
int cpm_launch_gather_cells<float>(const cpm_ctx *c, float cs, const float *u, float *a, int nrhs, int64_t ld,
                                   cudaStream_t st, bool /*diff*/, int rpl) {
  if (c->ncells == 0) return 0;
  if (rpl == 2) {
    launch_cells<2>(c, cs, u, a, nrhs, ld, st);
    return 1 + launch_correct<float, 2>(c, cs, u, a, nrhs, ld, st);
  }
  launch_cells<1>(c, cs, u, a, nrhs, ld, st);
  return 1 + launch_correct<float, 1>(c, cs, u, a, nrhs, ld, st);
}

template <>
int cpm_launch_gather_cells<double>(const cpm_ctx *c, double cs, const double *u, double *a, int nrhs, int64_t ld,
                                    cudaStream_t st, bool diff, int rpl) {
  if (c->ncells == 0) return 0;
  if (diff) launch_cells_fx<true>(c, cs, u, a, nrhs, ld, st);
  else launch_cells_fx<false>(c, cs, u, a, nrhs, ld, st);
  return 1 + (rpl == 2 ? launch_correct<double, 2>(c, cs, u, a, nrhs, ld, st)
                       : launch_correct<double, 1>(c, cs, u, a, nrhs, ld, st));
}

template <typename T>
void cpm_launch_gather1(const cpm_ctx *c, const ApplyArgs<T> &A, T cs, const T *u, T *a, cudaStream_t st) {
  const unsigned g = cpm_grid(c->NS, 256);
  const int2 *lines = reinterpret_cast<const int2 *>(c->d_cell_lines);
#define CPM_G1(D, NP)                                                                                         \
  gather1_kernel<T, true, D, NP><<<g, 256, 0, st>>>(A, c->d_cell_rows, c->d_row_cell, c->d_cell_key, lines, \
                                                    c->NS, cs, u, a)
  if (c->dim == 3) {
    if (c->p == 2) CPM_G1(3, 3); else CPM_G1(3, 4);
  } else {
    if (c->p == 2) CPM_G1(2, 3); else CPM_G1(2, 4);
  }
#undef CPM_G1
}
template void cpm_launch_gather1<float>(const cpm_ctx *, const ApplyArgs<float> &, float, const float *, float *,
                                        cudaStream_t);
template void cpm_launch_gather1<double>(const cpm_ctx *, const ApplyArgs<double> &, double, const double *, double *,
                                         cudaStream_t);
