// tile.cu -- E u for one or a few right-hand sides: warp tiles of stencil cells.
//
// A warp takes CT consecutive cells (cells.cu) and stages their node values in
// shared memory (FP64: as differences to each cell's base-node value u_c), then its
// lanes take the tile's rows (~5 per cell, in cell order), one row each: the
// weights of the row, the separable sum over the cell's nodes from shared
// memory, and a_i = sum_j w_j (u_j - u_i), in FP64 from sum_j w_j (u_j - u_c) + (u_c - u_i).  Rows, not cells, are
// spread over the lanes because cells hold between 1 and a dozen rows: one
// thread per cell left a warp waiting for its fullest cell, and 64 FP64 node
// values per thread left 2 blocks of 128 threads per SM.  The staging loads
// take 8 stencil lines of 4 consecutive DOFs per instruction.
//
// FP64 sums run in integers (fixed.cuh).
#include <algorithm>

#include "apply.cuh"
#include "cpm_internal.cuh"
#include "fixed.cuh"

namespace {

constexpr int TW = 4;  // warps per block; warps are independent

template <typename T> struct Node;
template <> struct Node<float> { typedef float t; };
template <> struct Node<double> { typedef int2 t; };

struct TileArgs {
  const int32_t *cstart, *crows, *row_cell;
  const uint32_t *ckey;
  const int2 *lines;
  int64_t ncells;
};

// DIFF: a_i = cs (E u - u)_i; otherwise a_i = cs (E u)_i.
//
// FP64, sphere h = 1/128 (1.70M rows, 309k cells): 140 us (one thread per cell in
// FP64 arithmetic: 820 us), with the multiply-add pipe busy 55 % and the integer
// pipe 46 %; what is left is the latency of the staging loads at 24 warps per SM,
// which is why they are unrolled over 8 cells.  FP32 keeps the node values as they are
// and takes the differences to u_i per row (one rounding less, and no base value to
// pass on: the product on the bumpy sphere at h = 1/640, 43M rows, 1335 -> 1192 us); it
// is held by L1 wavefronts (74 %).
template <typename T, bool DIFF, int DIM, int NP, int CT>
__global__ void __launch_bounds__(TW * 32, (sizeof(T) == 8) ? 6 : 8)
    gather_tile_kernel(TileArgs A, const T *__restrict__ tc, T cs, const T *__restrict__ u, T *__restrict__ a,
                       int nrhs, int64_t ld) {
  constexpr int NZ = (DIM == 3) ? NP : 1;
  constexpr int SLOTS = 16 * NZ;                           // 4 x 4 x NZ, x fastest
  constexpr bool FX = (sizeof(T) == 8);
  typedef typename Node<T>::t V;
  constexpr int STR = SLOTS + 16 / (int)sizeof(V);         // one 16-byte pad: cells start 4 banks apart
  constexpr int PER = (SLOTS + 31) / 32;                   // node slots of a lane per cell (3D)
  constexpr int CPI = (SLOTS < 32) ? 32 / SLOTS : 1;       // cells per staging step (2D: two)
  __shared__ __align__(16) V s_d[TW][CT][STR];
  __shared__ T s_uc[TW][CT];
  __shared__ T s_sc[FX ? TW : 1][FX ? CT : 1];             // FP64: scale of a cell's integers; < 0: plain FP64
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t c0 = ((int64_t)blockIdx.x * TW + w) * CT;
  if (c0 >= A.ncells) return;
  const int nc = (int)min((int64_t)CT, A.ncells - c0);
  const int32_t q0 = __ldg(A.cstart + c0), q1 = __ldg(A.cstart + c0 + nc);
  for (int r = (int)blockIdx.y; r < nrhs; r += (int)gridDim.y) {
    const T *ur = u + r;
    // ---- stage the tile's node values
#pragma unroll(FX ? 8 : 4)
    for (int cb = 0; cb < nc; cb += CPI) {
      const int sub = (CPI > 1) ? lane / SLOTS : 0;
      const int c = cb + sub;
      const bool live = c < nc;
      const int64_t cid = c0 + (live ? c : 0);
      const int lx = (int)(__ldg(A.ckey + cid) & 7u);
      const int split = (lx + NP - 1 < 8) ? NP : 8 - lx;
      T v[PER];
      bool on[PER];
#pragma unroll
      for (int k = 0; k < PER; ++k) {
        const int slot = (CPI > 1) ? (lane & (SLOTS - 1)) : lane + 32 * k;
        const int x = slot & 3, ln = slot >> 2;
        on[k] = live && slot < SLOTS && x < NP && (ln & 3) < NP;
        v[k] = T(0);
        if (on[k]) {
          const int2 se = __ldg(A.lines + cid * 16 + ln);
          const int32_t idx = (x < split) ? (se.x + x) : (se.y + (x - split));
          v[k] = __ldg(ur + (int64_t)idx * ld);
        }
      }
      const T uc = __shfl_sync(0xffffffffu, v[0], (CPI > 1) ? sub * SLOTS : 0);
      T d[PER];
#pragma unroll
      for (int k = 0; k < PER; ++k) d[k] = on[k] ? v[k] - uc : T(0);
      if constexpr (FX) {
        // exponent of the cell's largest difference (fx_key, fx_of and fx_cell_scale
        // written out: as calls they cost this unrolled loop 38 of 215 us a product)
        unsigned top = 0;
#pragma unroll
        for (int k = 0; k < PER; ++k)
          top = max(top, ((unsigned)__double2hiint(d[k]) & 0x7FFFFFFFu) | (unsigned)(__double2loint(d[k]) != 0));
        if (CPI > 1) {
#pragma unroll
          for (int o = SLOTS / 2; o; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
        } else {
          top = __reduce_max_sync(0xffffffffu, top);
        }
        const int em = (int)(top >> 20);
        // |d| < 2^(em - 1022); X = d 2^(1083 - em), |X| < 2^61
#pragma unroll
        for (int k = 0; k < PER; ++k) {
          const int slot = (CPI > 1) ? (lane & (SLOTS - 1)) : lane + 32 * k;
          const int hi = __double2hiint(d[k]);
          const int e = (hi >> 20) & 0x7FF;
          unsigned long long m = ((unsigned long long)(((unsigned)hi & 0xFFFFFu) | 0x100000u) << 32) |
                                 (unsigned)__double2loint(d[k]);
          m = (e == 0) ? 0ull : ((m << 8) >> min(em - e, 63));
          const long long X = (hi < 0) ? -(long long)m : (long long)m;
          if (SLOTS % 32 == 0 || slot < SLOTS) {
            int2 o;
            halves(X, o.x, o.y);
            if (live) s_d[w][c][slot] = o;
          }
        }
        if (live && (lane & (SLOTS - 1 < 31 ? SLOTS - 1 : 31)) == 0) {
          constexpr double back = (DIM == 3) ? 4096.0 / 216.0 : 256.0 / 36.0;
          const bool plain = em >= 2040 || (em < 140 && top != 0u);
          const double sc = __hiloint2double(__double2hiint(back) + ((em - 1083) * (1 << 20)), __double2loint(back));
          s_sc[w][c] = plain ? -1.0 : (top == 0u ? 1.0 : sc);
          s_uc[w][c] = uc;
        }
      } else {
#pragma unroll
        for (int k = 0; k < PER; ++k) {
          const int slot = (CPI > 1) ? (lane & (SLOTS - 1)) : lane + 32 * k;
          if (live && slot < SLOTS) s_d[w][c][slot] = v[k];  // (differences to u_i are taken per row)
        }
      }
    }
    __syncwarp();
    // ---- the tile's rows, one per lane
    for (int32_t q = q0 + lane; q < q1; q += 32) {
      const int64_t row = __ldg(A.crows + q);
      const int c = (int)(__ldg(A.row_cell + q) - c0);
      const T *tq = tc + 3 * (int64_t)q;
      const T ui = DIFF ? __ldg(ur + row * ld) : T(0);
      T acc;
      if constexpr (FX) {
        const T uc = s_uc[w][c];
        int32_t wxh[4], wxl[4], wyh[4], wyl[4], wzh[4], wzl[4];
        fixed_weights<NP>(__ldg(tq), wxh, wxl);
        fixed_weights<NP>(__ldg(tq + 1), wyh, wyl);
        if (DIM == 3) fixed_weights<NP>(__ldg(tq + 2), wzh, wzl);
        const int4 *dn = reinterpret_cast<const int4 *>(&s_d[w][c][0]);
        long long zh = 0, zr = HALF;
#pragma unroll
        for (int cz = 0; cz < NZ; ++cz) {
          long long yh = 0, yr = HALF;
#pragma unroll
          for (int cy = 0; cy < NP; ++cy) {
            const int4 p = dn[(cz * 4 + cy) * 2], s = dn[(cz * 4 + cy) * 2 + 1];
            long long xh = 0, xr = HALF;
            mac(xh, xr, wxh[0], wxl[0], p.x, p.y);
            mac(xh, xr, wxh[1], wxl[1], p.z, p.w);
            mac(xh, xr, wxh[2], wxl[2], s.x, s.y);
            if (NP == 4) mac(xh, xr, wxh[3], wxl[3], s.z, s.w);
            int32_t lh, ll;
            halves(xh + high_word(xr), lh, ll);
            mac(yh, yr, wyh[cy], wyl[cy], lh, ll);
          }
          if constexpr (DIM == 3) {
            int32_t mh, ml;
            halves(yh + high_word(yr), mh, ml);
            mac(zh, zr, wzh[cz], wzl[cz], mh, ml);
          } else {
            zh = yh;
            zr = yr;
          }
        }
        const double sc = s_sc[w][c];
        const double base = DIFF ? uc - ui : uc;
        if (sc > 0.0) {
          acc = scaled_sum(sc, zh + high_word(zr), base);
        } else {
          const int64_t cid = c0 + c;
          const int lx = (int)(__ldg(A.ckey + cid) & 7u);
          acc = slow_row<DIM, NP>(tq, A.lines + cid * 16, (lx + NP - 1 < 8) ? NP : 8 - lx, ur, ld, uc) + base;
        }
      } else {
        T wx[4], wy[4], wz[4];
        cpm_lagrange<NP, T>(__ldg(tq), wx);
        cpm_lagrange<NP, T>(__ldg(tq + 1), wy);
        if (DIM == 3) cpm_lagrange<NP, T>(__ldg(tq + 2), wz);
        else { wz[0] = T(1); wz[1] = wz[2] = wz[3] = T(0); }
        const float4 *dn = reinterpret_cast<const float4 *>(&s_d[w][c][0]);
        // (axis by axis: with products w_y w_z as weights every term took one rounding more)
        float2 p01 = make_float2(0.0f, 0.0f), p23 = p01;
        const float2 mu = make_float2(-ui, -ui);
#pragma unroll
        for (int cz = 0; cz < NZ; ++cz) {
          float2 q01 = make_float2(0.0f, 0.0f), q23 = q01;
#pragma unroll
          for (int cy = 0; cy < NP; ++cy) {
            const float2 g = make_float2(wy[cy], wy[cy]);
            const float4 p = dn[cz * 4 + cy];
            q01 = __ffma2_rn(g, __fadd2_rn(make_float2(p.x, p.y), mu), q01);
            q23 = __ffma2_rn(g, __fadd2_rn(make_float2(p.z, p.w), mu), q23);
          }
          const float2 g = make_float2(wz[cz], wz[cz]);
          p01 = (DIM == 3) ? __ffma2_rn(g, q01, p01) : q01;
          p23 = (DIM == 3) ? __ffma2_rn(g, q23, p23) : q23;
        }
        acc = wx[0] * p01.x;
        acc += wx[1] * p01.y;
        acc += wx[2] * p23.x;
        if (NP == 4) acc += wx[3] * p23.y;
      }
      if (cs != T(1)) acc *= cs;
      a[row * ld + r] = acc;
    }
    __syncwarp();
  }
}

// a_i += sum over the row's flipped entries of w (u_twin - cs u_node): four lanes
// per row and column.  A row has up to 32 flipped entries; one thread walking
// them was a chain of that many dependent loads (20 us on the sphere at h = 1/128).
template <typename T>
__global__ void __launch_bounds__(256) correct_few_kernel(const int32_t *__restrict__ crow,
                                                          const int32_t *__restrict__ cstart,
                                                          const int32_t *__restrict__ cnode,
                                                          const int32_t *__restrict__ ccol, const T *__restrict__ cw,
                                                          int64_t ncorr, T cs, const T *__restrict__ u,
                                                          T *__restrict__ a, int nrhs, int64_t ld) {
  const int sub = threadIdx.x & 3;
  const int64_t stride = ((int64_t)gridDim.x * blockDim.x) >> 2;
  for (int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 2; t < ncorr * nrhs; t += stride) {
    const int64_t q = (nrhs == 1) ? t : t / nrhs;
    const int r = (nrhs == 1) ? 0 : (int)(t - q * nrhs);
    const int32_t e1 = __ldg(cstart + q + 1);
    T acc = T(0);
    for (int32_t e = __ldg(cstart + q) + sub; e < e1; e += 4)
      acc += __ldg(cw + e) * (__ldg(u + (int64_t)__ldg(ccol + e) * ld + r) - cs * __ldg(u + (int64_t)__ldg(cnode + e) * ld + r));
    // the four lanes of a row are active together (the loop bound is theirs)
    const unsigned m = 0xFu << (threadIdx.x & 28);
    acc += __shfl_xor_sync(m, acc, 1);
    acc += __shfl_xor_sync(m, acc, 2);
    if (sub == 0) a[(int64_t)__ldg(crow + q) * ld + r] += acc;
  }
}

template <typename T, bool DIFF, int DIM, int NP, int CT>
void launch_tile(const cpm_ctx *c, const T *tc, T cs, const T *u, T *a, int nrhs, int64_t ld, cudaStream_t st) {
  TileArgs A{c->d_cell_start, c->d_cell_rows, c->d_row_cell, c->d_cell_key,
             reinterpret_cast<const int2 *>(c->d_cell_lines), c->ncells};
  const int64_t tiles = (c->ncells + CT - 1) / CT;
  // where the tiles leave resident warps idle (24 or 32 an SM), the columns are spread
  // over blocks instead of following each other in one: FP64 products of 15 columns on
  // the circle at h = 0.01 39 -> 18 us, on the sphere at h = 1/16 121 -> 98 us
  const int64_t warps = (int64_t)c->nsm * ((sizeof(T) == 8) ? 24 : 32);
  const unsigned gy = (unsigned)std::max<int64_t>(1, std::min<int64_t>(nrhs, warps / tiles));
  const dim3 grid((unsigned)((tiles + TW - 1) / TW), gy);
  gather_tile_kernel<T, DIFF, DIM, NP, CT><<<grid, TW * 32, 0, st>>>(A, tc, cs, u, a, nrhs, ld);
}

template <typename T, bool DIFF>
void launch_tile_any(const cpm_ctx *c, const T *tc, T cs, const T *u, T *a, int nrhs, int64_t ld, cudaStream_t st) {
  // 16 cells (~88 rows: three passes of 32 lanes, 92 % of them at work) where
  // that fills the SMs; 4 cells (two passes) on bands with fewer tiles than
  // 8 warps per SM, whose time is the latency of one tile
  const bool small = c->ncells < (int64_t)16 * 8 * c->nsm;
#define CPM_TILE(D, NP)                                                             \
  (small ? launch_tile<T, DIFF, D, NP, 4>(c, tc, cs, u, a, nrhs, ld, st)             \
         : launch_tile<T, DIFF, D, NP, 16>(c, tc, cs, u, a, nrhs, ld, st))
  if (c->dim == 3) {
    if (c->p == 2) CPM_TILE(3, 3); else CPM_TILE(3, 4);
  } else {
    if (c->p == 2) CPM_TILE(2, 3); else CPM_TILE(2, 4);
  }
#undef CPM_TILE
}

}  // namespace

template <typename T>
int cpm_launch_correct_few(const cpm_ctx *c, T cs, const T *u, T *a, int nrhs, int64_t ld, cudaStream_t st) {
  if (c->ncorr == 0) return 0;
  const T *cw;
  if constexpr (sizeof(T) == 8) cw = reinterpret_cast<const T *>(c->d_corr_w64);
  else cw = reinterpret_cast<const T *>(c->d_corr_w32);
  correct_few_kernel<T><<<cpm_grid(4 * c->ncorr * nrhs, 256), 256, 0, st>>>(c->d_corr_row, c->d_corr_start,
                                                                            c->d_corr_node, c->d_corr_col, cw,
                                                                            c->ncorr, cs, u, a, nrhs, ld);
  return 1;
}

template <typename T>
int cpm_launch_gather_tile(const cpm_ctx *c, T cs, const T *u, T *a, int nrhs, int64_t ld, cudaStream_t st,
                           bool diff) {
  if (c->ncells == 0) return 0;
  const T *tc;
  if constexpr (sizeof(T) == 8) tc = reinterpret_cast<const T *>(c->d_tc64);
  else tc = reinterpret_cast<const T *>(c->d_tc32);
  if constexpr (sizeof(T) == 8) {
    if (diff) launch_tile_any<T, true>(c, tc, cs, u, a, nrhs, ld, st);
    else launch_tile_any<T, false>(c, tc, cs, u, a, nrhs, ld, st);
  } else {  // (no caller wants E u itself in FP32)
    launch_tile_any<T, true>(c, tc, cs, u, a, nrhs, ld, st);
  }
  return 1 + cpm_launch_correct_few<T>(c, cs, u, a, nrhs, ld, st);
}
#define CPM_TILE_INST(T)                                                                                       \
  template int cpm_launch_correct_few<T>(const cpm_ctx *, T, const T *, T *, int, int64_t, cudaStream_t);     \
  template int cpm_launch_gather_tile<T>(const cpm_ctx *, T, const T *, T *, int, int64_t, cudaStream_t, bool);
CPM_TILE_INST(float)
CPM_TILE_INST(double)
