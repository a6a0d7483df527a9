// Kernels of the Fira step (Algorithm 1's loop body) in fp32 precision, grouped over a list of
// matrices of any size and pitch: one launch per phase covers every matrix of the list.
//
// What is to be made (l = unprojected index, d = projected index, Pi = the d x r projection):
//   1. project      R[l][j] = sum_d G(d,l) Pi[d][j]  (R = P^T G); epilogue: M, V update, N (Eq. 2-4) and the
//                   row sums ||N_l||^2, ||R_l||^2 of which k_l = ||N_l|| / (||R_l|| + eps) is made (Eq. 11)
//   2. norm         D = Pi R; part = sum (k_l (G - D))^2                   (||S||, literal residual)
//   3. finalize     lambda, ||S_prev||, t                                  (Eq. 12)
//   4. update       W -= lr (a_low Pi N + a_res lambda S), S = k_l (G - Pi R)
// By which kernels:
//   k_project, k_back_step          short lists of few tiles and ranks up to 128: 2 to 4 in one kernel whose blocks keep S
//   k_project, k_back_project<norm>, k_finalize, k_back_project<update>        other short lists.  S is not kept: the update is
//                                   D = Pi X with X = a_low N - a_res lambda k_l R, W -= lr (D + a_res lambda k_l G), by the identity
//                                   alpha (P N + lambda (G - P R) diag k) = P (alpha N - alpha lambda R diag k) + alpha lambda G diag k,
//                                   which needs one product instead of two; X is formed while the product loads N and R
//   k_split_projection, k_part_project, k_moments, then k_part_step or k_part_back<norm>, k_finalize, k_form_x, k_part_back<update>
//                                   long lists (part_project.cu, part_back.cu), by the same two ways
//
// The products are the 128 x 128 tile products of split_gemm.cuh: fp32 precision on the tensor cores.  Every
// epilogue takes the finished tile from shared memory, one warp per row, so that all traffic with
// global memory runs along rows.
//
// Short lists are bound by latency, so all of their kernels are chained (launch_chained): one's set-up (tables, barriers,
// tensor memory) runs while the one before it ends.  Step of one 512 x 1376 matrix: 74 us without that and without the
// split projection, 35 us with both, 26.6 us with 2 to 4 in one kernel (k_back_step).
#include <cuda.h>

#include <algorithm>
#include <atomic>

#include "common.cuh"
#include "limit.cuh"
#include "split_gemm.cuh"
#include "step_simt.cuh"

namespace fira {

namespace {

__device__ __forceinline__ int simt_tiles_dev(int extent) { return (extent + SIMT_TILE - 1) / SIMT_TILE; }

// Four entries of a row per lane: the neighbours 4 lane .. 4 lane + 3 where a row's groups of four are
// aligned (VEC), lane, lane + LANES, ... otherwise; either way the access of the LANES lanes that share a row is contiguous.
template <bool VEC, int LANES = 32>
__device__ __forceinline__ int lane_col(int lane, int c) { return VEC ? 4 * lane + c : lane + LANES * c; }

template <bool VEC, int LANES = 32>
__device__ __forceinline__ void load_row(const float* p, int lane, int n, float (&v)[4]) {
  if (VEC) {
    const float4 u = 4 * lane < n ? *reinterpret_cast<const float4*>(p + 4 * lane) : make_float4(0.f, 0.f, 0.f, 0.f);
    v[0] = u.x; v[1] = u.y; v[2] = u.z; v[3] = u.w;
  } else {
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = lane + LANES * c < n ? p[lane + LANES * c] : 0.f;
  }
}
template <bool VEC, int LANES = 32>
__device__ __forceinline__ void load_row(const __nv_bfloat16* p, int lane, int n, float (&v)[4]) {
  if (VEC) {
    const uint2 u = 4 * lane < n ? *reinterpret_cast<const uint2*>(p + 4 * lane) : make_uint2(0u, 0u);
    v[0] = __uint_as_float(u.x << 16); v[1] = __uint_as_float(u.x & 0xffff0000u);
    v[2] = __uint_as_float(u.y << 16); v[3] = __uint_as_float(u.y & 0xffff0000u);
  } else {
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = lane + LANES * c < n ? __bfloat162float(p[lane + LANES * c]) : 0.f;
  }
}
template <bool VEC, int LANES = 32>
__device__ __forceinline__ void store_row(float* p, int lane, int n, const float (&v)[4]) {
  if (VEC) {
    if (4 * lane < n) *reinterpret_cast<float4*>(p + 4 * lane) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
#pragma unroll
    for (int c = 0; c < 4; ++c) if (lane + LANES * c < n) p[lane + LANES * c] = v[c];
  }
}
template <bool VEC, int LANES = 32>
__device__ __forceinline__ void store_row(__nv_bfloat16* p, int lane, int n, const float (&v)[4]) {
  if (VEC) {
    if (4 * lane < n) {
      const __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]), b = __floats2bfloat162_rn(v[2], v[3]);
      uint2 u;
      u.x = *reinterpret_cast<const unsigned*>(&a); u.y = *reinterpret_cast<const unsigned*>(&b);
      *reinterpret_cast<uint2*>(p + 4 * lane) = u;
    }
  } else {
#pragma unroll
    for (int c = 0; c < 4; ++c) if (lane + LANES * c < n) p[lane + LANES * c] = __float2bfloat16_rn(v[c]);
  }
}
// The row's entries as three bf16 parts, `stride` elements apart.
template <bool VEC>
__device__ __forceinline__ void store_row_parts(__nv_bfloat16* p, long long stride, int lane, int n, const float (&v)[4]) {
  uint32_t a[3], b[3];                          // parts of entries 0, 1 and of 2, 3
  split::split3(v[0], v[1], a[0], a[1], a[2]);
  split::split3(v[2], v[3], b[0], b[1], b[2]);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    if (VEC) {
      if (4 * lane < n) *reinterpret_cast<uint2*>(p + i * stride + 4 * lane) = make_uint2(a[i], b[i]);
    } else {
      unsigned short* q = reinterpret_cast<unsigned short*>(p + i * stride) + lane;
      if (lane < n) q[0] = (unsigned short)a[i];
      if (lane + 32 < n) q[32] = (unsigned short)(a[i] >> 16);
      if (lane + 64 < n) q[64] = (unsigned short)b[i];
      if (lane + 96 < n) q[96] = (unsigned short)(b[i] >> 16);
    }
  }
}
template <bool VEC>
__device__ __forceinline__ void load_row_parts(const __nv_bfloat16* p, long long stride, int lane, int n, float (&v)[4]) {
  float h[4], m[4], l[4];
  load_row<VEC>(p, lane, n, h);
  load_row<VEC>(p + stride, lane, n, m);
  load_row<VEC>(p + 2 * stride, lane, n, l);
#pragma unroll
  for (int c = 0; c < 4; ++c) v[c] = h[c] + (m[c] + l[c]);        // exact: the number that was split
}
// n entries per row (a multiple of 4 from an aligned start, or any number), rows `pitch` entries apart
template <typename T>
__device__ __forceinline__ bool rows_vec(const T* base, long long pitch, int n) {
  return pitch % 4 == 0 && n % 4 == 0 && reinterpret_cast<unsigned long long>(base) % (4 * sizeof(T)) == 0;
}

constexpr int ROWS_AT_ONCE = 4;                 // rows of a warp whose loads are in flight together
constexpr int WARP_ROWS = SIMT_TILE / (split::THREADS / 32);

// ---------------------------------------------------------------- phase 1
constexpr int MAX_SPLIT = 8;                    // blocks of a cluster (a portable size)

// Four entries of row `row` of the tile that the blocks of the cluster hold parts of (in the order of their ranks).
template <bool VEC>
__device__ __forceinline__ void add_row_parts(uint32_t row, int blocks, int lane, int n, float (&v)[4]) {
  float u[MAX_SPLIT][4];
#pragma unroll
  for (int b = 0; b < MAX_SPLIT; ++b) {
    const uint32_t p = ptx::map_to_cta(row, min(b, blocks - 1));
    if (VEC) {
      const float4 w = ptx::ld_cluster_f4(p + 16 * lane);
      u[b][0] = w.x; u[b][1] = w.y; u[b][2] = w.z; u[b][3] = w.w;
    } else {
#pragma unroll
      for (int c = 0; c < 4; ++c) u[b][c] = ptx::ld_cluster_f1(p + 4 * (lane + 32 * c));
    }
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    v[c] = u[0][c];
#pragma unroll
    for (int b = 1; b < MAX_SPLIT; ++b) if (b < blocks) v[c] += u[b][c];
    if (lane_col<VEC>(lane, c) >= n) v[c] = 0.f;
  }
}

// Rows of the finished tile R: Adam (Eq. 2-4), N and R to scratch, row sums.  SPLIT: the blocks of the cluster share the
// rows; between cluster_arrive, which the caller has done, and the first look at the tile, M and V are fetched.  Where a
// wait of any of them ran out the tile is garbage, and nothing is stored.
template <int PSI, bool VEC, bool SPLIT>
__device__ __forceinline__ void adam_rows(const MatDev& mt, int l0, int j0, const float* C, const Hyper& hp, const split::Ctl* ctl) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n = min(SIMT_TILE, mt.r - j0);
  const int nrt = simt_tiles_dev(mt.r), q = j0 / SIMT_TILE;
  const int blocks = SPLIT ? (int)ptx::cluster_nctarank() : 1, rows = WARP_ROWS / blocks;
  const int row0 = SPLIT ? ((int)ptx::cluster_ctarank() * (split::THREADS / 32) + warp) * rows : warp * rows;
  constexpr bool momentum = PSI == PSI_ADAM;
  const float bias = ctl->bias;
  int aborted = 0;                              // (one block's flag per lane)
  for (int x = 0; x < rows; x += ROWS_AT_ONCE) {
    float m[ROWS_AT_ONCE][4], v[ROWS_AT_ONCE][4];
#pragma unroll
    for (int y = 0; y < ROWS_AT_ONCE; ++y) {
      const int l = l0 + row0 + x + y;
      const bool there = l < mt.l && (!SPLIT || x + y < rows);
      const long long at = (long long)l * mt.r + j0;
      load_row<VEC>(mt.V + at, lane, there ? n : 0, v[y]);
      load_row<VEC>(mt.M + at, lane, there && momentum ? n : 0, m[y]);
    }
    if (SPLIT && x == 0) {
      ptx::cluster_wait();
      aborted = ptx::ld_cluster_s32(ptx::map_to_cta(ptx::smem_u32(&ctl->abort_flag), min(lane, blocks - 1)));
    }
#pragma unroll
    for (int y = 0; y < ROWS_AT_ONCE; ++y) {
      const int row = row0 + x + y, l = l0 + row;
      if (l >= mt.l || (SPLIT && x + y >= rows)) continue;
      const long long at = (long long)l * mt.r + j0;
      float rv[4], nv[4], nn = 0.f, rn = 0.f;
      if (SPLIT) add_row_parts<VEC>(ptx::smem_u32(C + row * split::C_LD), blocks, lane, n, rv);
      else load_row<VEC>(C + row * split::C_LD, lane, n, rv);
      if (SPLIT && __any_sync(0xffffffffu, aborted)) return;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        nv[c] = adam_direction<PSI>(hp, bias, rv[c], m[y][c], v[y][c]);
        nn = fmaf(nv[c], nv[c], nn);            // (entries past the row's end are zeros throughout)
        rn = fmaf(rv[c], rv[c], rn);
      }
      if (momentum) store_row<VEC>(mt.M + at, lane, n, m[y]);
      store_row<VEC>(mt.V + at, lane, n, v[y]);
      store_row<VEC>(mt.Xt + at, lane, n, nv);
      store_row<VEC>(mt.Rt + at, lane, n, rv);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        nn += __shfl_xor_sync(0xffffffffu, nn, o);
        rn += __shfl_xor_sync(0xffffffffu, rn, o);
      }
      if (lane == 0) {
        if (hp.mode & HYPER_NO_SCALING) mt.kvec[l] = 1.f;
        else if (nrt == 1 && !(hp.mode & HYPER_MATRIX_SCALING)) mt.kvec[l] = sqrtf(nn) / (sqrtf(rn) + hp.eps);
        else { mt.aux[(long long)q * mt.l + l] = nn; mt.aux[(long long)(nrt + q) * mt.l + l] = rn; }
      }
    }
  }
}

// The part of the tile's product that k in [k0, k1) makes.
template <typename T, bool LONG_K, class F>
__device__ __forceinline__ bool project_tile(const MatDev& mt, int l0, int j0, int k0, int k1, unsigned char* smem, split::Ctl* ctl, const F& meanwhile) {
  // A(i = l, k = d): G[d][l] when left, G[l][d] when right.
  split::Operand<T> a(static_cast<const T*>(mt.G) + (mt.left ? k0 * mt.ld : (long long)k0), mt.left ? 1 : mt.ld, mt.left ? mt.ld : 1, mt.l, k1 - k0, l0);
  split::Operand<T> b(static_cast<const T*>(mt.P) + (long long)k0 * mt.r, 1, mt.r, mt.r, k1 - k0, j0);
  return split::tile_product<LONG_K>(a, b, k1 - k0, mt.r - j0, smem, ctl, meanwhile);
}

// SPLIT: the blocks of a cluster share the tile's product by k, each leaves its part in its shared memory, and they add the
// parts while they share the rows of the epilogue.  A list of few tiles leaves most SMs idle otherwise, and its time
// is the latency of one block's slabs, about 2 us each.  LONG_K: a block's part is longer than split::PROMOTE.
// Measured (one 512 x 1376 matrix, r = 128): 46 us as 11 blocks of 16 slabs, 15 us as 11 clusters of 8 blocks.
template <int PSI, bool SPLIT, bool LONG_K>
__global__ void __launch_bounds__(split::THREADS, 2)
k_project(const MatDev* mats, const int* list, int nlist, const int* tile_start, int first, Hyper hp, unsigned* status) {
  // (The tables are not __restrict__: the single-matrix entry point writes them in the kernel that this one is chained to,
  // so no load of them may come before grid_wait, and a compiler that takes them for constants may move it there.)
  extern __shared__ __align__(128) unsigned char smem[];
  split::Ctl* ctl = reinterpret_cast<split::Ctl*>(smem + split::STAGES * split::STAGE_BYTES);
  ptx::grid_wait();
  const int blocks = SPLIT ? (int)ptx::cluster_nctarank() : 1, block = SPLIT ? (int)ptx::cluster_ctarank() : 0;
  const int gt = blockIdx.x / blocks + first;
  const int p = find_matrix(tile_start, nlist, gt);
  const MatDev mt = mats[list[p]];
  const int tile = gt - tile_start[p], rt = simt_tiles_dev(mt.r);
  const int l0 = (tile / rt) * SIMT_TILE, j0 = (tile % rt) * SIMT_TILE;
  split::begin(ctl);
  ptx::grid_launch_next();
  if (mt.shares && tile == 0 && block == 0) {    // (k_back_step waits for them; the one of the step before is done)
    for (int i = threadIdx.x; i < 2 * simt_tiles_dev(mt.m) * simt_tiles_dev(mt.n); i += split::THREADS) mt.shares[i] = 0ull;
    if (threadIdx.x == 0) mt.bias->prev = mt.sc->prev_norm;
  }
  const int slabs = (mt.d + split::BK - 1) / split::BK;
  const int k0 = slabs * block / blocks * split::BK, k1 = min(mt.d, slabs * (block + 1) / blocks * split::BK);
  const float* C = reinterpret_cast<const float*>(smem);
  // The bias factor, by one thread: while its first loads are on their way, or before them (not SPLIT: registers).
  const long long step = mt.sc->t + 1;
  BiasSlot slot;
  slot.step = mt.bias->step; slot.next = mt.bias->next;
  auto put_bias = [&] { if (PSI == PSI_ADAM && threadIdx.x == split::THREADS - 1) ctl->bias = step_bias(slot, step, hp); };
  if (!SPLIT) put_bias();
  auto bias_factor_of_step = [&] { if (SPLIT) put_bias(); };
  bool ok = true;
  if (k1 > k0) {
    ok = mt.bf16 ? project_tile<__nv_bfloat16, LONG_K>(mt, l0, j0, k0, k1, smem, ctl, bias_factor_of_step)
                 : project_tile<float, LONG_K>(mt, l0, j0, k0, k1, smem, ctl, bias_factor_of_step);
  } else {                                      // fewer slabs than blocks
    bias_factor_of_step();
    __syncthreads();
    for (int i = threadIdx.x; i < SIMT_TILE * split::C_LD; i += split::THREADS) reinterpret_cast<float*>(smem)[i] = 0.f;
  }
  if (SPLIT) ptx::cluster_arrive();
  if (SPLIT || ok) {                            // (a block whose wait ran out still meets the others)
    if (mt.r % 4 == 0) adam_rows<PSI, true, SPLIT>(mt, l0, j0, C, hp, ctl);
    else adam_rows<PSI, false, SPLIT>(mt, l0, j0, C, hp, ctl);
  }
  if (SPLIT) ptx::cluster_sync_all();           // nobody leaves while others read its part
  split::end(ctl, status);
}

// ---------------------------------------------------------------- phases 2 and 4
enum { MODE_NORM = 0, MODE_UPDATE = 1 };

// ks[x] <- the factor of the tile's column (left) or row (right) x.  The first phase that asks makes them
// from the row sums and leaves them in the k table for the phases that follow.
template <int MODE>
__device__ __forceinline__ void tile_factors(const MatDev& mt, int i0, int j0, int tile, const Hyper& hp, float* ks) {
  const bool ones = MODE == MODE_NORM && (hp.mode & (HYPER_NO_SCALING | HYPER_MATRIX_SCALING));
  const bool from_sums = MODE == MODE_NORM && !ones && !factors_ready(mt, hp);
  if ((int)threadIdx.x < tile) {
    const int l = (mt.left ? j0 : i0) + threadIdx.x;
    float k = 0.f;
    if (l < mt.l) {
      k = ones ? 1.f : from_sums ? row_factor(mt, l, hp) : mt.kvec[l];
      if (from_sums && (mt.left ? i0 : j0) == 0) mt.kvec[l] = k;
    }
    ks[threadIdx.x] = k;
  }
}

// Rows of the finished tile D.  ks[]: the factors of the tile's columns (left) or rows (right).
template <typename T, int MODE, bool VEC>
__device__ __forceinline__ float back_rows(const MatDev& mt, int i0, int j0, const float* C, const float* ks, float lr, float cres) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n = min(SIMT_TILE, mt.n - j0);
  const T* G = static_cast<const T*>(mt.G);
  T* W = static_cast<T*>(mt.W);
  float kc[4], ss = 0.f;
#pragma unroll
  for (int c = 0; c < 4; ++c) kc[c] = mt.left ? ks[lane_col<VEC>(lane, c)] : 0.f;
  for (int x = 0; x < WARP_ROWS; x += ROWS_AT_ONCE) {
    float g[ROWS_AT_ONCE][4], w[ROWS_AT_ONCE][4];
#pragma unroll
    for (int y = 0; y < ROWS_AT_ONCE; ++y) {
      const int i = i0 + warp * WARP_ROWS + x + y;
      const long long at = (long long)i * mt.ld + j0;
      load_row<VEC>(G + at, lane, i < mt.m ? n : 0, g[y]);
      if (MODE == MODE_UPDATE) load_row<VEC>(W + at, lane, i < mt.m ? n : 0, w[y]);
    }
#pragma unroll
    for (int y = 0; y < ROWS_AT_ONCE; ++y) {
      const int row = warp * WARP_ROWS + x + y, i = i0 + row;
      if (i >= mt.m) continue;
      float dv[4];
      load_row<VEC>(C + row * split::C_LD, lane, n, dv);
      const float kr = mt.left ? 0.f : ks[row];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float kf = mt.left ? kc[c] : kr;
        if (MODE == MODE_NORM) {
          const float sv = kf * (g[y][c] - dv[c]);          // (zero past the row's end)
          ss = fmaf(sv, sv, ss);
        } else {
          w[y][c] = w[y][c] - lr * (dv[c] + cres * kf * g[y][c]);
        }
      }
      if (MODE == MODE_UPDATE) store_row<VEC>(W + (long long)i * mt.ld + j0, lane, n, w[y]);
    }
  }
  return ss;
}

template <typename T, int MODE, bool LONG_K>
__device__ __forceinline__ bool back_product(const MatDev& mt, int i0, int j0, float a_low, float cres,
                                             unsigned char* smem, split::Ctl* ctl) {
  // left: D[d][l] = sum_j Pi[d][j] X[l][j]; right: D[l][d] = sum_j X[l][j] Pi[d][j]
  const int cols = mt.n - j0;
  split::Operand<T> p(static_cast<const T*>(mt.P), mt.r, 1, mt.d, mt.r, mt.left ? i0 : j0);
  p.along_x = false; p.ld = mt.r;               // (r = 1 would count as contiguous along d)
  const int x0 = mt.left ? j0 : i0;
  if (MODE == MODE_NORM) {
    split::Operand<float> x(mt.Rt, mt.r, 1, mt.l, mt.r, x0);
    x.along_x = false; x.ld = mt.r;
    return mt.left ? split::tile_product<LONG_K>(p, x, mt.r, cols, smem, ctl) : split::tile_product<LONG_K>(x, p, mt.r, cols, smem, ctl);
  } else {
    split::CombinedOperand x(mt.Xt, mt.Rt, mt.r, mt.l, mt.r, x0, mt.kvec, a_low, cres);
    return mt.left ? split::tile_product<LONG_K>(p, x, mt.r, cols, smem, ctl) : split::tile_product<LONG_K>(x, p, mt.r, cols, smem, ctl);
  }
}

template <typename T, int MODE, bool LONG_K>
__device__ __forceinline__ float back_tile(const MatDev& mt, int i0, int j0, const Hyper& hp, unsigned char* smem,
                                           split::Ctl* ctl, float* ks) {
  const float cres = MODE == MODE_UPDATE ? hp.a_res * mt.sc->lambda : 0.f;
  tile_factors<MODE>(mt, i0, j0, SIMT_TILE, hp, ks);
  if (!back_product<T, MODE, LONG_K>(mt, i0, j0, hp.a_low, cres, smem, ctl)) return 0.f;
  const float* C = reinterpret_cast<const float*>(smem);
  const bool vec = rows_vec(static_cast<const T*>(mt.G), mt.ld, mt.n) && rows_vec(static_cast<const T*>(mt.W), mt.ld, mt.n);
  return vec ? back_rows<T, MODE, true>(mt, i0, j0, C, ks, hp.lr, cres) : back_rows<T, MODE, false>(mt, i0, j0, C, ks, hp.lr, cres);
}

// LONG_K: some rank of the list is above split::PROMOTE, the main product is added up in registers.  With those, two blocks
// per SM spill (the update 2 KiB per thread); a grid of no more tiles than SMs has one block per SM in any case (BLOCKS = 1).
// Measured with BLOCKS 2 / 1: one 768 x 2048 matrix, r = 300 (96 tiles) 129 / 117 us; 7 of 512 / 1376, r = 200 (240 tiles)
// 127 / 156; 7 of 2048 / 5461, r = 640 1851 / 1976.
template <int MODE, bool LONG_K, int BLOCKS>
__global__ void __launch_bounds__(split::THREADS, BLOCKS)
k_back_project(const MatDev* __restrict__ mats, const int* __restrict__ list, int nlist,
               const int* __restrict__ tile_start, int first, Hyper hp, unsigned* __restrict__ status) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ float ks[SIMT_TILE];
  split::Ctl* ctl = reinterpret_cast<split::Ctl*>(smem + split::STAGES * split::STAGE_BYTES);
  const int gt = blockIdx.x + first;
  const int p = find_matrix(tile_start, nlist, gt);
  const MatDev mt = mats[list[p]];
  const int tile = gt - tile_start[p], ct = simt_tiles_dev(mt.n);
  const int i0 = (tile / ct) * SIMT_TILE, j0 = (tile % ct) * SIMT_TILE;
  split::begin(ctl);
  ptx::grid_wait();
  ptx::grid_launch_next();
  float ss = mt.bf16 ? back_tile<__nv_bfloat16, MODE, LONG_K>(mt, i0, j0, hp, smem, ctl, ks)
                     : back_tile<float, MODE, LONG_K>(mt, i0, j0, hp, smem, ctl, ks);
  if (MODE == MODE_NORM) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if ((threadIdx.x & 31) == 0) ctl->red[threadIdx.x >> 5] = ss;
    __syncthreads();
    if (threadIdx.x == 0) {
      float tot = 0.f;
      for (int w = 0; w < split::THREADS / 32; ++w) tot += ctl->red[w];
      mt.part[tile] = tot;
    }
  }
  split::end(ctl, status);
}

// ---------------------------------------------------------------- phases 2 to 4 in one kernel
// Short lists of no more tiles than SMs (ranks up to 128): a block per tile of W, or per half of one, 64 columns, where the SMs suffice
// for that, keeps its residual S = k (G - Pi R) in registers while it
// makes D = Pi N, waits for the shares of ||S||^2 of its matrix's other tiles, and updates W <- W - lr (a_low D + a_res lambda S).
// G is read once; the blocks wait for one another (a cooperative launch).  One block more per matrix stores its state and works out
// the next step's bias factor.
// Bound by latency, that of fetching instructions included: the code runs once, from start to end.  So all of the projection's and
// of R's slabs are loaded at once and each is multiplied as soon as it is stored, N and G are on their way meanwhile, the
// projection's parts stay for the second product, N's take R's place; and 512 threads have half the code of 256.
// Measured, one 512 x 1376 matrix, r = 128, the kernel's time: 22 us as two ordinary tile products in a row, 18.6 with all slabs loaded at
// once, 15 with all of them stored before the first MMA is issued (of that 5.5 to the first product's end, 2 the second's, the rest rows
// and conversions), 10.9 with half tiles (88 blocks).
// Steps by the three kernels / by this one, us, whole tiles: 1280 x 1280, r = 64 (100 tiles) 38.3 / 35.2; 768 x 2048, r = 128 (96) 40.3 / 35.7;
// 1024 x 2048, r = 128 (128) 41.3 / 37.2; 1152 x 2048, r = 128 (144) 46.0 / 41.3; 2048 x 1000, r = 100 (128, scalar loads of the factors) 47.5 / 47.1.
// Half tiles: 7 matrices 256 / 688, r = 64, 39.2 / 31.2; bf16 600 x 1200, r = 110, 41.3 / 33.3.  The single-matrix entry point, 512 x 1376 and
// 768 x 2304, r = 128: fp32 39.2 / 30.7 and 45.2 / 39.3, bf16 36.0 / 27.0 and 37.1 / 31.9.
constexpr int STEP_THREADS = 512, STEP_ROWS = SIMT_TILE / (STEP_THREADS / 32);         // rows per warp
constexpr int STEP_SLABS = 128 / split::BK;
constexpr int STEP_X = STEP_SLABS * split::OPERAND_BYTES;       // the slabs of R, then N, behind those of the projection; the finished tile overlays them
constexpr int STEP_SMEM = 2 * STEP_X + (int)sizeof(split::Ctl);
static_assert(STEP_SMEM <= 227 * 1024 - 2048 && SIMT_TILE * split::C_LD * 4 <= STEP_X, "shared memory budget");
static_assert(STEP_THREADS == SIMT_TILE * split::BK / 8, "a unit of eight per thread and slab");

// This thread's units, one per slab, of rows [x0, x0 + rows) of Op(x, k) = base[x r + k], zero outside X x r.
template <typename T>
struct StepOperand {
  static constexpr int PARTS = sizeof(T) == 4 ? 3 : 1;
  split::Frag<T> f[STEP_SLABS];

  // REGULAR: whole aligned units only; rows past the matrix read its last one again, for rows of the result that nobody looks
  // at, and slabs past the rank the last one.
  template <bool REGULAR>
  __device__ __forceinline__ void load(const T* base, int r, int X, int x0, int ns) {
    const int x = x0 + threadIdx.x / 4, k = threadIdx.x % 4 * 8;
    const T* row = base + (long long)(REGULAR ? min(x, X - 1) : x) * r + k;
#pragma unroll
    for (int s = 0; s < STEP_SLABS; ++s) {
      if (REGULAR) split::load_frag(row + min(s, ns - 1) * split::BK, f[s]);
      else split::load_frag(row + s * split::BK, x < X ? max(0, r - k - s * split::BK) : 0, false, f[s]);
    }
  }
  __device__ __forceinline__ void store(int s, int rows, unsigned char* place) const {
    if ((int)threadIdx.x / 4 < rows) split::store_parts(place + (threadIdx.x % 4) * split::K_LBO + (threadIdx.x / 4) * 16, f[s]);
  }
};

template <typename T, int COLS, bool VEC, bool REGULAR>
__device__ __forceinline__ void step_tile(const MatDev& mt, int tile, int i0, int j0, const Hyper& hp, unsigned char* smem, split::Ctl* ctl, float* ks, float* coef) {
  __shared__ float red[STEP_THREADS / 32];
  constexpr int LANES = COLS / 4, AT_ONCE = 32 / LANES, PASSES = STEP_ROWS / AT_ONCE;    // lanes to a row, rows of a warp at a time
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, row0 = warp * STEP_ROWS + lane / LANES, hl = lane % LANES;
  const int rows_p = mt.left ? SIMT_TILE : COLS, rows_x = mt.left ? COLS : SIMT_TILE;
  const int n = min(COLS, mt.n - j0), cols = (n + 15) / 16 * 16, ns = (mt.r + split::BK - 1) / split::BK;
  unsigned char* xs = smem + STEP_X;
  float* C = reinterpret_cast<float*>(xs);
  const uint32_t tmem = ctl->tmem_base;
  const T* G = static_cast<const T*>(mt.G);
  T* W = static_cast<T*>(mt.W);
  StepOperand<T> p;
  StepOperand<float> x;
  p.template load<REGULAR>(static_cast<const T*>(mt.P), mt.r, mt.d, mt.left ? i0 : j0, ns);
  x.template load<REGULAR>(mt.Rt, mt.r, mt.l, mt.left ? j0 : i0, ns);
  const float prev = mt.bias->prev;
  // All of the product's slabs at once: a thread that issues MMAs between its slabs' conversions holds up the other warps' next slab.
  auto multiply = [&](bool with_p, uint64_t* done) {
#pragma unroll
    for (int s = 0; s < STEP_SLABS; ++s) {
      if (s >= ns) break;
      if (with_p) p.store(s, rows_p, smem + s * split::OPERAND_BYTES);
      x.store(s, rows_x, xs + s * split::OPERAND_BYTES);
    }
    ptx::fence_proxy_async_smem();
    ptx::tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0) {
      ptx::tc_fence_after();
      uint32_t pa = ptx::smem_u32(smem), xa = ptx::smem_u32(xs);
#pragma unroll 1
      for (int s = 0; s < ns; ++s, pa += split::OPERAND_BYTES, xa += split::OPERAND_BYTES) {
        const int steps = min(split::BK, mt.r - s * split::BK + 15) / 16;
        if (mt.left) split::issue_slab<StepOperand<T>::PARTS, 3, false, false>(tmem, pa, xa, cols, steps, s == 0, s == 0);
        else split::issue_slab<3, StepOperand<T>::PARTS, false, false>(tmem, xa, pa, cols, steps, s == 0, s == 0);
      }
      ptx::umma_commit(ptx::smem_u32(done));
    }
  };
  // The finished tile into shared memory, in the place of the X slabs.
  auto read_back = [&](uint64_t* done) {
    const bool ok = ptx::mbar_wait(ptx::smem_u32(done), 0, &ctl->abort_flag);
    if (__syncthreads_or(!ok)) return false;
    ptx::tc_fence_after();
    const int c0 = (warp >> 2) * (COLS / 4);
    if (c0 < cols) {
      const uint32_t from = tmem + ((uint32_t)((warp & 3) * 32) << 16) + c0;
      float* to = C + (32 * (warp & 3) + lane) * split::C_LD + c0;
#pragma unroll 1
      for (int q = 0; q < COLS / 4; q += 16) {
        uint32_t v[16], w[16];
        __syncwarp();
        ptx::tmem_ld_32x32b_x16(from + q, v);
        ptx::tmem_ld_32x32b_x16(from + split::TILE + q, w);
        ptx::tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 16; e += 4)
          *reinterpret_cast<float4*>(to + q + e) = make_float4(__uint_as_float(v[e]) + __uint_as_float(w[e]), __uint_as_float(v[e + 1]) + __uint_as_float(w[e + 1]),
                                                               __uint_as_float(v[e + 2]) + __uint_as_float(w[e + 2]), __uint_as_float(v[e + 3]) + __uint_as_float(w[e + 3]));
      }
    }
    ptx::tc_fence_before();
    __syncthreads();
    return true;
  };
  multiply(true, &ctl->done[0]);
  float s[PASSES][4];                            // G, then the residual
#pragma unroll
  for (int y = 0; y < PASSES; ++y) load_row<VEC, LANES>(G + (long long)(i0 + row0 + AT_ONCE * y) * mt.ld + j0, hl, i0 + row0 + AT_ONCE * y < mt.m ? n : 0, s[y]);
  x.template load<REGULAR>(mt.Xt, mt.r, mt.l, mt.left ? j0 : i0, ns);          // N
  tile_factors<MODE_NORM>(mt, i0, j0, SIMT_TILE, hp, ks);
  if (!read_back(&ctl->done[0])) return;
  float kc[4], ss = 0.f;
#pragma unroll
  for (int c = 0; c < 4; ++c) kc[c] = mt.left ? ks[lane_col<VEC, LANES>(hl, c)] : 0.f;
#pragma unroll
  for (int y = 0; y < PASSES; ++y) {
    const int row = row0 + AT_ONCE * y;
    float dv[4];
    load_row<VEC, LANES>(C + row * split::C_LD, hl, n, dv);
    const float kr = mt.left ? 0.f : ks[row];
    const bool there = i0 + row < mt.m;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      s[y][c] = there ? (mt.left ? kc[c] : kr) * (s[y][c] - dv[c]) : 0.f;       // (zero past the row's end)
      ss = fmaf(s[y][c], s[y][c], ss);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  if (lane == 0) red[warp] = ss;
  __syncthreads();                               // (also: nobody reads the first product any more)
  if (warp == 1) {
    float tot = lane < STEP_THREADS / 32 ? red[lane] : 0.f;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
    if (lane == 0) ptx::put_marked(mt.shares + tile, tot);
  }
  multiply(false, &ctl->done[1]);
  float w[PASSES][4];
#pragma unroll
  for (int y = 0; y < PASSES; ++y) load_row<VEC, LANES>(W + (long long)(i0 + row0 + AT_ONCE * y) * mt.ld + j0, hl, i0 + row0 + AT_ONCE * y < mt.m ? n : 0, w[y]);
  if (warp == STEP_THREADS / 32 - 1) {           // (while the product is made)
    Limit lim;
    const bool known = wait_limit<float>(mt.shares, SIMT_TILE / COLS * simt_tiles_dev(mt.m) * simt_tiles_dev(mt.n), mt, prev, hp, &ctl->abort_flag, lim);
    if (lane == 0 && known) *coef = hp.a_res * lim.lambda * lim.kmat;
  }
  if (!read_back(&ctl->done[1]) || *(volatile int*)&ctl->abort_flag) return;
  const float cres = *coef;
#pragma unroll
  for (int y = 0; y < PASSES; ++y) {
    const int row = row0 + AT_ONCE * y;
    if (i0 + row >= mt.m) continue;
    float dv[4];
    load_row<VEC, LANES>(C + row * split::C_LD, hl, n, dv);
#pragma unroll
    for (int c = 0; c < 4; ++c) w[y][c] = w[y][c] - hp.lr * (hp.a_low * dv[c] + cres * s[y][c]);
    store_row<VEC, LANES>(W + (long long)(i0 + row) * mt.ld + j0, hl, n, w[y]);
  }
}
template <typename T, int COLS>
__device__ __forceinline__ void step_tile(const MatDev& mt, int tile, int i0, int j0, const Hyper& hp, unsigned char* smem, split::Ctl* ctl, float* ks, float* coef) {
  if (j0 >= mt.n) {                              // the second half of a tile that has none
    if (threadIdx.x == 0) ptx::put_marked(mt.shares + tile, 0.f);
    return;
  }
  const bool vec = rows_vec(static_cast<const T*>(mt.G), mt.ld, mt.n) && rows_vec(static_cast<const T*>(mt.W), mt.ld, mt.n);
  const bool regular = mt.r % split::BK == 0 && reinterpret_cast<unsigned long long>(mt.P) % 16 == 0;       // (R and N are aligned)
  if (vec && regular) step_tile<T, COLS, true, true>(mt, tile, i0, j0, hp, smem, ctl, ks, coef);
  else if (regular) step_tile<T, COLS, false, true>(mt, tile, i0, j0, hp, smem, ctl, ks, coef);
  else step_tile<T, COLS, false, false>(mt, tile, i0, j0, hp, smem, ctl, ks, coef);
}
// norm_out, t_out: where the caller keeps the remembered norm and the step count (may be null).
// tiles: blocks that have a tile (COLS = 128) or half of one (64).
template <int COLS>
__global__ void __launch_bounds__(STEP_THREADS, 1)
k_back_step(const MatDev* mats, const int* list, int nlist, const int* tile_start, int first, int tiles, int first_matrix, Hyper hp, float* norm_out,
            long long* t_out, unsigned* status) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ float ks[SIMT_TILE], coef;
  __shared__ int waited;
  split::Ctl* ctl = reinterpret_cast<split::Ctl*>(smem + 2 * STEP_X);
  if ((int)blockIdx.x >= tiles) {                // a matrix's state
    const int lane = threadIdx.x & 31;
    if (threadIdx.x == 0) waited = 0;
    __syncthreads();
    ptx::grid_wait();
    ptx::grid_launch_next();
    const MatDev& mt = mats[list[first_matrix + blockIdx.x - tiles]];
    const long long next = mt.sc->t + 2;
    __syncthreads();                             // (t is read before it is stored)
    if (threadIdx.x == 32 && !(hp.mode & (HYPER_PSI_RMSPROP | HYPER_PSI_ADAGRAD))) {
      mt.bias->next = bias_factor_call(hp.beta1, hp.beta2, next);
      mt.bias->step = next;
    }
    if (threadIdx.x < 32) {
      Limit lim;
      if (wait_limit<float>(mt.shares, SIMT_TILE / COLS * simt_tiles_dev(mt.m) * simt_tiles_dev(mt.n), mt, mt.bias->prev, hp, &waited, lim)) store_limit(mt, hp, lim, status);
      else if (lane == 0) atomicOr(status, DEV_STATUS_TIMEOUT);
      if (lane == 0 && norm_out) { *norm_out = mt.sc->prev_norm; *t_out = mt.sc->t; }
    }
    return;
  }
  split::begin(ctl);
  ptx::grid_wait();
  ptx::grid_launch_next();
  constexpr int PER = SIMT_TILE / COLS;
  const int gt = blockIdx.x / PER + first, half = blockIdx.x % PER;
  const int q = find_matrix(tile_start, nlist, gt);
  const MatDev mt = mats[list[q]];
  const int tile = gt - tile_start[q], ct = simt_tiles_dev(mt.n);
  const int i0 = (tile / ct) * SIMT_TILE, j0 = (tile % ct) * SIMT_TILE + half * COLS;
  if (mt.bf16) step_tile<__nv_bfloat16, COLS>(mt, PER * tile + half, i0, j0, hp, smem, ctl, ks, &coef);
  else step_tile<float, COLS>(mt, PER * tile + half, i0, j0, hp, smem, ctl, ks, &coef);
  split::end(ctl, status);
}

// ---------------------------------------------------------------- long lists
// Adam (Eq. 2-4) on rows of R that the projection left as parts, the rows' factors k_l, and X for limiter factor 1 (or N: see
// HYPER_X_IS_N) as parts: one warp per row, R whole in registers (CHUNKS of 128 columns), ROWS rows with their loads in flight together.
template <int PSI, bool VEC, int CHUNKS, int ROWS>
__device__ __forceinline__ void moment_rows(const MatDev& mt, int l0, int count, const Hyper& hp, float bias) {
  const int lane = threadIdx.x & 31;
  const long long stride = (long long)mt.l * mt.rp_pitch;
  float m[ROWS][CHUNKS][4], v[ROWS][CHUNKS][4], rv[ROWS][CHUNKS][4];
#pragma unroll
  for (int y = 0; y < ROWS; ++y)
#pragma unroll
    for (int c = 0; c < CHUNKS; ++c) {
      const int l = l0 + y, j = 128 * c, n = y < count ? min(128, mt.r - j) : 0;
      load_row<VEC>(mt.V + (long long)l * mt.r + j, lane, n, v[y][c]);
      load_row<VEC>(mt.M + (long long)l * mt.r + j, lane, PSI == PSI_ADAM ? n : 0, m[y][c]);
      load_row_parts<VEC>(mt.Rp + (long long)l * mt.rp_pitch + j, stride, lane, n, rv[y][c]);
    }
#pragma unroll
  for (int y = 0; y < ROWS; ++y) {
    if (y >= count) break;
    const int l = l0 + y;
    float nv[CHUNKS][4], nn = 0.f, rn = 0.f;
#pragma unroll
    for (int c = 0; c < CHUNKS; ++c) {
      const int j = 128 * c, n = min(128, mt.r - j);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        nv[c][q] = adam_direction<PSI>(hp, bias, rv[y][c][q], m[y][c][q], v[y][c][q]);
        nn = fmaf(nv[c][q], nv[c][q], nn);      // (entries past the row's end are zeros throughout)
        rn = fmaf(rv[y][c][q], rv[y][c][q], rn);
      }
      if (PSI == PSI_ADAM) store_row<VEC>(mt.M + (long long)l * mt.r + j, lane, n, m[y][c]);
      store_row<VEC>(mt.V + (long long)l * mt.r + j, lane, n, v[y][c]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      nn += __shfl_xor_sync(0xffffffffu, nn, o);
      rn += __shfl_xor_sync(0xffffffffu, rn, o);
    }
    const float k = hp.mode & HYPER_NO_SCALING ? 1.f : sqrtf(nn) / (sqrtf(rn) + hp.eps);
    if (lane == 0) {
      if (hp.mode & HYPER_MATRIX_SCALING) { mt.aux[l] = nn; mt.aux[mt.l + l] = rn; }
      else mt.kvec[l] = k;
    }
    if (part_forms_x(hp)) {
      const float ck = hp.a_res * k;
#pragma unroll
      for (int c = 0; c < CHUNKS; ++c) {
        float x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) x[q] = hp.a_low * nv[c][q] - ck * rv[y][c][q];
        store_row_parts<VEC>(mt.Xp + (long long)l * mt.rp_pitch + 128 * c, stride, lane, min(128, mt.r - 128 * c), x);
      }
    }
  }
}
// Row passes: so many rows per warp that the grid is resident at once (rows_per_warp): what it costs a warp to find its
// matrix, five dependent loads and more, is paid once.
// Bound by memory: 28 bytes per entry.  As an epilogue of the projection the same work held up its product (part_project.cu).
// CHUNKS: for ranks up to 128 CHUNKS.  (One kernel for all ranks has the registers of the
// largest: 56 matrices 512 / 1376, r = 128, took 45 us instead of 35.)
template <int PSI, int CHUNKS>
__global__ void __launch_bounds__(256, CHUNKS == 1 ? 4 : CHUNKS == 2 ? 3 : 2)
k_moments(const MatDev* __restrict__ mats, const int* __restrict__ list, int nlist, const int* __restrict__ row_start, int first_row,
          int rows_end, int per_warp, Hyper hp) {
  int row = first_row + (blockIdx.x * 8 + (threadIdx.x >> 5)) * per_warp;
  int p = row < rows_end ? find_matrix(row_start, nlist, row) : 0;
  ptx::grid_wait();
  ptx::grid_launch_next();
  const int end = min(row + per_warp, rows_end);
  while (row < end) {
    const MatDev& mt = mats[list[p]];
    const int l0 = row - row_start[p], l1 = min(l0 + end - row, mt.l);
    const float bias = mt.bias->now;
    constexpr int ROWS = CHUNKS == 1 ? 2 : 1;
    if (mt.r % 4 == 0) {
      for (int l = l0; l < l1; l += ROWS) moment_rows<PSI, true, CHUNKS, ROWS>(mt, l, min(ROWS, l1 - l), hp, bias);
    } else {
      for (int l = l0; l < l1; l += ROWS) moment_rows<PSI, false, CHUNKS, ROWS>(mt, l, min(ROWS, l1 - l), hp, bias);
    }
    row += l1 - l0;
    ++p;
  }
}

// X = a_low N - a_res lambda k_l R as parts, one warp per row l; N from the updated moments, by the arithmetic that
// k_moments used.  (r % 4 != 0: scalar accesses.)  Two rows with their loads in flight together.
template <int PSI, bool VEC>
__device__ __forceinline__ void form_x_rows(const MatDev& mt, int l0, int count, const Hyper& hp, float bias, float c) {
  constexpr int ROWS = 2;
  const int lane = threadIdx.x & 31;
  const long long stride = (long long)mt.l * mt.rp_pitch;
  float ck[ROWS];
#pragma unroll
  for (int y = 0; y < ROWS; ++y) ck[y] = y < count ? c * mt.kvec[l0 + y] : 0.f;
  for (int j = 0; j < mt.r; j += 128) {
    float m[ROWS][4], v[ROWS][4], rv[ROWS][4];
#pragma unroll
    for (int y = 0; y < ROWS; ++y) {
      const int n = y < count ? min(128, mt.r - j) : 0;
      load_row<VEC>(mt.M + (long long)(l0 + y) * mt.r + j, lane, PSI == PSI_ADAM ? n : 0, m[y]);
      load_row<VEC>(mt.V + (long long)(l0 + y) * mt.r + j, lane, n, v[y]);
      load_row_parts<VEC>(mt.Rp + (long long)(l0 + y) * mt.rp_pitch + j, stride, lane, n, rv[y]);
    }
#pragma unroll
    for (int y = 0; y < ROWS; ++y) {
      float x[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) x[q] = hp.a_low * direction<PSI>(hp, bias, rv[y][q], m[y][q], v[y][q]) - ck[y] * rv[y][q];
      store_row_parts<VEC>(mt.Xp + (long long)(l0 + y) * mt.rp_pitch + j, stride, lane, y < count ? min(128, mt.r - j) : 0, x);
    }
  }
}
constexpr int FORM_X_BLOCKS = 3;                // resident per SM
template <int PSI>
__global__ void __launch_bounds__(256, FORM_X_BLOCKS)
k_form_x(const MatDev* __restrict__ mats, const int* __restrict__ list, int nlist, const int* __restrict__ row_start, int first_row,
         int rows_end, int per_warp, Hyper hp) {
  int row = first_row + (blockIdx.x * 8 + (threadIdx.x >> 5)) * per_warp;
  ptx::grid_wait();
  ptx::grid_launch_next();
  if (row >= rows_end) return;
  int p = find_matrix(row_start, nlist, row);
  const int end = min(row + per_warp, rows_end);
  while (row < end) {
    const MatDev& mt = mats[list[p]];
    const int l0 = row - row_start[p], l1 = min(l0 + end - row, mt.l);
    const float lambda = mt.sc->lambda, c = hp.a_res * lambda, bias = mt.bias->now;
    if (part_forms_x(hp) && lambda == 1.f) {
      // k_moments has formed it
    } else if (mt.r % 4 == 0) {
      for (int l = l0; l < l1; l += 2) form_x_rows<PSI, true>(mt, l, min(2, l1 - l), hp, bias, c);
    } else {
      for (int l = l0; l < l1; l += 2) form_x_rows<PSI, false>(mt, l, min(2, l1 - l), hp, bias, c);
    }
    row += l1 - l0;
    ++p;
  }
}

// The projection's parts, eight neighbours per thread and pass, `per` blocks per matrix, and by one more the step's scalars.  In
// every step: projection and step count are in the caller's state buffer, whose bytes may have changed since the last one.
// (56 matrices 512 / 1376, r = 128: 37 MB, 5.5 of the step's 242 us; k_part_project's set-up, which is chained to it, runs
// meanwhile.)
template <typename T>
__device__ __forceinline__ void split_units(const MatDev& mt, int block, int blocks) {
  const unsigned per_row = mt.pp_pitch / 8, units = mt.d * per_row, step = 256 * blocks;        // (r <= PART_STEP_MAX_RANK)
  const long long stride = 2ll * mt.d * mt.pp_pitch;
  const bool vec = mt.r % 8 == 0;
  for (unsigned u = 256 * block + threadIdx.x; u < units; u += step) {
    const unsigned i = u / per_row, j = u % per_row * 8;
    split::Frag<T> f;
    split::load_frag(static_cast<const T*>(mt.P) + (long long)i * mt.r + j, mt.r - (int)j, vec, f);
    split::store_parts(reinterpret_cast<unsigned char*>(mt.Pp + (long long)i * mt.pp_pitch + j), f, stride);
  }
}
__global__ void __launch_bounds__(256)
k_split_projection(const MatDev* __restrict__ mats, const int* __restrict__ list, int per, Hyper hp) {
  ptx::grid_launch_next();
  const MatDev& mt = mats[list[blockIdx.x / (per + 1)]];
  const int block = blockIdx.x % (per + 1);
  if (block == per) {                           // the scalars
    if (threadIdx.x == 0) {
      mt.bias->prev = mt.sc->prev_norm;
      mt.bias->now = step_bias(*mt.bias, mt.sc->t + 1, hp);
    }
    for (int i = threadIdx.x; i < PART_SHARE_WORDS * part_step_tiles(mt.m, mt.n); i += 256) reinterpret_cast<unsigned long long*>(mt.part)[i] = 0ull;
    return;
  }
  if (mt.bf16) split_units<__nv_bfloat16>(mt, block, per);
  else split_units<float>(mt, block, per);
}

// ---------------------------------------------------------------- Fira-only-scaling
// W <- W - lr phi(R) G: no product.  One block per tile x tile elements of W, a warp per row.
template <typename T, int UPDATE, bool VEC>
__device__ __forceinline__ float scaled_gradient_rows(const MatDev& mt, int i0, int j0, int tile, const float* ks, float c) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const T* G = static_cast<const T*>(mt.G);
  T* W = static_cast<T*>(mt.W);
  float ss = 0.f;
  for (int jc = 0; jc < tile && j0 + jc < mt.n; jc += 128) {
    const int n = min(128, mt.n - j0 - jc);
    float kc[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) kc[q] = mt.left ? ks[jc + lane_col<VEC>(lane, q)] : 0.f;
    for (int x = warp * ROWS_AT_ONCE; x < tile; x += 8 * ROWS_AT_ONCE) {
      float g[ROWS_AT_ONCE][4], w[ROWS_AT_ONCE][4];
#pragma unroll
      for (int y = 0; y < ROWS_AT_ONCE; ++y) {
        const int i = i0 + x + y;
        const long long at = (long long)i * mt.ld + j0 + jc;
        load_row<VEC>(G + at, lane, i < mt.m ? n : 0, g[y]);
        if (UPDATE) load_row<VEC>(W + at, lane, i < mt.m ? n : 0, w[y]);
      }
#pragma unroll
      for (int y = 0; y < ROWS_AT_ONCE; ++y) {
        const int i = i0 + x + y;
        if (i >= mt.m) continue;
        const float kr = mt.left ? 0.f : ks[x + y];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float kf = mt.left ? kc[q] : kr;
          if (UPDATE) w[y][q] = w[y][q] - c * kf * g[y][q];
          else { const float sv = kf * g[y][q]; ss = fmaf(sv, sv, ss); }
        }
        if (UPDATE) store_row<VEC>(W + (long long)i * mt.ld + j0 + jc, lane, n, w[y]);
      }
    }
  }
  return ss;
}

template <typename T, int UPDATE>
__device__ __forceinline__ float scaled_gradient_tile(const MatDev& mt, int i0, int j0, int tile, const float* ks, float c) {
  const bool vec = rows_vec(static_cast<const T*>(mt.G), mt.ld, mt.n) && rows_vec(static_cast<const T*>(mt.W), mt.ld, mt.n);
  return vec ? scaled_gradient_rows<T, UPDATE, true>(mt, i0, j0, tile, ks, c)
             : scaled_gradient_rows<T, UPDATE, false>(mt, i0, j0, tile, ks, c);
}

template <int UPDATE>
__global__ void __launch_bounds__(256)
k_scaled_gradient(const MatDev* __restrict__ mats, const int* __restrict__ list, int nlist,
                  const int* __restrict__ tile_start, int first, int tile, Hyper hp) {
  __shared__ float ks[256];
  __shared__ float red[8];
  const int gt = blockIdx.x + first;
  const int p = find_matrix(tile_start, nlist, gt);
  const MatDev mt = mats[list[p]];
  const int t = gt - tile_start[p];
  const int ct = (mt.n + tile - 1) / tile;
  const int i0 = (t / ct) * tile, j0 = (t % ct) * tile;
  tile_factors<UPDATE ? MODE_UPDATE : MODE_NORM>(mt, i0, j0, tile, hp, ks);
  __syncthreads();
  const float c = UPDATE ? hp.lr * hp.a_res * mt.sc->lambda : 0.f;
  float ss = mt.bf16 ? scaled_gradient_tile<__nv_bfloat16, UPDATE>(mt, i0, j0, tile, ks, c)
                     : scaled_gradient_tile<float, UPDATE>(mt, i0, j0, tile, ks, c);
  if (!UPDATE) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
    __syncthreads();
    if (threadIdx.x == 0) {
      float tot = 0.f;
      for (int w = 0; w < 8; ++w) tot += red[w];
      mt.part[t] = tot;
    }
  }
}

}  // namespace

void launch_scaled_gradient(const MatDev* mats, const int* list, int nlist, const int* tile_start, int first,
                            int tiles, int tile, int update, const Hyper& hp, cudaStream_t st) {
  if (tiles <= 0) return;
  if (update) k_scaled_gradient<1><<<tiles, 256, 0, st>>>(mats, list, nlist, tile_start, first, tile, hp);
  else k_scaled_gradient<0><<<tiles, 256, 0, st>>>(mats, list, nlist, tile_start, first, tile, hp);
}

// ---------------------------------------------------------------- phase 3
__global__ void __launch_bounds__(256)
k_finalize(const MatDev* __restrict__ mats, const int* __restrict__ list, int nlist,
           const int* __restrict__ npart_of, Hyper hp, unsigned* __restrict__ status) {
  __shared__ double sred[256];
  __shared__ float smin[256], smax[256];
  const MatDev mt = mats[list[blockIdx.x]];
  const int npart = npart_of[blockIdx.x];
  if (threadIdx.x == 255 && mt.bias && !(hp.mode & (HYPER_PSI_RMSPROP | HYPER_PSI_ADAGRAD))) {    // the next step's bias factor
    const long long next = mt.sc->t + 2;
    mt.bias->next = bias_factor(hp.beta1, hp.beta2, next);
    mt.bias->step = next;
  }
  ptx::grid_wait();
  ptx::grid_launch_next();
  double acc = 0.0;
  for (int i = threadIdx.x; i < npart; i += 256) acc += (double)mt.part[i];
  // Matrix-level factor (Eq. 9): the phases before ran with k = 1, so `part` holds ||G - P R||^2;
  // the factor scales the norm here and fills the k table for the phases after.
  float kmat = 1.f;
  if (hp.mode & HYPER_MATRIX_SCALING) {
    __shared__ double sn[256], sr[256];
    double an = 0.0, ar = 0.0;
    const long long sums = (long long)mt.aux_slots * mt.l;
    for (long long i = threadIdx.x; i < sums; i += 256) { an += (double)mt.aux[i]; ar += (double)mt.aux[sums + i]; }
    sn[threadIdx.x] = an; sr[threadIdx.x] = ar;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
      if (threadIdx.x < o) { sn[threadIdx.x] += sn[threadIdx.x + o]; sr[threadIdx.x] += sr[threadIdx.x + o]; }
      __syncthreads();
    }
    kmat = (float)(sqrt(sn[0]) / (sqrt(sr[0]) + (double)hp.eps));
    for (int i = threadIdx.x; i < mt.l; i += 256) mt.kvec[i] = kmat;
  }
  float kmin = INFINITY, kmax = -INFINITY;
  for (int i = threadIdx.x; i < mt.l; i += 256) {
    const float kv = (hp.mode & HYPER_MATRIX_SCALING) ? kmat : mt.kvec[i];
    kmin = fminf(kmin, kv);
    kmax = fmaxf(kmax, kv);
  }
  sred[threadIdx.x] = acc; smin[threadIdx.x] = kmin; smax[threadIdx.x] = kmax;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      sred[threadIdx.x] += sred[threadIdx.x + o];
      smin[threadIdx.x] = fminf(smin[threadIdx.x], smin[threadIdx.x + o]);
      smax[threadIdx.x] = fmaxf(smax[threadIdx.x], smax[threadIdx.x + o]);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double tot = sred[0] > 0.0 ? sred[0] : 0.0;
    const float norm = kmat * (float)sqrt(tot);
    const float prev = mt.sc->prev_norm;
    float lam = 1.f;
    if (hp.mode & HYPER_NO_RESIDUAL) {           // Eq. 6: no residual, nothing to limit or remember
      mt.sc->norm_scaled = 0.f;
      mt.sc->lambda = 1.f;
      mt.sc->k_min = 0.f;
      mt.sc->k_max = 0.f;
      mt.sc->t = mt.sc->t + 1;
      return;
    }
    if (prev >= 0.f && !isinf(hp.gamma)) {
      const float ratio = norm / (prev + hp.eps);
      lam = hp.gamma / fmaxf(ratio, hp.gamma);
    }
    if (!isfinite((float)sred[0]) || !isfinite(smax[0])) atomicOr(status, DEV_STATUS_NONFINITE);
    mt.sc->norm_scaled = norm;
    mt.sc->lambda = lam;
    mt.sc->prev_norm = lam * norm;
    mt.sc->k_min = smin[0];
    mt.sc->k_max = smax[0];
    mt.sc->t = mt.sc->t + 1;
  }
}

std::vector<const char*> simt_phase_names(const SimtPlan& pl, bool only_scaling) {
  if (pl.resident && !only_scaling) return {"k_project", "k_back_step"};
  if (pl.parts.one_kernel_pairs && !only_scaling) return {"k_project", "k_moments", "k_part_step"};
  return {"k_project", "k_moments", "k_back_project<norm>", "k_finalize", "k_form_x", "k_back_project<update>"};
}

// Measured (fp32 / bf16 storage, times of a step in us, short against long): 6 matrices 512 x 1376, r = 128, 63 / 51 against 71 / 62,
// 8 of them 102 / 72 against 82 / 69; 4 of 1024 x 1024, r = 256, 92 / 65 against 94 / 71, 6 of them 151 / 98 against 113 / 82; 24 of
// 300 x 417, r = 64, whose rows are copied to an aligned pitch first, 78 / 77 against 114 / 110.
constexpr long long LONG_LIST_ELEMENTS = 5 << 20;
bool simt_long_list(const std::vector<fira_matrix_desc>& list) {
  long long elements = 0;
  for (const fira_matrix_desc& d : list) {
    if (d.r > PART_STEP_MAX_RANK) return false;
    elements += (long long)d.m * d.n;
  }
  return elements >= LONG_LIST_ELEMENTS;
}

int stream_sms(cudaStream_t st) {
  struct Driver {
    CUresult (*current)(CUcontext*) = nullptr;
    CUresult (*of_context)(CUcontext, CUdevResource*, CUdevResourceType) = nullptr;
    CUresult (*green)(CUstream, CUgreenCtx*) = nullptr;
    CUresult (*of_green)(CUgreenCtx, CUdevResource*, CUdevResourceType) = nullptr;
  };
  static const Driver drv = [] {                 // (an older driver has none of them, and no such parts)
    Driver d;
    auto get = [](const char* name, void** f) {
      cudaDriverEntryPointQueryResult q;
      if (cudaGetDriverEntryPoint(name, f, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess) *f = nullptr;
    };
    get("cuCtxGetCurrent", (void**)&d.current);
    get("cuCtxGetDevResource", (void**)&d.of_context);
    get("cuStreamGetGreenCtx", (void**)&d.green);
    get("cuGreenCtxGetDevResource", (void**)&d.of_green);
    return d;
  }();
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  CUdevResource part;
  CUcontext ctx = nullptr;
  CUgreenCtx green = nullptr;
  if (drv.current && drv.of_context && drv.current(&ctx) == CUDA_SUCCESS && ctx && drv.of_context(ctx, &part, CU_DEV_RESOURCE_TYPE_SM) == CUDA_SUCCESS)
    sms = std::min(sms, (int)part.sm.smCount);
  if (drv.green && drv.of_green && drv.green((CUstream)st, &green) == CUDA_SUCCESS && green && drv.of_green(green, &part, CU_DEV_RESOURCE_TYPE_SM) == CUDA_SUCCESS)
    sms = std::min(sms, (int)part.sm.smCount);
  return sms;
}

static void split_projections(const SimtPlan& pl, int qa, int qb, const Hyper& hp, cudaStream_t st) {
  const int per = (int)std::min<long long>(64, (pl.max_proj_units + 255) / 256);
  k_split_projection<<<(unsigned)((qb - qa) * (per + 1)), 256, 0, st>>>(pl.mats, pl.list + qa, per, hp);
}

// The products' shared memory is above the default limit: a per-device, per-kernel setting.
static bool allow_smem() {
  static std::atomic<bool> done[64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess && (dev < 0 || dev >= 64)) e = cudaErrorInvalidDevice;
  if (e == cudaSuccess && !done[dev].load()) {
    const void* kernels[15] = {(const void*)k_project<PSI_ADAM, false, true>, (const void*)k_project<PSI_RMSPROP, false, true>,
                               (const void*)k_project<PSI_ADAGRAD, false, true>, (const void*)k_project<PSI_ADAM, true, true>,
                               (const void*)k_project<PSI_RMSPROP, true, true>, (const void*)k_project<PSI_ADAGRAD, true, true>,
                               (const void*)k_project<PSI_ADAM, true, false>, (const void*)k_project<PSI_RMSPROP, true, false>,
                               (const void*)k_project<PSI_ADAGRAD, true, false>,
                               (const void*)k_back_project<MODE_NORM, false, 2>, (const void*)k_back_project<MODE_UPDATE, false, 2>,
                               (const void*)k_back_project<MODE_NORM, true, 2>, (const void*)k_back_project<MODE_UPDATE, true, 2>,
                               (const void*)k_back_project<MODE_NORM, true, 1>, (const void*)k_back_project<MODE_UPDATE, true, 1>};
    for (const void* k : kernels)
      if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, split::SMEM_BYTES);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_back_step<SIMT_TILE>, cudaFuncAttributeMaxDynamicSharedMemorySize, STEP_SMEM);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_back_step<SIMT_TILE / 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, STEP_SMEM);
    if (e == cudaSuccess) done[dev].store(true);
  }
  if (e != cudaSuccess) set_error(std::string("step kernels, shared memory: ") + cudaGetErrorString(e));
  return e == cudaSuccess;
}

constexpr int SMS = 148;
template <int MODE>
static auto back_kernel(const SimtPlan& pl, int tiles) {
  return pl.max_r <= split::PROMOTE ? k_back_project<MODE, false, 2> : tiles <= SMS ? k_back_project<MODE, true, 1> : k_back_project<MODE, true, 2>;
}

// Blocks that share a tile of the projection: of a short list as many as keep the grid within one block per SM (but no
// part below two slabs).  Counted over the whole list, whatever range of it is stepped: the sums have the same order then.
static int split_of(const SimtPlan& pl) {
  int split = 1;
  while (split < MAX_SPLIT && 2 * split * pl.proj_tiles <= SMS && 4 * split * split::BK <= pl.max_d) split *= 2;
  return split;
}

template <int PSI>
static cudaError_t launch_project(const SimtPlan& pl, int first, int tiles, const Hyper& hp, unsigned* status_dev, cudaStream_t st) {
  const int split = split_of(pl);
  const bool long_k = (pl.max_d + split::BK - 1) / split::BK > split * (split::PROMOTE / split::BK);
  auto k = split == 1 ? k_project<PSI, false, true> : long_k ? k_project<PSI, true, true> : k_project<PSI, true, false>;
  return launch_chained(k, tiles * split, split::THREADS, split::SMEM_BYTES, st, pl.chained, split, pl.mats, pl.list, pl.nlist, pl.proj_tile_start, first, hp, status_dev);
}

static int rows_per_warp(int rows, int blocks_per_sm) {
  const int warps = SMS * blocks_per_sm * 8;
  return std::max(2, (rows + warps - 1) / warps);
}
template <int PSI>
static cudaError_t launch_moments(const SimtPlan& pl, int r0, int r1, const Hyper& hp, cudaStream_t st) {
  auto k = pl.max_r <= 128 ? k_moments<PSI, 1> : pl.max_r <= 256 ? k_moments<PSI, 2> : k_moments<PSI, PART_STEP_MAX_RANK / 128>;
  const int per = rows_per_warp(r1 - r0, pl.max_r <= 128 ? 4 : pl.max_r <= 256 ? 3 : 2);
  return launch_chained(k, (r1 - r0 + 8 * per - 1) / (8 * per), 256, 0, st, true, 1, pl.mats, pl.list, pl.nlist, pl.row_start, r0, r1, per, hp);
}

int launch_simt_step(const SimtPlan& pl, const Hyper& hp, unsigned* status_dev, cudaStream_t st,
                     PhaseTimer* tm, int qa, int qb) {
  if (pl.nlist == 0) return 0;
  if (!allow_smem()) return -1;
  // the sub-range [qa, qb) of the list: first tile and their counts from the host copies of the
  // prefix arrays; the kernels still search the whole arrays with absolute indices
  int pt0 = 0, pt1 = pl.proj_tiles, wt0 = 0, wt1 = pl.w_tiles, nq = pl.nlist;
  if (qb >= 0) {
    if (qa >= qb) return 0;
    pt0 = pl.h_proj_tile_start[qa]; pt1 = pl.h_proj_tile_start[qb];
    wt0 = pl.h_w_tile_start[qa]; wt1 = pl.h_w_tile_start[qb];
    nq = qb - qa;
  } else {
    qa = 0;
  }
  constexpr int TH = split::THREADS, SM = split::SMEM_BYTES;
  cudaError_t error = cudaSuccess;
  auto launch_error = [&](cudaError_t e) { if (error == cudaSuccess) error = e; };
  const bool only_scaling = hp.mode & HYPER_ONLY_SCALING;     // W <- W - lr phi(R) G: no back-projection
  const bool parts = pl.parts.table && !only_scaling;          // (a long list's only-scaling step has no back-projection)
  const bool one_kernel = parts && pl.parts.one_kernel_pairs;  // norm, limiter and update
  const int psi = psi_of(hp);
  const int qe = qb >= 0 ? qb : pl.nlist;
  const int s0 = pl.parts.table ? pl.h_stage_start[pl.h_stage_pos[qa]] : 0;
  const int staged = pl.parts.table ? pl.h_stage_start[pl.h_stage_pos[qe]] - s0 : 0, nstage = pl.parts.table ? pl.h_stage_pos.back() : 0;
  tm->mark(st);
  launch_stage(pl.mats, pl.stage_list, nstage, pl.stage_start, s0, staged, 0, st);
  if (pl.parts.table) {                // (also before only-scaling, which needs the factors)
    split_projections(pl, qa, qe, hp, st);
    if (part_project_run(pl.parts, pl.mats, qa, qe, status_dev, st) != FIRA_OK) return -1;
    tm->mark(st);
    const int r0 = pl.h_row_start[qa], r1 = pl.h_row_start[qe];
    Hyper hm = hp;
    if (one_kernel) { hm.mode |= HYPER_X_IS_N; hm.a_low = 1.f; hm.a_res = 0.f; }
    launch_error((psi == PSI_ADAM ? launch_moments<PSI_ADAM> : psi == PSI_RMSPROP ? launch_moments<PSI_RMSPROP> : launch_moments<PSI_ADAGRAD>)(pl, r0, r1, hm, st));
  } else {
    launch_error((psi == PSI_ADAM ? launch_project<PSI_ADAM> : psi == PSI_RMSPROP ? launch_project<PSI_RMSPROP> : launch_project<PSI_ADAGRAD>)(
        pl, pt0, pt1 - pt0, hp, status_dev, st));
    tm->mark(st);
  }
  if (pl.resident && !only_scaling) {
    const int per = short_one_kernel(2 * pl.w_tiles, pl.nlist, pl.max_r, pl.resident) ? 2 : 1, blocks = per * (wt1 - wt0);       // (of the whole list, whatever range is stepped)
    launch_error(launch_resident(per == 2 ? k_back_step<SIMT_TILE / 2> : k_back_step<SIMT_TILE>, blocks + nq, STEP_THREADS, STEP_SMEM, st, true, 1, pl.mats, pl.list,
                                 pl.nlist, pl.w_tile_start, wt0, blocks, qa, hp, pl.norm_out, pl.t_out, status_dev));
    tm->mark(st);
    if (error != cudaSuccess) { set_error(std::string("step kernels: ") + cudaGetErrorString(error)); return -1; }
    return 2;
  }
  tm->mark(st);
  if (one_kernel) {
    if (part_step_run_one_kernel(pl.parts, pl.mats, qa, qe, hp, status_dev, st) != FIRA_OK) return -1;
    launch_stage(pl.mats, pl.stage_list, nstage, pl.stage_start, s0, staged, 1, st);
    tm->mark(st);
    if (error != cudaSuccess) { set_error(std::string("step kernels: ") + cudaGetErrorString(error)); return -1; }
    return 4 + (staged ? 2 : 0);
  }
  if (only_scaling)
    launch_scaled_gradient(pl.mats, pl.list, pl.nlist, pl.w_tile_start, wt0, wt1 - wt0, SIMT_TILE, 0, hp, st);
  else if (parts) {
    if (part_step_run(pl.parts, pl.mats, qa, qe, 0, hp, status_dev, st) != FIRA_OK) return -1;
  } else
    launch_error(launch_chained(back_kernel<MODE_NORM>(pl, wt1 - wt0), wt1 - wt0, TH, SM, st, true, 1, pl.mats, pl.list, pl.nlist, pl.w_tile_start, wt0, hp, status_dev));
  tm->mark(st);
  // (only-scaling leaves one partial sum per 128 x 128 tile whatever the list)
  launch_error(launch_chained(k_finalize, nq, 256, 0, st, true, 1, pl.mats, pl.list + qa, nq, (only_scaling ? pl.npart_tiles : pl.npart) + qa, hp, status_dev));
  tm->mark(st);
  if (parts) {
    const int r0 = pl.h_row_start[qa], r1 = pl.h_row_start[qe];
    const int per = rows_per_warp(r1 - r0, FORM_X_BLOCKS);
    launch_error(launch_chained(psi == PSI_ADAM ? k_form_x<PSI_ADAM> : psi == PSI_RMSPROP ? k_form_x<PSI_RMSPROP> : k_form_x<PSI_ADAGRAD>,
                                (r1 - r0 + 8 * per - 1) / (8 * per), 256, 0, st, true, 1, pl.mats, pl.list, pl.nlist, pl.row_start, r0, r1, per, hp));
  }
  tm->mark(st);
  if (only_scaling)
    launch_scaled_gradient(pl.mats, pl.list, pl.nlist, pl.w_tile_start, wt0, wt1 - wt0, SIMT_TILE, 1, hp, st);
  else if (parts) {
    if (part_step_run(pl.parts, pl.mats, qa, qe, 1, hp, status_dev, st) != FIRA_OK) return -1;
    launch_stage(pl.mats, pl.stage_list, nstage, pl.stage_start, s0, staged, 1, st);
  } else
    launch_error(launch_chained(back_kernel<MODE_UPDATE>(pl, wt1 - wt0), wt1 - wt0, TH, SM, st, true, 1, pl.mats, pl.list, pl.nlist, pl.w_tile_start, wt0, hp, status_dev));
  tm->mark(st);
  if (error != cudaSuccess) { set_error(std::string("step kernels: ") + cudaGetErrorString(error)); return -1; }
  return 4 + (pl.parts.table ? 2 : 0) + (parts ? 1 : 0) + (staged ? (parts ? 2 : 1) : 0);
}

}  // namespace fira
