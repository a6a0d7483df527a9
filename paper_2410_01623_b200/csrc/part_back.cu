// The step's two products with the projection in fp32 precision, for long lists (part_gemm.cuh: PartStepPlan):
//   MODE_NORM    D = Pi R (or R Pi^T); partial sums of ||S||^2 = sum (k (G - D))^2
//   MODE_UPDATE  D = Pi X (or X Pi^T); W <- W - lr (D + a_res lambda k G)
//
// CTA pairs, one CTA per SM, persistent; 256 x 128 tiles of W; the operands are parts, both contiguous along the rank
// index, and come as TMA slabs (part_slab.cuh).  G and W move through shared memory by TMA in both directions, in boxes of
// 128 rows x 64 bytes (64-byte swizzle: a thread per row reads without bank conflicts), W updated in place; two groups of
// four epilogue warps take alternate boxes.  (Warps that took their patch of the tile through shared memory and read G
// and W along rows with ordinary loads needed 10 us per tile where this needs 4: four times the instructions, and two
// load latencies per tile that nothing covered.)
//
// Tensor memory: main and small products (split_gemm.cuh) of a tile take 2 x 128 columns, two such sets alternate.  That is
// for lists of ranks up to PROMOTE.  With a longer one among them (DEEP) the main product alternates between two accumulators
// every PROMOTE of k and the small products between two others from tile to tile, as in part_project.cu; all pieces but the
// last are added to fp32 sums in registers.  (256 of k in one accumulator and 512 in two saved the sums, but MMAs add by
// truncation: D was biased towards zero by 2.8e-7 at r = 256, positive operands, where pieces of 128 leave 1.2e-7.  Norm and
// update of 14 matrices 1024 / 2736, r = 256: 77 and 90 us then, 89 and 95 now; with the sums
// kept in tensor memory 100 and 112.)
//
// What bounds it: G (and W in and out) at the copy bandwidth.
//
// Warp roles: 0 operand producer, 1 MMA issuer (even CTA) and owner of the tensor memory, 2 box loader, 3-10 epilogue,
// 11-12 W box storers.
#include <string.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "part_slab.cuh"
#include "split_gemm.cuh"
#include "step_simt.cuh"

namespace fira {

namespace {

enum { MODE_NORM = 0, MODE_UPDATE = 1 };

constexpr int SLAB_BYTES = 3 * (A_PART + B_PART);
constexpr int GROUPS = 2;
constexpr int BOX_BYTES = PM / 2 * 64;          // 8 KiB: 128 rows of 16 fp32 or 32 bf16
constexpr int GROUP_THREADS = 128;
constexpr int THREADS = 32 * 3 + GROUPS * GROUP_THREADS + 32 * GROUPS;
constexpr int KS = PN / GROUPS;                 // factors that a group needs per tile (its boxes' columns)
constexpr int PROMOTE_SLABS = split::PROMOTE / PK;
constexpr int stages_of(int mode) { return mode == MODE_NORM ? 4 : 3; }
constexpr int bufs_of(int mode) { return mode == MODE_NORM ? 4 : 3; }            // box buffers per group
constexpr int buf_bytes(int mode) { return (mode == MODE_NORM ? 1 : 2) * BOX_BYTES; }

struct alignas(64) BackJob {
  CUtensorMap a, b, g, w;
  int mat;                                      // index into the problem table
  int shape;                                    // see issue_parts
};
static_assert(sizeof(BackJob) % 64 == 0, "tensor maps must stay 64-byte aligned");
struct TileDev { int job, i0, j0, nk; };

struct BackCtl {
  uint64_t full[4], empty[4];
  uint64_t tmem_full[2], tmem_empty[2];         // a set, or (DEEP) a main accumulator
  uint64_t small_empty[2];                      // (DEEP) the small products of a tile have been read
  uint64_t efull[GROUPS][4], eready[GROUPS][4], eempty[GROUPS][4];
  uint64_t esync[GROUPS];
  uint32_t tmem_base;
  int abort_flag;
  float ks[GROUPS][2][KS];
};
constexpr size_t smem_bytes(int mode) {
  return (size_t)stages_of(mode) * SLAB_BYTES + (size_t)GROUPS * bufs_of(mode) * buf_bytes(mode) + sizeof(BackCtl);
}
static_assert(smem_bytes(MODE_NORM) <= 227 * 1024 && smem_bytes(MODE_UPDATE) <= 227 * 1024, "shared memory budget");

__device__ __forceinline__ TileDev load_tile(const TileDev* t) {
  const int4 v = __ldg(reinterpret_cast<const int4*>(t));
  return TileDev{v.x, v.y, v.z, v.w};
}

// The factor k_l; the norm of a matrix with one factor is scaled in the end.
template <int MODE>
__device__ __forceinline__ float step_factor(const MatDev& mt, int l, const Hyper& hp) {
  return MODE == MODE_NORM && (hp.mode & HYPER_MATRIX_SCALING) ? 1.f : mt.kvec[l];
}

__device__ __forceinline__ void unpack(const uint4& u, float (&v)[4]) {
  v[0] = __uint_as_float(u.x); v[1] = __uint_as_float(u.y); v[2] = __uint_as_float(u.z); v[3] = __uint_as_float(u.w);
}
__device__ __forceinline__ void unpack(const uint4& u, float (&v)[8]) {
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) { v[2 * i] = __uint_as_float(w[i] << 16); v[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u); }
}
__device__ __forceinline__ uint4 pack(const float (&v)[4]) {
  return make_uint4(__float_as_uint(v[0]), __float_as_uint(v[1]), __float_as_uint(v[2]), __float_as_uint(v[3]));
}
__device__ __forceinline__ uint4 pack(const float (&v)[8]) {
  uint32_t w[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
    w[i] = *reinterpret_cast<const uint32_t*>(&p);
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

template <int MODE, bool DEEP>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS, 1)
k_part_back(const BackJob* __restrict__ jobs, const TileDev* __restrict__ tiles, int count, const MatDev* __restrict__ mats, Hyper hp,
            unsigned* __restrict__ status) {
  constexpr int STAGES = stages_of(MODE), BUFS = bufs_of(MODE), BUF_BYTES = buf_bytes(MODE);
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char* boxes = smem + STAGES * SLAB_BYTES;
  BackCtl* ctl = reinterpret_cast<BackCtl*>(boxes + GROUPS * BUFS * BUF_BYTES);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = ptx::cluster_ctarank();
  const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  const bool smem_ok = (ptx::smem_u32(smem) & 1023u) == 0;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      ptx::mbar_init(ptx::smem_u32(&ctl->full[s]), 1);
      ptx::mbar_init(ptx::smem_u32(&ctl->empty[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      ptx::mbar_init(ptx::smem_u32(&ctl->tmem_full[b]), 1);
      ptx::mbar_init(ptx::smem_u32(&ctl->tmem_empty[b]), 2 * GROUPS * 4);        // every epilogue warp of the pair
      ptx::mbar_init(ptx::smem_u32(&ctl->small_empty[b]), 2 * GROUPS * 4);
    }
    for (int g = 0; g < GROUPS; ++g) {
      for (int b = 0; b < BUFS; ++b) {
        ptx::mbar_init(ptx::smem_u32(&ctl->efull[g][b]), 1);
        ptx::mbar_init(ptx::smem_u32(&ctl->eready[g][b]), GROUP_THREADS);
        ptx::mbar_init(ptx::smem_u32(&ctl->eempty[g][b]), 1);
      }
      ptx::mbar_init(ptx::smem_u32(&ctl->esync[g]), GROUP_THREADS);
    }
    ctl->abort_flag = smem_ok ? 0 : 1;
    ptx::fence_barrier_init();
  }
  if (warp == 1) {
    ptx::tmem_alloc_pair(ptx::smem_u32(&ctl->tmem_base), 512);
    ptx::tmem_relinquish_pair();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::cluster_sync_all();
  ptx::tc_fence_after();
  ptx::grid_wait();
  ptx::grid_launch_next();
  volatile int* abort_flag = &ctl->abort_flag;
  const uint32_t slabs = ptx::smem_u32(smem), boxes_u32 = ptx::smem_u32(boxes);

  if (warp == 0) {
    if (lane == 0 && smem_ok) {
      int stage = 0; uint32_t phase = 0; bool ok = true;
      for (int t = pair; t < count && ok; t += npairs) {
        const TileDev d = load_tile(tiles + t);
        const BackJob* jb = jobs + d.job;
        const int shape = jb->shape, pa = shape & 3, pb = (shape >> 2) & 3;
        const int i0 = d.i0 + PM / 2 * (int)rank, j0 = d.j0 + PN / 2 * (int)rank;
        for (int k = 0; k < d.nk; ++k) {
          if (!ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->empty[stage]), phase ^ 1u, abort_flag)) { ok = false; break; }
          const uint32_t fb = ptx::map_to_cta(ptx::smem_u32(&ctl->full[stage]), 0);
          const uint32_t sa = slabs + stage * SLAB_BYTES;
          if (rank == 0) ptx::mbar_expect_tx(ptx::smem_u32(&ctl->full[stage]), 2 * (pa * A_PART + pb * B_PART));
          ptx::tma_load_3d_pair(sa, &jb->a, fb, k * PK, i0, 0);
          ptx::tma_load_3d_pair(sa + 3 * A_PART, &jb->b, fb, k * PK, j0, 0);
          if (++stage == STAGES) { stage = 0; phase ^= 1u; }
        }
      }
      if (!ok && rank == 0) {   // give copies in flight a bounded time to land
        for (int s = 0; s < STAGES; ++s)
          for (uint32_t it = 0; it < (1u << 16); ++it)
            if (ptx::mbar_try_wait_cluster(ptx::smem_u32(&ctl->full[s]), (s < stage) ? phase : (phase ^ 1u))) break;
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && smem_ok && rank == 0) {
      int stage = 0; uint32_t phase = 0; bool ok = true;
      uint32_t set = 0, sphase = 0;                     // of a tile, or (DEEP) main accumulator of a piece
      uint32_t tile = 0;
      for (int t = pair; t < count && ok; t += npairs, ++tile) {
        const TileDev d = load_tile(tiles + t);
        const int shape = jobs[d.job].shape;
        if (DEEP && !ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->small_empty[tile & 1]), ((tile >> 1) & 1) ^ 1u, abort_flag)) break;
        if (!DEEP && !ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->tmem_empty[set]), sphase ^ 1u, abort_flag)) break;
        for (int k = 0; k < d.nk; ++k) {
          const bool first = DEEP ? k % PROMOTE_SLABS == 0 : k == 0;
          if (DEEP && first && !ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->tmem_empty[set]), sphase ^ 1u, abort_flag)) { ok = false; break; }
          if (!ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->full[stage]), phase, abort_flag)) { ok = false; break; }
          ptx::tc_fence_after();
          // main, small | main, small; DEEP: main, main | small, small
          const uint32_t main = ctl->tmem_base + set * (DEEP ? 1 : 2) * PN, small = DEEP ? ctl->tmem_base + (2 + (tile & 1)) * PN : main + PN;
          issue_parts(shape, main, small, slabs + stage * SLAB_BYTES, 3 * A_PART, first, k == 0);
          ptx::umma_commit_pair(ptx::smem_u32(&ctl->empty[stage]), 3);
          if (++stage == STAGES) { stage = 0; phase ^= 1u; }
          if (DEEP && ((k + 1) % PROMOTE_SLABS == 0 || k + 1 == d.nk)) {
            ptx::umma_commit_pair(ptx::smem_u32(&ctl->tmem_full[set]), 3);
            if (++set == 2) { set = 0; sphase ^= 1u; }
          }
        }
        if (!ok) break;
        if (!DEEP) {
          ptx::umma_commit_pair(ptx::smem_u32(&ctl->tmem_full[set]), 3);
          if (++set == 2) { set = 0; sphase ^= 1u; }
        }
      }
    }
  } else if (warp == 2) {
    // ------------------------------------------------------------ box loader
    if (lane == 0 && smem_ok) {
      int eb[GROUPS] = {0, 0}; uint32_t ephase[GROUPS] = {0, 0}; bool ok = true;
      for (int t = pair; t < count && ok; t += npairs) {
        const TileDev d = load_tile(tiles + t);
        const BackJob* jb = jobs + d.job;
        const MatDev* mt = mats + jb->mat;
        const int i0 = d.i0 + PM / 2 * (int)rank, cols = mt->bf16 ? 32 : 16, n = mt->n;
        for (int c = 0; c < PN / cols; ++c) {
          const int j = d.j0 + cols * c, g = c & 1;
          if (j >= n) break;
          if (!ptx::mbar_wait(ptx::smem_u32(&ctl->eempty[g][eb[g]]), ephase[g] ^ 1u, abort_flag)) { ok = false; break; }
          const uint32_t fb = ptx::smem_u32(&ctl->efull[g][eb[g]]);
          const uint32_t dst = boxes_u32 + (g * BUFS + eb[g]) * BUF_BYTES;
          ptx::mbar_expect_tx(fb, BUF_BYTES);
          ptx::tma_load_2d(dst, &jb->g, fb, j, i0);
          if (MODE == MODE_UPDATE) ptx::tma_load_2d(dst + BOX_BYTES, &jb->w, fb, j, i0);
          if (++eb[g] == BUFS) { eb[g] = 0; ephase[g] ^= 1u; }
        }
      }
    }
  } else if (warp >= 3 + 4 * GROUPS) {
    // ------------------------------------------------------------ box storer of one group (MODE_NORM: hands the buffers back)
    if (lane == 0 && smem_ok) {
      const int g = warp - (3 + 4 * GROUPS);
      int eb = 0; uint32_t rphase = 0; bool ok = true;
      for (int t = pair; t < count && ok; t += npairs) {
        const TileDev d = load_tile(tiles + t);
        const BackJob* jb = jobs + d.job;
        const MatDev* mt = mats + jb->mat;
        const int i0 = d.i0 + PM / 2 * (int)rank, cols = mt->bf16 ? 32 : 16, n = mt->n, m = mt->m;
        for (int c = g; c < PN / cols && d.j0 + cols * c < n; c += GROUPS) {
          if (!ptx::mbar_wait(ptx::smem_u32(&ctl->eready[g][eb]), rphase, abort_flag)) { ok = false; break; }
          if (MODE == MODE_UPDATE && i0 < m) {
            ptx::tma_store_2d(&jb->w, boxes_u32 + (g * BUFS + eb) * BUF_BYTES + BOX_BYTES, d.j0 + cols * c, i0);
            ptx::bulk_commit_group();
            ptx::bulk_wait_group_read<0>();              // the box has been read: the buffer is free
          }
          ptx::mbar_arrive(ptx::smem_u32(&ctl->eempty[g][eb]));
          if (++eb == BUFS) { eb = 0; rphase ^= 1u; }
        }
      }
      ptx::bulk_wait_group_all();
    }
  } else if (smem_ok) {
    // ------------------------------------------------------------ epilogue
    const int ew = warp - 3, g = ew >> 2;
    const int quarter = warp & 3;                       // TMEM lanes 32 * quarter .. + 31
    const int row = quarter * 32 + lane, tid_g = (ew & 3) * 32 + lane;
    const uint32_t rowoff = (uint32_t)row * 64, sw = (uint32_t)(row >> 1) & 3u;    // 64-byte swizzle: slot ^= (row / 2) % 4
    const uint32_t esync = ptx::smem_u32(&ctl->esync[g]);
    const uint32_t te[2] = {ptx::map_to_cta(ptx::smem_u32(&ctl->tmem_empty[0]), 0), ptx::map_to_cta(ptx::smem_u32(&ctl->tmem_empty[1]), 0)};
    const uint32_t se[2] = {ptx::map_to_cta(ptx::smem_u32(&ctl->small_empty[0]), 0), ptx::map_to_cta(ptx::smem_u32(&ctl->small_empty[1]), 0)};
    const uint32_t tmem = ctl->tmem_base + ((uint32_t)(quarter * 32) << 16);
    uint32_t yphase = 0, set = 0, sphase = 0, ephase = 0, tile = 0;
    int eb = 0, parity = 0;
    bool ok = true;
    for (int t = pair; t < count && ok; t += npairs) {
      const TileDev d = load_tile(tiles + t);
      const MatDev& mt = mats[jobs[d.job].mat];
      const int left = mt.left, n = mt.n, m = mt.m, cols = mt.bf16 ? 32 : 16;
      const int i0 = d.i0 + PM / 2 * (int)rank;
      const float cres = MODE == MODE_UPDATE ? hp.a_res * mt.sc->lambda : 0.f;
      float* ks = ctl->ks[g][parity];
      float krow = 0.f;
      if (left) {
        if (tid_g < KS) {                                // column x of the group's boxes, one box after the other
          const int j = d.j0 + (GROUPS * (tid_g / cols) + g) * cols + tid_g % cols;
          ks[tid_g] = j < n ? step_factor<MODE>(mt, j, hp) : 0.f;
        }
      } else if (i0 + row < m) {
        krow = step_factor<MODE>(mt, i0 + row, hp);
      }
      ptx::mbar_arrive(esync);                           // the group's factors are in place
      if (!ptx::mbar_wait(esync, yphase, abort_flag)) break;
      yphase ^= 1u;
      float dv[DEEP ? PN / GROUPS : 32];                 // D: DEEP: in the columns of all of the group's boxes; else of one
      if (DEEP) {
#pragma unroll
        for (int e = 0; e < PN / GROUPS; ++e) dv[DEEP ? e : 0] = 0.f;
        for (int k = PROMOTE_SLABS; k < d.nk; k += PROMOTE_SLABS) {       // all pieces but the last
          if (!ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->tmem_full[set]), sphase, abort_flag)) { ok = false; break; }
          ptx::tc_fence_after();
#pragma unroll
          for (int e = 0; e < PN / GROUPS; e += 16) {
            uint32_t v[16];
            __syncwarp();
            ptx::tmem_ld_32x32b_x16(tmem + set * PN + (cols == 32 ? 32 * (GROUPS * (e / 32) + g) + e % 32 : GROUPS * e + 16 * g), v);
            ptx::tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 16; ++i) dv[DEEP ? e + i : 0] += __uint_as_float(v[i]);
          }
          ptx::tc_fence_before();
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive_cluster(te[set]);
          if (++set == 2) { set = 0; sphase ^= 1u; }
        }
      }
      if (!ok || !ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->tmem_full[set]), sphase, abort_flag)) break;
      ptx::tc_fence_after();
      const uint32_t tbase = tmem + set * (DEEP ? 1 : 2) * PN, tsmall = DEEP ? tmem + (2 + (tile & 1)) * PN : tbase + PN;
      const int nch = min(PN / cols, (n - d.j0 + cols - 1) / cols);
      float ss = 0.f;
      auto accumulators_read = [&] {                     // this warp has read all it needs of them
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          ptx::mbar_arrive_cluster(te[set]);
          if (DEEP) ptx::mbar_arrive_cluster(se[tile & 1]);
        }
      };
      if (g >= nch) accumulators_read();                 // this group has no box in this tile
      // 16 columns of the accumulators
      auto product = [&](int col, float* out) {
        uint32_t v[16], w[16];
        __syncwarp();
        ptx::tmem_ld_32x32b_x16(tbase + col, v);
        ptx::tmem_ld_32x32b_x16(tsmall + col, w);
        ptx::tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 16; ++e) out[e] = (DEEP ? out[e] + __uint_as_float(v[e]) : __uint_as_float(v[e])) + __uint_as_float(w[e]);
      };
      // PER values of one 16-byte word of the row: per group of 16 product columns 16 / PER words
      auto word = [&](unsigned char* gb, int q, const float* dv, const float* kf, auto zero) {
        constexpr int PER = sizeof(zero) / sizeof(float);
        const uint32_t off = rowoff + (((uint32_t)q ^ sw) << 4);
        float gv[PER], wv[PER];
        unpack(*reinterpret_cast<const uint4*>(gb + off), gv);
        if (MODE == MODE_NORM) {
#pragma unroll
          for (int e = 0; e < PER; ++e) {
            const float sv = (left ? kf[e] : krow) * (gv[e] - dv[e]);      // (G is zero past the matrix, D as well: its operands are)
            ss = fmaf(sv, sv, ss);
          }
        } else {
          unpack(*reinterpret_cast<const uint4*>(gb + BOX_BYTES + off), wv);
#pragma unroll
          for (int e = 0; e < PER; ++e) wv[e] = wv[e] - hp.lr * (dv[e] + cres * (left ? kf[e] : krow) * gv[e]);
          *reinterpret_cast<uint4*>(gb + BOX_BYTES + off) = pack(wv);
        }
      };
      struct F4 { float v[4]; };
      struct F8 { float v[8]; };
      // kind: F4 or F8 where the type of the matrix is known, int where it is not
      auto box = [&](int c, float* dbox, auto kind) {
        const bool wide = std::is_same<decltype(kind), int>::value ? cols == 32 : std::is_same<decltype(kind), F8>::value;
        unsigned char* gb = boxes + (g * BUFS + eb) * BUF_BYTES;
        const float* kf = ks + (c / GROUPS) * cols;
        product(c * cols, dbox);
        if (wide) product(c * cols + 16, dbox + 16);
        if (c + GROUPS >= nch) accumulators_read();
        if (!ptx::mbar_wait(ptx::smem_u32(&ctl->efull[g][eb]), ephase, abort_flag)) { ok = false; return; }
        if (wide) {
#pragma unroll
          for (int q = 0; q < 4; ++q) word(gb, q, dbox + 8 * q, kf + 8 * q, F8());
        } else {
#pragma unroll
          for (int q = 0; q < 4; ++q) word(gb, q, dbox + 4 * q, kf + 4 * q, F4());
        }
        if (MODE == MODE_UPDATE) ptx::fence_proxy_async_smem();
        ptx::mbar_arrive(ptx::smem_u32(&ctl->eready[g][eb]));
        if (++eb == BUFS) { eb = 0; ephase ^= 1u; }
      };
      if (!DEEP) {
        for (int c = g; c < nch && ok; c += GROUPS) box(c, dv, 0);
      } else if (cols == 32) {
#pragma unroll
        for (int b = 0; b < 2; ++b)
          if (ok && GROUPS * b + g < nch) box(GROUPS * b + g, dv + (DEEP ? 32 * b : 0), F8());
      } else {
#pragma unroll
        for (int b = 0; b < 4; ++b)
          if (ok && GROUPS * b + g < nch) box(GROUPS * b + g, dv + (DEEP ? 16 * b : 0), F4());
      }
      if (!ok) break;
      if (MODE == MODE_NORM) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
        const int in_matrix = (d.i0 / PM) * ((n + PN - 1) / PN) + d.j0 / PN;
        if (lane == 0) mt.part[in_matrix * PART_SUMS_PER_TILE + (int)rank * 8 + ew] = ss;
      }
      parity ^= 1;
      if (++set == 2) { set = 0; sphase ^= 1u; }
      ++tile;
    }
  }
  // neither CTA may leave while its partner can still reach into its shared memory
  ptx::tc_fence_before();
  __syncthreads();
  ptx::cluster_sync_all();
  if (warp == 1) {
    __syncwarp();
    ptx::tc_fence_after();
    ptx::tmem_dealloc_pair(ctl->tmem_base, 512);
  }
  if (threadIdx.x == 0 && ctl->abort_flag) atomicOr(status, DEV_STATUS_TIMEOUT);
}

auto kernel_of(int mode, int deep) {
  return mode == MODE_NORM ? (deep ? k_part_back<MODE_NORM, true> : k_part_back<MODE_NORM, false>)
                           : (deep ? k_part_back<MODE_UPDATE, true> : k_part_back<MODE_UPDATE, false>);
}

// SMs of the current device (0: error) once the kernels may use their shared memory there.
int prepared_sms() {
  static std::atomic<int> sms_of_device[64];    // (the shared-memory limit is a per-device setting)
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess && (dev < 0 || dev >= 64)) e = cudaErrorInvalidDevice;
  if (e == cudaSuccess && (sms = sms_of_device[dev].load()) == 0) {
    for (int deep = 0; deep < 2; ++deep)
      for (int mode : {MODE_NORM, MODE_UPDATE})
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel_of(mode, deep), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes(mode));
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) sms_of_device[dev].store(sms);
  }
  if (e != cudaSuccess) { set_error(std::string("step products: ") + cudaGetErrorString(e)); return 0; }
  return sms;
}

// Box of 128 rows x 64 bytes over G or W (or their aligned copies).
bool encode_box(CUtensorMap* map, const void* base, const MatDev& mt) {
  const int es = mt.bf16 ? 2 : 4;
  const unsigned long long extent[2] = {(unsigned long long)mt.n, (unsigned long long)mt.m};
  const unsigned long long stride[1] = {(unsigned long long)(mt.Gs ? mt.lds : mt.ld) * es};
  const unsigned box[2] = {64u / es, PM / 2};
  return encode_tiled(map, base, !mt.bf16, 2, extent, stride, box, 64);
}

}  // namespace

size_t part_step_table_bytes(int njobs, int ntiles) {
  return align_up(2 * sizeof(BackJob) * (size_t)njobs) + align_up(sizeof(TileDev) * (size_t)ntiles);
}

fira_status part_step_prepare(const std::vector<MatDev>& mats, const std::vector<int>& list, char* table_dev, PartStepPlan* plan, cudaStream_t st) {
  std::vector<TileDev> td;
  plan->jobs.assign(2 * list.size() * sizeof(BackJob), 0);
  plan->tile_start.assign(1, 0);
  plan->deep = 0;
  BackJob* jd = reinterpret_cast<BackJob*>(plan->jobs.data());
  for (size_t q = 0; q < list.size(); ++q) {
    const MatDev& mt = mats[list[q]];
    for (int update = 0; update < 2; ++update) {
      PartMatrix pi, x;
      pi.base = mt.Pp; pi.rows = mt.d; pi.cols = mt.r; pi.pitch = mt.pp_pitch; pi.part_stride = (long long)mt.d * mt.pp_pitch; pi.parts = mt.bf16 ? 1 : 3;
      x.base = update ? mt.Xp : mt.Rp; x.rows = mt.l; x.cols = mt.r; x.pitch = mt.rp_pitch; x.part_stride = (long long)mt.l * mt.rp_pitch; x.parts = 3;
      const PartMatrix &a = mt.left ? pi : x, &b = mt.left ? x : pi;       // D[d][l] = Pi X^T, D[l][d] = X Pi^T
      BackJob j;
      memset(&j, 0, sizeof(j));
      if (!encode_operand(&j.a, a, false, PM / 2) || !encode_operand(&j.b, b, false, PN / 2)) return FIRA_ERR_CUDA;
      j.mat = list[q];
      j.shape = a.parts | (b.parts << 2) | 32;
      memcpy(&jd[update * list.size() + q], &j, sizeof(j));
    }
    for (int i0 = 0; i0 < mt.m; i0 += PM)
      for (int j0 = 0; j0 < mt.n; j0 += PN) td.push_back(TileDev{(int)q, i0, j0, (mt.r + PK - 1) / PK});
    plan->tile_start.push_back((int)td.size());
    if (mt.r > split::PROMOTE) plan->deep = 1;
  }
  plan->table = table_dev; plan->njobs = (int)list.size();
  cudaError_t e = cudaMemcpyAsync(table_dev + align_up(plan->jobs.size()), td.data(), sizeof(TileDev) * td.size(), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) { set_error(std::string("step products, tables: ") + cudaGetErrorString(e)); return FIRA_ERR_CUDA; }
  return FIRA_OK;
}

fira_status part_step_update_pointers(const std::vector<MatDev>& mats, const std::vector<int>& list, PartStepPlan* plan, cudaStream_t st) {
  BackJob* jd = reinterpret_cast<BackJob*>(plan->jobs.data());
  for (size_t q = 0; q < list.size(); ++q) {
    const MatDev& mt = mats[list[q]];
    CUtensorMap g, w;
    if (!encode_box(&g, mt.Gs ? mt.Gs : mt.G, mt) || !encode_box(&w, mt.Gs ? mt.Ws : mt.W, mt)) return FIRA_ERR_CUDA;
    for (size_t at : {q, list.size() + q}) {
      memcpy(&jd[at].g, &g, sizeof(g));
      memcpy(&jd[at].w, &w, sizeof(w));
    }
  }
  const cudaError_t e = cudaMemcpyAsync(const_cast<char*>(plan->table), plan->jobs.data(), plan->jobs.size(), cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) { set_error(std::string("step products, tables: ") + cudaGetErrorString(e)); return FIRA_ERR_CUDA; }
  return FIRA_OK;
}

fira_status part_step_run(const PartStepPlan& plan, const MatDev* mats_dev, int qa, int qb, int update, const Hyper& hp,
                          unsigned* status_dev, cudaStream_t st) {
  const int sms = prepared_sms();
  if (!sms) return FIRA_ERR_CUDA;
  const int first = plan.tile_start[qa], count = plan.tile_start[qb] - first;
  if (count == 0) return FIRA_OK;
  const BackJob* jobs = reinterpret_cast<const BackJob*>(plan.table) + (update ? plan.njobs : 0);
  const TileDev* tiles = reinterpret_cast<const TileDev*>(plan.table + align_up(plan.jobs.size())) + first;
  const int grid = 2 * std::min(count, sms / 2);
  const cudaError_t e = launch_chained(kernel_of(update ? MODE_UPDATE : MODE_NORM, plan.deep), grid, THREADS,
                                       smem_bytes(update ? MODE_UPDATE : MODE_NORM), st, true, 1, jobs, tiles, count, mats_dev, hp, status_dev);
  if (e != cudaSuccess) { set_error(std::string("step back-projection: ") + cudaGetErrorString(e)); return FIRA_ERR_CUDA; }
  return FIRA_OK;
}

}  // namespace fira
