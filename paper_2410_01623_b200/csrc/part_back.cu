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

#include "limit.cuh"
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
// A tile with what its kernels need to know of its matrix (in the tables that is a chain of dependent loads).
struct alignas(32) TileDev {
  const float* kvec;
  int job, i0, j0, m, n;
  unsigned short nk;
  unsigned char shape;                          // see issue_parts
  unsigned char left;
};
static_assert(sizeof(TileDev) == 32, "TileDev layout");
struct alignas(32) TileNorm {
  unsigned long long* shares;                   // of ||S||^2: a double in two marked words per tile of the matrix (k_part_step)
  int index, tiles, mat, unused;                // the tile's index among them
};

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

// (Loads that stay where they are: k_part_step fetches the records one tile ahead.)
__device__ __forceinline__ TileDev load_tile(const TileDev* t) {
  union { TileDev d; int v[8]; } u;
#pragma unroll
  for (int i = 0; i < 8; i += 4)
    asm volatile("ld.global.nc.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(u.v[i]), "=r"(u.v[i + 1]), "=r"(u.v[i + 2]), "=r"(u.v[i + 3]) : "l"(reinterpret_cast<const int*>(t) + i));
  return u.d;
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

// ---------------------------------------------------------------- norm and update in one kernel (lists of fp32 matrices)
// A tile keeps its residual S = k (G - Pi R) on the chip until the limiter factor of its matrix is known:
//   first pass   D = Pi R; S, its share of ||S||^2
//   second pass  D = Pi N; W <- W - lr (a_low D + a_res lambda S)
// G is read once, and neither the correction of X for lambda nor a kernel for lambda is left.  S, and with it the update, has
// the precision of the residual itself.
//
// lambda takes its time: all tiles of the matrix have to finish their first pass.  So a pair makes the first pass of its next tile
// before the second pass of the one before: 1st of tile 0, 1st of 1, 2nd of 0, 1st of 2, 2nd of 1, ...  S waits in tensor memory
// meanwhile.
//
// Tiles of one matrix wait for one another.  A pair takes its tiles in the list's order, and the first pass of tile x waits for
// nothing but the second pass of tile x - 2 pairs, which waits for the first passes of that tile's matrix: all of
// them come before x as long as no matrix has more than 2 pairs tiles (other lists: two kernels).  So the waits cannot form a cycle
// when all pairs of the grid are resident, which a cooperative launch ensures.
//
// Tensor memory: the main product alternates between two accumulators every PROMOTE of k, the small products have one, S waits in
// the last 128 columns.  All pieces are added up in registers.  (Two regions for every pass of a rank up to PROMOTE, S in the place
// of the main products just read, so that the second pass's MMAs need not wait for the first's reading: 111 us where this takes 95.)
//
// The box loader brings a tile's boxes of G in its first and those of W in its second pass, 128 rows x 32 columns (128-byte
// swizzle), through one ring of buffers.  A thread that waits for a buffer, arms its barrier and
// issues one load does that every 460 cycles whatever the size, one that waits, stores and hands on as well: with smaller
// boxes those two threads set the pace.  Warp 1 of the odd CTA deals with the other pairs: it adds up the shares of the pair's
// epilogue warps, leaves the tile's, waits for those of the matrix's other tiles and hands lambda to the epilogue.  (Counting tiles
// and polling in every epilogue warp, lambda came 20 us after the last share.)
//
// Warp roles: 0 operand producer, 1 MMA issuer (even CTA) and owner of the tensor memory, the norm (odd CTA), 2 box loader, 3-10 epilogue
// (12 warps in all: a thirteenth would leave 128 registers per thread), 11 box storer.
constexpr int RU_STAGES = 4;
constexpr int RU_BUFS = 5;
constexpr int RU_RECORDS = 4;                   // (the box loader, who brings them, may be as many passes ahead as there are buffers: it waits for a free place)
constexpr int RU_GROUPS = 2;                    // of epilogue warps
constexpr int RU_COLS = PN / RU_GROUPS;         // a group's columns: neighbours
constexpr int RU_BOX_COLS = 32;
constexpr int RU_BOXES = RU_COLS / RU_BOX_COLS; // of G, of W, per group and tile
constexpr int RU_BOX_BYTES = PM / 2 * RU_BOX_COLS * 4;
constexpr int RU_WARPS = 4 * RU_GROUPS;         // epilogue warps of a CTA
constexpr int RU_THREADS = 32 * 3 + 32 * RU_WARPS + 32;

struct StepCtl {
  uint64_t full[RU_STAGES], empty[RU_STAGES];
  uint64_t main_full[2];                        // a piece of the main product is complete
  uint64_t main_empty[2], small_empty;          // a piece, the small products of a pass have been read
  uint64_t efull[RU_BUFS], eready[RU_BUFS], eempty[RU_BUFS];
  uint64_t esync[RU_GROUPS];
  uint64_t shared_in[2];                        // (odd CTA; tiles in turn) the shares of the epilogue warps
  uint64_t lambda_in[2];
  uint64_t record_in[RU_RECORDS];               // the epilogue's copies of the tiles' records
  uint64_t record_out[RU_RECORDS];              //   "  the epilogue warps have made the tile's second pass
  uint32_t tmem_base;
  int abort_flag;
  alignas(16) float ks[RU_GROUPS][2][RU_COLS];
  float shares[2][2 * RU_WARPS], lambda[2];
  TileDev records[RU_RECORDS];
};
constexpr size_t RU_SMEM_BYTES = (size_t)RU_STAGES * SLAB_BYTES + (size_t)RU_BUFS * RU_BOX_BYTES + sizeof(StepCtl);
static_assert(RU_SMEM_BYTES <= 227 * 1024, "shared memory budget");

// A pair's passes in their order: f(pass, tile, its index), false: stop.  The tiles' records are fetched one ahead; ahead(tile) sees
// them between the passes, before their turn.
struct NoLook { __device__ __forceinline__ void operator()(const TileDev&) const {} };
template <class F, class A = NoLook>
__device__ __forceinline__ void passes(const TileDev* tiles, int pair, int count, int npairs, const F& f, const A& ahead = A()) {
  TileDev last = load_tile(tiles + pair), next = last;           // (every pair has a tile)
  for (int t = pair;; t += npairs) {
    const TileDev d = next;
    if (t < count) {
      if (t + npairs < count) next = load_tile(tiles + t + npairs);
      if (!f(0, d, t)) return;
      ahead(next);
    }
    if (t > pair && !f(1, last, t - npairs)) return;
    if (t >= count) return;
    last = d;
  }
}
// f(first column) for a tile's boxes in their order: the first of either group, the second, ...
template <class F>
__device__ __forceinline__ bool each_box(const TileDev& d, const F& f) {
#pragma unroll
  for (int b = 0; b < RU_BOXES; ++b)
#pragma unroll
    for (int g = 0; g < RU_GROUPS; ++g) {
      const int j = d.j0 + RU_COLS * g + RU_BOX_COLS * b;
      if (j < d.n && !f(j)) return false;
    }
  return true;
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(RU_THREADS, 1)
k_part_step(const BackJob* __restrict__ jobs, int njobs, const TileDev* __restrict__ tiles, const TileNorm* __restrict__ norms, int count,
            const MatDev* __restrict__ mats, Hyper hp, unsigned* __restrict__ status) {
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char* boxes = smem + RU_STAGES * SLAB_BYTES;
  StepCtl* ctl = reinterpret_cast<StepCtl*>(boxes + RU_BUFS * RU_BOX_BYTES);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = ptx::cluster_ctarank();
  const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  const bool smem_ok = (ptx::smem_u32(smem) & 1023u) == 0;
  if (threadIdx.x == 0) {
    for (int s = 0; s < RU_STAGES; ++s) {
      ptx::mbar_init(ptx::smem_u32(&ctl->full[s]), 1);
      ptx::mbar_init(ptx::smem_u32(&ctl->empty[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      ptx::mbar_init(ptx::smem_u32(&ctl->main_full[b]), 1);
      ptx::mbar_init(ptx::smem_u32(&ctl->main_empty[b]), 2 * RU_WARPS);          // every epilogue warp of the pair
      ptx::mbar_init(ptx::smem_u32(&ctl->shared_in[b]), 1);
      ptx::mbar_init(ptx::smem_u32(&ctl->lambda_in[b]), 1);
    }
    ptx::mbar_init(ptx::smem_u32(&ctl->small_empty), 2 * RU_WARPS);
    for (int b = 0; b < RU_BUFS; ++b) {
      ptx::mbar_init(ptx::smem_u32(&ctl->efull[b]), 1);
      ptx::mbar_init(ptx::smem_u32(&ctl->eready[b]), GROUP_THREADS);
      ptx::mbar_init(ptx::smem_u32(&ctl->eempty[b]), 1);
    }
    for (int g = 0; g < RU_GROUPS; ++g) ptx::mbar_init(ptx::smem_u32(&ctl->esync[g]), GROUP_THREADS);
    for (int b = 0; b < RU_RECORDS; ++b) {
      ptx::mbar_init(ptx::smem_u32(&ctl->record_in[b]), 1);
      ptx::mbar_init(ptx::smem_u32(&ctl->record_out[b]), RU_WARPS);
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
      passes(tiles, pair, count, npairs, [&](int pass, const TileDev& d, int) {
        const BackJob* jb = jobs + pass * njobs + d.job;
        const int bytes = 2 * ((d.shape & 3) * A_PART + ((d.shape >> 2) & 3) * B_PART);
        const int i0 = d.i0 + PM / 2 * (int)rank, j0 = d.j0 + PN / 2 * (int)rank;
        for (int k = 0; k < d.nk; ++k) {
          if (!ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->empty[stage]), phase ^ 1u, abort_flag)) return ok = false;
          const uint32_t fb = ptx::map_to_cta(ptx::smem_u32(&ctl->full[stage]), 0);
          const uint32_t sa = slabs + stage * SLAB_BYTES;
          if (rank == 0) ptx::mbar_expect_tx(ptx::smem_u32(&ctl->full[stage]), bytes);
          ptx::tma_load_3d_pair(sa, &jb->a, fb, k * PK, i0, 0);
          ptx::tma_load_3d_pair(sa + 3 * A_PART, &jb->b, fb, k * PK, j0, 0);
          if (++stage == RU_STAGES) { stage = 0; phase ^= 1u; }
        }
        return true;
      }, [&](const TileDev& d) {
        ptx::prefetch_map(&jobs[d.job].a); ptx::prefetch_map(&jobs[d.job].b);
        ptx::prefetch_map(&jobs[njobs + d.job].a); ptx::prefetch_map(&jobs[njobs + d.job].b);
      });
      if (!ok && rank == 0) {   // give copies in flight a bounded time to land
        for (int s = 0; s < RU_STAGES; ++s)
          for (uint32_t it = 0; it < (1u << 16); ++it)
            if (ptx::mbar_try_wait_cluster(ptx::smem_u32(&ctl->full[s]), (s < stage) ? phase : (phase ^ 1u))) break;
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && smem_ok && rank == 0) {
      int stage = 0; uint32_t phase = 0;
      int piece = 0; uint32_t sphase = 0;
      const uint32_t tmem = ctl->tmem_base, small = tmem + 2 * PN;
      passes(tiles, pair, count, npairs, [&](int, const TileDev& d, int) {
        if (!ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->small_empty), sphase ^ 1u, abort_flag)) return false;
        sphase ^= 1u;
        for (int k = 0; k < d.nk; ++k) {
          const int mb = piece & 1;
          const bool fresh = k % PROMOTE_SLABS == 0;
          if (fresh && !ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->main_empty[mb]), ((piece >> 1) & 1) ^ 1u, abort_flag)) return false;
          if (!ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->full[stage]), phase, abort_flag)) return false;
          ptx::tc_fence_after();
          issue_parts(d.shape, tmem + mb * PN, small, slabs + stage * SLAB_BYTES, 3 * A_PART, fresh, k == 0);
          ptx::umma_commit_pair(ptx::smem_u32(&ctl->empty[stage]), 3);
          if (++stage == RU_STAGES) { stage = 0; phase ^= 1u; }
          if ((k + 1) % PROMOTE_SLABS == 0 || k + 1 == d.nk) {   // (covers the small products so far as well)
            ptx::umma_commit_pair(ptx::smem_u32(&ctl->main_full[mb]), 3);
            ++piece;
          }
        }
        return true;
      });
    } else if (smem_ok && rank == 1) {
      // ---------------------------------------------------------- the norm
      int firsts = 0, seconds = 0;
      passes(tiles, pair, count, npairs, [&](int pass, const TileDev& d, int t) {
        const TileNorm tn = norms[t];
        if (pass == 0) {
          const int b = firsts & 1;
          if (lane == 0) ptx::mbar_expect_tx(ptx::smem_u32(&ctl->shared_in[b]), sizeof(ctl->shares[b]));
          if (!ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->shared_in[b]), (firsts >> 1) & 1, abort_flag)) return false;
          ++firsts;
          const double sum = warp_sum(lane < 2 * RU_WARPS ? (double)ctl->shares[b][lane] : 0.0);
          if (lane == 0) ptx::put_marked(tn.shares + PART_SHARE_WORDS * tn.index, sum);
          return true;
        }
        const int b = seconds++ & 1;
        Limit lim;
        const MatDev& mt = mats[tn.mat];
        if (!wait_limit<double>(tn.shares, tn.tiles, mt, mt.bias->prev, hp, abort_flag, lim)) return false;
        if (lane < 2)
          ptx::st_async_f32(ptx::map_to_cta(ptx::smem_u32(&ctl->lambda[b]), lane), lim.lambda * lim.kmat, ptx::map_to_cta(ptx::smem_u32(&ctl->lambda_in[b]), lane));
        if (tn.index == 0) store_limit(mt, hp, lim, status);
        return true;
      });
    }
  } else if (warp == 2) {
    // ------------------------------------------------------------ box loader
    if (lane == 0 && smem_ok) {
      int box = 0, records = 0;
      passes(tiles, pair, count, npairs, [&](int pass, const TileDev& d, int) {
        const BackJob* jb = jobs + d.job;
        if (pass == 0) {
          const int place = records % RU_RECORDS;
          if (!ptx::mbar_wait(ptx::smem_u32(&ctl->record_out[place]), ((records / RU_RECORDS) & 1) ^ 1u, abort_flag)) return false;
          ctl->records[place] = d;
          ptx::mbar_arrive(ptx::smem_u32(&ctl->record_in[place]));
          ++records;
        }
        const int i0 = d.i0 + PM / 2 * (int)rank;
        return each_box(d, [&](int j) {
          const int slot = box % RU_BUFS;
          if (!ptx::mbar_wait(ptx::smem_u32(&ctl->eempty[slot]), ((box / RU_BUFS) & 1) ^ 1u, abort_flag)) return false;
          const uint32_t fb = ptx::smem_u32(&ctl->efull[slot]);
          ptx::mbar_expect_tx(fb, RU_BOX_BYTES);
          ptx::tma_load_2d(boxes_u32 + slot * RU_BOX_BYTES, pass ? &jb->w : &jb->g, fb, j, i0);
          ++box;
          return true;
        });
      }, [&](const TileDev& d) {
        ptx::prefetch_map(&jobs[d.job].g); ptx::prefetch_map(&jobs[d.job].w);
      });
    }
  } else if (warp >= 3 + RU_WARPS) {
    // ------------------------------------------------------------ box storer; hands the buffers back
    if (lane == 0 && smem_ok) {
      int box = 0;
      passes(tiles, pair, count, npairs, [&](int pass, const TileDev& d, int) {
        const BackJob* jb = jobs + d.job;
        const int i0 = d.i0 + PM / 2 * (int)rank;
        // A box of W is handed back when the next one is on its way: the reading of one overlaps the issue of the next.
        uint32_t held = 0;                              // barrier to arrive on (0: none)
        if (!each_box(d, [&](int j) {
              const int slot = box % RU_BUFS;
              if (!ptx::mbar_wait(ptx::smem_u32(&ctl->eready[slot]), (box / RU_BUFS) & 1, abort_flag)) return false;
              const uint32_t freed = ptx::smem_u32(&ctl->eempty[slot]);
              if (pass == 0) {
                ptx::mbar_arrive(freed);
              } else {
                if (i0 < d.m) ptx::tma_store_2d(&jb->w, boxes_u32 + slot * RU_BOX_BYTES, j, i0);
                ptx::bulk_commit_group();                // (empty where the rows are past the matrix)
                ptx::bulk_wait_group_read<1>();          // the box before this one has been read
                if (held) ptx::mbar_arrive(held);
                held = freed;
              }
              ++box;
              return true;
            })) return false;
        if (held) {
          ptx::bulk_wait_group_read<0>();
          ptx::mbar_arrive(held);
        }
        return true;
      });
      ptx::bulk_wait_group_all();
    }
  } else if (smem_ok) {
    // ------------------------------------------------------------ epilogue
    const int ew = warp - 3, g = ew >> 2;
    const int quarter = warp & 3;                       // TMEM lanes 32 * quarter .. + 31
    const int row = quarter * 32 + lane, tid_g = (ew & 3) * 32 + lane;
    const uint32_t esync = ptx::smem_u32(&ctl->esync[g]);
    const uint32_t me[2] = {ptx::map_to_cta(ptx::smem_u32(&ctl->main_empty[0]), 0), ptx::map_to_cta(ptx::smem_u32(&ctl->main_empty[1]), 0)};
    const uint32_t se = ptx::map_to_cta(ptx::smem_u32(&ctl->small_empty), 0);
    const uint32_t tmem = ctl->tmem_base + ((uint32_t)(quarter * 32) << 16) + g * RU_COLS, parked = tmem + 3 * PN;
    uint32_t yphase = 0;
    int base = 0, parity = 0, piece = 0;                // base: boxes of the passes so far
    // This thread's row of a pass's product, the group's columns.
    auto product = [&](const TileDev& d, float (&v)[RU_COLS]) {
#pragma unroll
      for (int e = 0; e < RU_COLS; ++e) v[e] = 0.f;
      for (int k = 0; k < d.nk; k += PROMOTE_SLABS, ++piece) {
        if (!ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->main_full[piece & 1]), (piece >> 1) & 1, abort_flag)) return false;
        ptx::tc_fence_after();
        if (k + PROMOTE_SLABS >= d.nk) {                 // the small products first: the next pass waits for their place
          add_columns(v, tmem + 2 * PN);
          if (lane == 0) ptx::mbar_arrive_cluster(se);
        }
        add_columns(v, tmem + (piece & 1) * PN);
        if (lane == 0) ptx::mbar_arrive_cluster(me[piece & 1]);
      }
      return true;
    };
    // f(place in shared memory, first column) on every 16-byte word of this thread's row of the group's boxes; hands them on.
    auto boxes_of = [&](const TileDev& d, bool written, auto f) {
      const uint32_t sw = (uint32_t)row & 7u;            // 128-byte swizzle: slot ^= row % 8
      auto boxes_in = [&](int group) { return max(0, min(RU_BOXES, (d.n - d.j0 - RU_COLS * group + RU_BOX_COLS - 1) / RU_BOX_COLS)); };
      const int n0 = boxes_in(0), n1 = boxes_in(1), own = g ? n1 : n0, first = base;
      base += n0 + n1;
#pragma unroll
      for (int b = 0; b < RU_BOXES; ++b) {
        if (b >= own) break;
        const int box = first + (g ? 2 * b + 1 : b + min(b, n1)), slot = box % RU_BUFS;
        if (!ptx::mbar_wait(ptx::smem_u32(&ctl->efull[slot]), (box / RU_BUFS) & 1, abort_flag)) return false;
        unsigned char* place = boxes + slot * RU_BOX_BYTES + row * 128;
#pragma unroll
        for (int q = 0; q < 8; ++q) f(reinterpret_cast<float4*>(place + (((uint32_t)q ^ sw) << 4)), RU_BOX_COLS * b + 4 * q);
        if (written) ptx::fence_proxy_async_smem();
        ptx::mbar_arrive(ptx::smem_u32(&ctl->eready[slot]));
      }
      return true;
    };
    float s[RU_COLS];                                   // the residual of the first pass's tile
    int firsts = 0, seconds = 0;                        // passes made
    auto park = [&] {
#pragma unroll
      for (int h = 0; h < RU_COLS; h += 16) {
        uint32_t v[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) v[e] = __float_as_uint(s[h + e]);
        __syncwarp();
        ptx::tmem_st_32x32b_x16(parked + h, v);
      }
      ptx::tmem_st_wait();
    };
    auto first_pass = [&](const TileDev& d) {
      const int left = d.left, i0 = d.i0 + PM / 2 * (int)rank, j0 = d.j0 + RU_COLS * g;
      const bool one = hp.mode & HYPER_MATRIX_SCALING;
      const int l = left ? j0 + tid_g : i0 + row, L = left ? d.n : d.m;
      float k = 0.f;                                     // of column j0 + tid_g (left) or of this row
      if (l < L && (!left || tid_g < RU_COLS)) k = one ? 1.f : __ldg(d.kvec + l);
      if (firsts) park();
      if (!product(d, s)) return false;
      float* ks = ctl->ks[g][parity];
      if (left && tid_g < RU_COLS) ks[tid_g] = k;
      ptx::mbar_arrive(esync);                           // the group's factors are in place
      if (!ptx::mbar_wait(esync, yphase, abort_flag)) return false;
      yphase ^= 1u;
      parity ^= 1;
      float ss = 0.f;
      if (!boxes_of(d, false, [&](const float4* p, int c) {
            const float4 gv = *p, k4 = left ? *reinterpret_cast<const float4*>(ks + c) : make_float4(k, k, k, k);
            const float ge[4] = {gv.x, gv.y, gv.z, gv.w}, kf[4] = {k4.x, k4.y, k4.z, k4.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {                // (G is zero past the matrix, D as well: its operands are)
              s[c + e] = kf[e] * (ge[e] - s[c + e]);
              ss = fmaf(s[c + e], s[c + e], ss);
            }
          })) return false;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
      if (lane == 0)
        ptx::st_async_f32(ptx::map_to_cta(ptx::smem_u32(&ctl->shares[firsts & 1][(int)rank * RU_WARPS + ew]), 1), ss,
                          ptx::map_to_cta(ptx::smem_u32(&ctl->shared_in[firsts & 1]), 1));
      ++firsts;
      return true;
    };
    auto second_pass = [&](const TileDev& d) {
      float dv[RU_COLS];
      const int x = seconds++;
      if (threadIdx.x == 32 * 3) ptx::mbar_expect_tx(ptx::smem_u32(&ctl->lambda_in[x & 1]), sizeof(float));
      if (!product(d, dv)) return false;
      if (!ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->lambda_in[x & 1]), (x >> 1) & 1, abort_flag)) return false;
      const float cres = hp.a_res * ctl->lambda[x & 1];
      if (seconds == firsts) park();                     // (no tile has followed this one)
      uint32_t sv[16];
      return boxes_of(d, true, [&](float4* p, int c) {
        if (c % 16 == 0) {
          __syncwarp();
          ptx::tmem_ld_32x32b_x16(parked + c, sv);
          ptx::tmem_ld_wait();
        }
        const float4 w = *p;
        float we[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) we[e] = we[e] - hp.lr * (hp.a_low * dv[c + e] + cres * __uint_as_float(sv[c % 16 + e]));
        *p = make_float4(we[0], we[1], we[2], we[3]);
      });
    };
    // (The records come through shared memory: the registers that would hold the next one are not there.)
    for (int t = pair;; t += npairs) {
      const int r = firsts;
      if (t < count && (!ptx::mbar_wait(ptx::smem_u32(&ctl->record_in[r % RU_RECORDS]), (r / RU_RECORDS) & 1, abort_flag) ||
                        !first_pass(ctl->records[r % RU_RECORDS]))) break;
      if (t > pair) {
        const int q = seconds % RU_RECORDS;
        if (!second_pass(ctl->records[q])) break;
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&ctl->record_out[q]));
      }
      if (t >= count) break;
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
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_part_step, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RU_SMEM_BYTES);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) sms_of_device[dev].store(sms);
  }
  if (e != cudaSuccess) { set_error(std::string("step products: ") + cudaGetErrorString(e)); return 0; }
  return sms;
}

// CTA pairs of k_part_step that are resident at once (0: error).
int resident_pairs() {
  const int sms = prepared_sms();
  if (!sms) return 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * (sms / 2)); cfg.blockDim = dim3(RU_THREADS); cfg.dynamicSmemBytes = RU_SMEM_BYTES;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  cfg.attrs = at; cfg.numAttrs = 1;
  int pairs = 0;
  const cudaError_t e = cudaOccupancyMaxActiveClusters(&pairs, k_part_step, &cfg);
  if (e != cudaSuccess || pairs <= 0) { set_error(std::string("step products, cudaOccupancyMaxActiveClusters: ") + cudaGetErrorString(e)); return 0; }
  return std::min(pairs, sms / 2);
}

// Box of 128 rows x row_bytes over G or W (or their aligned copies).
bool encode_box(CUtensorMap* map, const void* base, const MatDev& mt, int row_bytes) {
  const int es = mt.bf16 ? 2 : 4;
  const unsigned long long extent[2] = {(unsigned long long)mt.n, (unsigned long long)mt.m};
  const unsigned long long stride[1] = {(unsigned long long)(mt.Gs ? mt.lds : mt.ld) * es};
  const unsigned box[2] = {(unsigned)(row_bytes / es), PM / 2};
  return encode_tiled(map, base, !mt.bf16, 2, extent, stride, box, row_bytes);
}

}  // namespace

size_t part_step_table_bytes(int njobs, int ntiles) {
  return align_up(2 * sizeof(BackJob) * (size_t)njobs) + align_up(sizeof(TileDev) * (size_t)ntiles) + align_up(sizeof(TileNorm) * (size_t)ntiles);
}

fira_status part_step_prepare(const std::vector<MatDev>& mats, const std::vector<int>& list, char* table_dev, PartStepPlan* plan, cudaStream_t st) {
  std::vector<TileDev> td;
  std::vector<TileNorm> tns;
  plan->jobs.assign(2 * list.size() * sizeof(BackJob), 0);
  plan->tile_start.assign(1, 0);
  plan->deep = 0;
  int pairs = resident_pairs();
  if (!pairs) return FIRA_ERR_CUDA;
  pairs = std::min(pairs, stream_sms(st) / 2);
  // One kernel for norm and update.  Steps with two kernels / with one, us, lists back to back, limiter acting on all: 56 matrices 512 / 1376 fp32
  // r = 64 246 / 201, 128 256 / 210, 160 372 / 289, 192 391 / 306, 256 429 / 338; 14 of 1024 / 2736 r = 128 223 / 198, 192 319 / 260, 256 347 / 288,
  // 384 484 / 399, 512 628 / 528; 14 of 768 / 2048 r = 64 132 / 116, 384 304 / 247; 112 of 288 / 992, r = 64, 286 / 238; 140 of 160 / 416, r = 40, 150 / 117;
  // 28 of 640 / 1707 r = 100 (copies to an aligned pitch) 271 / 233.  Limiter acting on none, inputs not in L2: 56 of 512 / 1376, r = 128, 246 / 239.
  // bf16, where G is half of the traffic less: 28 of 640 / 1707, 185 / 189.
  plan->one_kernel_pairs = pairs;
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
      for (int j0 = 0; j0 < mt.n; j0 += PN) {
        TileDev d;
        d.kvec = mt.kvec;
        d.job = (int)q; d.i0 = i0; d.j0 = j0; d.m = mt.m; d.n = mt.n;
        d.nk = (unsigned short)((mt.r + PK - 1) / PK);
        d.shape = (unsigned char)reinterpret_cast<const BackJob*>(&jd[q])->shape;
        d.left = (unsigned char)(mt.left != 0);
        TileNorm tn;
        tn.shares = reinterpret_cast<unsigned long long*>(mt.part);
        tn.index = (int)td.size() - plan->tile_start.back(); tn.tiles = part_step_tiles(mt.m, mt.n); tn.mat = list[q]; tn.unused = 0;
        td.push_back(d);
        tns.push_back(tn);
      }
    plan->tile_start.push_back((int)td.size());
    if (mt.r > split::PROMOTE) plan->deep = 1;
    if (mt.bf16 || part_step_tiles(mt.m, mt.n) > 2 * pairs) plan->one_kernel_pairs = 0;
  }
  plan->table = table_dev; plan->njobs = (int)list.size();
  cudaError_t e = cudaMemcpyAsync(table_dev + align_up(plan->jobs.size()), td.data(), sizeof(TileDev) * td.size(), cudaMemcpyHostToDevice, st);
  plan->ntiles = (int)td.size();
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(table_dev + align_up(plan->jobs.size()) + align_up(sizeof(TileDev) * td.size()), tns.data(), sizeof(TileNorm) * tns.size(), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) { set_error(std::string("step products, tables: ") + cudaGetErrorString(e)); return FIRA_ERR_CUDA; }
  return FIRA_OK;
}

fira_status part_step_update_pointers(const std::vector<MatDev>& mats, const std::vector<int>& list, PartStepPlan* plan, cudaStream_t st) {
  BackJob* jd = reinterpret_cast<BackJob*>(plan->jobs.data());
  for (size_t q = 0; q < list.size(); ++q) {
    const MatDev& mt = mats[list[q]];
    CUtensorMap g, w;
    const int row_bytes = plan->one_kernel_pairs ? RU_BOX_COLS * 4 : 64;
    if (!encode_box(&g, mt.Gs ? mt.Gs : mt.G, mt, row_bytes) || !encode_box(&w, mt.Gs ? mt.Ws : mt.W, mt, row_bytes)) return FIRA_ERR_CUDA;
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

fira_status part_step_run_one_kernel(const PartStepPlan& plan, const MatDev* mats_dev, int qa, int qb, const Hyper& hp, unsigned* status_dev, cudaStream_t st) {
  if (!prepared_sms()) return FIRA_ERR_CUDA;
  const int first = plan.tile_start[qa], count = plan.tile_start[qb] - first;
  if (count == 0) return FIRA_OK;
  const BackJob* jobs = reinterpret_cast<const BackJob*>(plan.table);
  const char* table = plan.table + align_up(plan.jobs.size());
  const TileDev* tiles = reinterpret_cast<const TileDev*>(table) + first;
  const TileNorm* norms = reinterpret_cast<const TileNorm*>(table + align_up(sizeof(TileDev) * (size_t)plan.ntiles)) + first;
  const cudaError_t e = launch_resident(k_part_step, 2 * std::min(count, plan.one_kernel_pairs), RU_THREADS, RU_SMEM_BYTES, st,
                                        true, 1, jobs, plan.njobs, tiles, norms, count, mats_dev, hp, status_dev);
  if (e != cudaSuccess) { set_error(std::string("step residual and update: ") + cudaGetErrorString(e)); return FIRA_ERR_CUDA; }
  return FIRA_OK;
}

}  // namespace fira
