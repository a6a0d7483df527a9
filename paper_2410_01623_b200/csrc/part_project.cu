// The step's projection R = G^T Pi (or G Pi) in fp32 precision, for long lists (part_gemm.cuh: PartStepPlan).  G is split
// into bf16 parts on its way into shared memory, the projection is kept as parts, R is left as parts.
//
//   R[l][j] = sum_d G(d,l) Pi[d][j]
//
// CTA pairs, one CTA per SM, persistent; 256 l x 128 j tiles.  Eight converter warps per CTA read a slab of G (32 deep, 128 of
// its l) with ordinary loads, two slabs ahead, whatever its alignment, and write its parts in the operand's swizzled layout:
// no copy of G in another form is made in memory.  The projection's slabs come by TMA (part_slab.cuh).  Tensor memory as in
// part_gemm.cu: the main product alternates between two accumulators every PROMOTE of k and is summed in fp32 registers.
//
// Epilogue: two groups of four warps, each on half of the tile's columns, one row per thread; R's parts leave as TMA boxes of
// 128 rows x 16 columns x three parts.  The moments are a pass of their own (k_moments).  With Adam in this epilogue, M and V as
// boxes, the epilogue took 30000 cycles per tile and the product, whose main accumulators wait for the same warps
// every PROMOTE of k, stood still for half of them; and M and V had to be addressable by TMA.
// Measured (56 matrices 512 / 1376, r = 128): 61 us, 0.65 of the MMAs' time at full rate.
//
// What bounds it: the MMAs (12 per slab), G at the copy bandwidth close behind.
//
// Warp roles: 0 producer of the projection's slabs, 1 MMA issuer (even CTA) and owner of the tensor memory, 2-9 epilogue,
// 10 box storer, 11-18 converters, 19 and (odd CTA) 1 relays.
//
// The odd CTA's converted slabs are announced to the issuer, in the other CTA, by relays: the converters release their writes
// to a barrier of their own CTA, a relay's thread acquires them there and releases them to the issuer's barrier at cluster
// scope.  (Measured, 56 matrices 512 / 1376 fp32 / 28 of 640 / 1707 bf16: 72 / 62 us with two relays for the slabs in turn, 73 / 70
// with one, 74 / 63 with three, 79 / 68 with a lane of one warp per stage, 100 / 88 where the converters release at cluster scope
// themselves, which waits for their loads in flight.  70 / 60 with the barrier's default scope, the CTA: not enough by the
// memory model.)
#include <string.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "part_slab.cuh"
#include "split_gemm.cuh"
#include "step_simt.cuh"

namespace fira {

namespace {

constexpr int STAGES = 4;
constexpr int PROMOTE_SLABS = split::PROMOTE / PK;
constexpr int SLAB_BYTES = 3 * (A_PART + B_PART);
constexpr int EPI_WARPS = 8, CONV_WARPS = 8, CONV_THREADS = 32 * CONV_WARPS;
constexpr int GROUPS = 2, GROUP_THREADS = 128;
constexpr int FIRST_CONV = 3 + EPI_WARPS;                 // warp
constexpr int RELAYS = 2, FIRST_RELAY = FIRST_CONV + CONV_WARPS;     // (the first relay is warp 1)
constexpr int THREADS = 32 * (FIRST_RELAY + RELAYS - 1);
constexpr int COLS = 16;                        // of a box
constexpr int OUT_BUFS = 2;                     // per group
constexpr int OUT_PART = PM / 2 * COLS * 2, OUT_BUF = 3 * OUT_PART;         // 4 KiB; three parts
constexpr int GROUP_BYTES = OUT_BUFS * OUT_BUF;
constexpr int BOXES = PN / 2 / COLS;            // of a group per tile
constexpr int UNITS = PM / 2 * PK / 8 / CONV_THREADS;      // units of eight neighbours of a slab per converter thread

struct alignas(64) ProjJob {
  CUtensorMap b;                                // the projection's parts, [d][r]
  CUtensorMap ro;                               // parts of R, [3][l][r]
  int mat;                                      // index into the problem table
  int shape;                                    // see issue_parts
};
static_assert(sizeof(ProjJob) % 64 == 0, "tensor maps must stay 64-byte aligned");
struct TileDev { int job, l0, j0, nk; };

struct ProjCtl {
  uint64_t full[STAGES], empty[STAGES];
  uint64_t converted[STAGES];                   // (odd CTA) its converters have written the slab
  uint64_t main_full[2], main_empty[2];         // a piece of the main product is complete / has been read
  uint64_t small_empty[2];                      // the small products of a tile have been read
  uint64_t oready[GROUPS][OUT_BUFS], oempty[GROUPS][OUT_BUFS];   // R's parts written / stored
  uint32_t tmem_base;
  int abort_flag;
};
constexpr size_t SMEM_BYTES = (size_t)STAGES * SLAB_BYTES + GROUPS * GROUP_BYTES + sizeof(ProjCtl);
static_assert(SMEM_BYTES <= 227 * 1024, "shared memory budget");

__device__ __forceinline__ TileDev load_tile(const TileDev* t) {
  const int4 v = __ldg(reinterpret_cast<const int4*>(t));
  return TileDev{v.x, v.y, v.z, v.w};
}

// A converter thread's units of one slab.  left (G is [d][l]): unit (l / 8, d), 128-byte rows of 64 l with the 128-byte swizzle;
// right (G is [l][d]): unit (l, d / 8), 64-byte rows with the 64-byte swizzle.
template <typename T>
struct Slab {
  split::Frag<T> f[UNITS];

  __device__ __forceinline__ static void coords(int u, bool left, int& l, int& d) {
    const int e = (threadIdx.x - 32 * FIRST_CONV) + CONV_THREADS * u;
    if (left) { l = e % 16 * 8; d = e / 16; } else { d = e % 4 * 8; l = e / 4; }
  }
  // REGULAR: whole aligned units only (see load_frag); l past the matrix reads its last rows again, for rows of R that
  // nobody looks at (L: the extent that may be read).
  template <bool REGULAR>
  __device__ __forceinline__ void load(const MatDev& mt, const T* G, long long ld, int L, int l0, int d0, bool left, bool vec) {
#pragma unroll
    for (int u = 0; u < UNITS; ++u) {
      int l, d;
      coords(u, left, l, d);
      l += l0; d += d0;
      if (REGULAR) l = min(l, left ? L - 8 : L - 1);
      const T* p = G + (left ? (long long)d * ld + l : (long long)l * ld + d);
      if (REGULAR) { split::load_frag(p, f[u]); continue; }
      split::load_frag(p, left ? (d < mt.d ? mt.l - l : 0) : (l < mt.l ? mt.d - d : 0), vec, f[u]);
    }
  }
  __device__ __forceinline__ void store(unsigned char* slab, bool left) const {
#pragma unroll
    for (int u = 0; u < UNITS; ++u) {
      int l, d;
      coords(u, left, l, d);
      const int at = left ? (l >> 6) * (PK * 128) + d * 128 + ((((l >> 3) & 7) ^ (d & 7)) << 4)
                          : l * 64 + (((d >> 3) ^ ((l >> 1) & 3)) << 4);
      split::store_parts(slab + at, f[u], A_PART);
    }
  }
};

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS, 1)
k_part_project(const ProjJob* __restrict__ jobs, const TileDev* __restrict__ tiles, int count, const MatDev* __restrict__ mats,
               unsigned* __restrict__ status) {
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char* boxes = smem + STAGES * SLAB_BYTES;
  ProjCtl* ctl = reinterpret_cast<ProjCtl*>(boxes + GROUPS * GROUP_BYTES);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = ptx::cluster_ctarank();
  const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  const bool smem_ok = (ptx::smem_u32(smem) & 1023u) == 0;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      ptx::mbar_init(ptx::smem_u32(&ctl->full[s]), 1 + CONV_WARPS + 1);          // the producer, this CTA's converters, a relay
      ptx::mbar_init(ptx::smem_u32(&ctl->converted[s]), CONV_WARPS);
      ptx::mbar_init(ptx::smem_u32(&ctl->empty[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      ptx::mbar_init(ptx::smem_u32(&ctl->main_full[b]), 1);
      ptx::mbar_init(ptx::smem_u32(&ctl->main_empty[b]), 2 * EPI_WARPS);
      ptx::mbar_init(ptx::smem_u32(&ctl->small_empty[b]), 2 * EPI_WARPS);
    }
    for (int g = 0; g < GROUPS; ++g)
      for (int b = 0; b < OUT_BUFS; ++b) {
        ptx::mbar_init(ptx::smem_u32(&ctl->oready[g][b]), GROUP_THREADS);
        ptx::mbar_init(ptx::smem_u32(&ctl->oempty[g][b]), 1);
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
  const uint32_t slabs = ptx::smem_u32(smem);

  // Every RELAYS-th slab of this pair's, from the `which`-th on.
  auto relay = [&](int which) {
    int slab = 0;                               // running number
    for (int t = pair; t < count; t += npairs) {
      const int end = slab + load_tile(tiles + t).nk;
      for (int s = slab + (which + RELAYS - slab % RELAYS) % RELAYS; s < end; s += RELAYS) {
        if (!ptx::mbar_wait(ptx::smem_u32(&ctl->converted[s % STAGES]), (s / STAGES) & 1, abort_flag)) return;
        ptx::mbar_arrive_release_cluster(ptx::map_to_cta(ptx::smem_u32(&ctl->full[s % STAGES]), 0));
      }
      slab = end;
    }
  };
  if (warp == 0) {
    if (lane == 0 && smem_ok) {
      int stage = 0; uint32_t phase = 0; bool ok = true;
      for (int t = pair; t < count && ok; t += npairs) {
        const TileDev d = load_tile(tiles + t);
        const ProjJob* jb = jobs + d.job;
        const int pb = (jb->shape >> 2) & 3, j0 = d.j0 + PN / 2 * (int)rank;
        for (int k = 0; k < d.nk; ++k) {
          if (!ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->empty[stage]), phase ^ 1u, abort_flag)) { ok = false; break; }
          const uint32_t fb = ptx::map_to_cta(ptx::smem_u32(&ctl->full[stage]), 0);
          if (rank == 0) ptx::mbar_expect_tx(ptx::smem_u32(&ctl->full[stage]), 2 * pb * B_PART);
          ptx::tma_load_4d_pair(slabs + stage * SLAB_BYTES + 3 * A_PART, &jb->b, fb, 0, k * PK, j0 >> 6, 0);
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
      int piece = 0, tile = 0;
      const uint32_t tmem = ctl->tmem_base;
      for (int t = pair; t < count && ok; t += npairs) {
        const TileDev d = load_tile(tiles + t);
        const int shape = jobs[d.job].shape;
        const uint32_t small = tmem + 2 * PN + (tile & 1) * PN;
        if (!ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->small_empty[tile & 1]), ((tile >> 1) & 1) ^ 1u, abort_flag)) break;
        for (int k = 0; k < d.nk; ++k) {
          const int mb = piece & 1;
          const bool fresh = k % PROMOTE_SLABS == 0;
          if (fresh && !ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->main_empty[mb]), ((piece >> 1) & 1) ^ 1u, abort_flag)) { ok = false; break; }
          if (!ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->full[stage]), phase, abort_flag)) { ok = false; break; }
          ptx::tc_fence_after();
          issue_parts(shape, tmem + mb * PN, small, slabs + stage * SLAB_BYTES, 3 * A_PART, fresh, k == 0);
          ptx::umma_commit_pair(ptx::smem_u32(&ctl->empty[stage]), 3);
          if (++stage == STAGES) { stage = 0; phase ^= 1u; }
          if ((k + 1) % PROMOTE_SLABS == 0 || k + 1 == d.nk) {   // (covers the small products so far as well)
            ptx::umma_commit_pair(ptx::smem_u32(&ctl->main_full[mb]), 3);
            ++piece;
          }
        }
        ++tile;
      }
    } else if (lane == 0 && smem_ok) {
      relay(0);
    }
  } else if (warp == 2 + EPI_WARPS) {
    // ------------------------------------------------------------ box storer
    if (lane == 0 && smem_ok) {
      int out[GROUPS] = {0, 0}; uint32_t ophase[GROUPS] = {0, 0}; bool ok = true;
      // A box's buffer is handed back when the next box is on its way: that one has another (two per group), so nobody
      // waits for what is held back, and the reading of one box overlaps the issue of the next.
      uint32_t held = 0;                                // barrier to arrive on (0: none)
      for (int t = pair; t < count && ok; t += npairs) {
        const TileDev d = load_tile(tiles + t);
        const ProjJob* jb = jobs + d.job;
        const MatDev& mt = mats[jb->mat];
        const int l0 = d.l0 + PM / 2 * (int)rank, R = mt.r;
        const bool rows = l0 < mt.l;
        for (int b = 0; b < BOXES && ok; ++b)
#pragma unroll
          for (int g = 0; g < GROUPS; ++g) {
            const int j = d.j0 + g * (PN / 2) + b * COLS;
            if (j >= R) continue;
            if (!ptx::mbar_wait(ptx::smem_u32(&ctl->oready[g][out[g]]), ophase[g], abort_flag)) { ok = false; break; }
            if (rows) ptx::tma_store_3d(&jb->ro, slabs + STAGES * SLAB_BYTES + g * GROUP_BYTES + out[g] * OUT_BUF, j, l0, 0);
            ptx::bulk_commit_group();                  // (empty where the rows are past the matrix)
            ptx::bulk_wait_group_read<1>();            // the box before this one has been read
            if (held) ptx::mbar_arrive(held);
            held = ptx::smem_u32(&ctl->oempty[g][out[g]]);
            if (++out[g] == OUT_BUFS) { out[g] = 0; ophase[g] ^= 1u; }
          }
      }
      ptx::bulk_wait_group_read<0>();
      if (held) ptx::mbar_arrive(held);
      ptx::bulk_wait_group_all();
    }
  } else if (warp >= FIRST_RELAY) {
    if (lane == 0 && smem_ok && rank == 1) relay(warp - FIRST_RELAY + 1);
  } else if (warp >= FIRST_CONV) {
    // ------------------------------------------------------------ converters
    if (smem_ok) {
      int stage = 0; uint32_t phase = 0; bool ok = true;
      auto convert = [&](const MatDev& mt, int l0, int nk, auto zero, auto regular) {
        typedef decltype(zero) T;
        constexpr bool REGULAR = decltype(regular)::value;
        const bool left = mt.left;
        const T* G = static_cast<const T*>(mt.Gs ? mt.Gs : mt.G);
        const long long ld = mt.Gs ? mt.lds : mt.ld;
        const int L = left && mt.Gs ? (int)ld : mt.l;           // (the copies' padding may be read)
        const bool vec = ld * (long long)sizeof(T) % 16 == 0 && reinterpret_cast<unsigned long long>(G) % 16 == 0;
        Slab<T> s[2];
        s[0].template load<REGULAR>(mt, G, ld, L, l0, 0, left, vec);
        s[1].template load<REGULAR>(mt, G, ld, L, l0, min(1, nk - 1) * PK, left, vec);
#pragma unroll 1
        for (int k = 0; k < nk; k += 2) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (k + h >= nk) break;
            if (!ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->empty[stage]), phase ^ 1u, abort_flag)) { ok = false; return; }
            s[h].store(smem + stage * SLAB_BYTES, left);
            ptx::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(rank ? &ctl->converted[stage] : &ctl->full[stage]));
            s[h].template load<REGULAR>(mt, G, ld, L, l0, min(k + h + 2, nk - 1) * PK, left, vec);   // (at the end the last once more)
            if (++stage == STAGES) { stage = 0; phase ^= 1u; }
          }
        }
      };
      for (int t = pair; t < count && ok; t += npairs) {
        const TileDev d = load_tile(tiles + t);
        const MatDev& mt = mats[jobs[d.job].mat];
        const int l0 = d.l0 + PM / 2 * (int)rank;
        const int es = mt.bf16 ? 2 : 4;
        const bool regular = mt.d % PK == 0 && (mt.Gs || (mt.ld * es % 16 == 0 && reinterpret_cast<unsigned long long>(mt.G) % 16 == 0 &&
                                                         (!mt.left || mt.l % 8 == 0)));
        if (mt.bf16) {
          if (regular) convert(mt, l0, d.nk, __nv_bfloat16(), std::true_type()); else convert(mt, l0, d.nk, __nv_bfloat16(), std::false_type());
        } else {
          if (regular) convert(mt, l0, d.nk, float(), std::true_type()); else convert(mt, l0, d.nk, float(), std::false_type());
        }
      }
    }
  } else if (smem_ok) {
    // ------------------------------------------------------------ epilogue
    const int g = (warp - 2) >> 2;                      // group: half of the tile's columns
    const int quarter = warp & 3, c0 = g * (PN / 2);    // TMEM lanes 32 * quarter .. + 31
    const int row = 32 * quarter + lane;
    int out = 0;
    uint32_t ophase = 0;
    const uint32_t tmem = ctl->tmem_base + ((uint32_t)(quarter * 32) << 16) + c0;
    const uint32_t me[2] = {ptx::map_to_cta(ptx::smem_u32(&ctl->main_empty[0]), 0), ptx::map_to_cta(ptx::smem_u32(&ctl->main_empty[1]), 0)};
    const uint32_t se[2] = {ptx::map_to_cta(ptx::smem_u32(&ctl->small_empty[0]), 0), ptx::map_to_cta(ptx::smem_u32(&ctl->small_empty[1]), 0)};
    int piece = 0, tile = 0;
    bool ok = true;
    for (int t = pair; t < count && ok; t += npairs, ++tile) {
      const TileDev d = load_tile(tiles + t);
      const ProjJob& jb = jobs[d.job];
      const int npieces = (d.nk + PROMOTE_SLABS - 1) / PROMOTE_SLABS, R = mats[jb.mat].r;
      float r[PN / 2];
#pragma unroll
      for (int e = 0; e < PN / 2; ++e) r[e] = 0.f;
      for (int p = 0; p < npieces; ++p, ++piece) {
        const int mb = piece & 1;
        if (!ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->main_full[mb]), (piece >> 1) & 1, abort_flag)) { ok = false; break; }
        ptx::tc_fence_after();
        add_columns(r, tmem + mb * PN);
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive_cluster(me[mb]);
      }
      if (!ok) break;
      if ((jb.shape & 15) != 5) add_columns(r, tmem + 2 * PN + (tile & 1) * PN);      // G and the projection have more than one part
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive_cluster(se[tile & 1]);
#pragma unroll
      for (int b = 0; b < BOXES; ++b) {
        if (d.j0 + c0 + COLS * b >= R) break;
        if (!ptx::mbar_wait(ptx::smem_u32(&ctl->oempty[g][out]), ophase ^ 1u, abort_flag)) { ok = false; break; }
        unsigned char* o = boxes + g * GROUP_BYTES + out * OUT_BUF + row * (COLS * 2);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t hi[4], mid[4], lo[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) split::split3(r[COLS * b + 8 * h + 2 * i], r[COLS * b + 8 * h + 2 * i + 1], hi[i], mid[i], lo[i]);
          *reinterpret_cast<uint4*>(o + 16 * h) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
          *reinterpret_cast<uint4*>(o + OUT_PART + 16 * h) = make_uint4(mid[0], mid[1], mid[2], mid[3]);
          *reinterpret_cast<uint4*>(o + 2 * OUT_PART + 16 * h) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        }
        ptx::fence_proxy_async_smem();
        ptx::mbar_arrive(ptx::smem_u32(&ctl->oready[g][out]));
        if (++out == OUT_BUFS) { out = 0; ophase ^= 1u; }
      }
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

int prepared_sms() {
  static std::atomic<int> sms_of_device[64];    // (the shared-memory limit is a per-device setting)
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess && (dev < 0 || dev >= 64)) e = cudaErrorInvalidDevice;
  if (e == cudaSuccess && (sms = sms_of_device[dev].load()) == 0) {
    e = cudaFuncSetAttribute(k_part_project, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_BYTES);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) sms_of_device[dev].store(sms);
  }
  if (e != cudaSuccess) { set_error(std::string("step projection: ") + cudaGetErrorString(e)); return 0; }
  return sms;
}

}  // namespace

size_t part_project_table_bytes(int njobs, int ntiles) {
  return align_up(sizeof(ProjJob) * (size_t)njobs) + align_up(sizeof(TileDev) * (size_t)ntiles);
}

fira_status part_project_prepare(const std::vector<MatDev>& mats, const std::vector<int>& list, char* table_dev, PartStepPlan* plan, cudaStream_t st) {
  std::vector<ProjJob> jd(list.size());
  std::vector<TileDev> td;
  plan->proj_start.assign(1, 0);
  for (size_t q = 0; q < list.size(); ++q) {
    const MatDev& mt = mats[list[q]];
    PartMatrix pi;
    pi.base = mt.Pp; pi.rows = mt.d; pi.cols = mt.r; pi.pitch = mt.pp_pitch; pi.part_stride = (long long)mt.d * mt.pp_pitch; pi.parts = mt.bf16 ? 1 : 3;
    ProjJob j;
    memset(&j, 0, sizeof(j));
    if (!encode_operand(&j.b, pi, true, PN / 2)) return FIRA_ERR_CUDA;
    {
      const unsigned long long extent[3] = {(unsigned long long)mt.r, (unsigned long long)mt.l, 3};
      const unsigned long long pstride[2] = {2ull * mt.rp_pitch, 2ull * mt.l * mt.rp_pitch};
      const unsigned box[3] = {COLS, PM / 2, 3};
      if (!encode_tiled(&j.ro, mt.Rp, false, 3, extent, pstride, box, 0))
        return FIRA_ERR_CUDA;
    }
    j.mat = list[q];
    j.shape = pi.parts | (pi.parts << 2) | (mt.left ? 16 : 0);
    memcpy(&jd[q], &j, sizeof(j));
    // the tiles of one range of l are neighbours: they share G in L2
    for (int l0 = 0; l0 < mt.l; l0 += PM)
      for (int j0 = 0; j0 < mt.r; j0 += PN) td.push_back(TileDev{(int)q, l0, j0, (mt.d + PK - 1) / PK});
    plan->proj_start.push_back((int)td.size());
  }
  plan->proj_table = table_dev; plan->njobs = (int)list.size();
  cudaError_t e = cudaMemcpyAsync(table_dev, jd.data(), sizeof(ProjJob) * jd.size(), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(table_dev + align_up(sizeof(ProjJob) * jd.size()), td.data(), sizeof(TileDev) * td.size(), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) { set_error(std::string("step projection, tables: ") + cudaGetErrorString(e)); return FIRA_ERR_CUDA; }
  return FIRA_OK;
}

fira_status part_project_run(const PartStepPlan& plan, const MatDev* mats_dev, int qa, int qb, unsigned* status_dev, cudaStream_t st) {
  const int sms = prepared_sms();
  if (!sms) return FIRA_ERR_CUDA;
  const int first = plan.proj_start[qa], count = plan.proj_start[qb] - first;
  if (count == 0) return FIRA_OK;
  const ProjJob* jobs = reinterpret_cast<const ProjJob*>(plan.proj_table);
  const TileDev* tiles = reinterpret_cast<const TileDev*>(plan.proj_table + align_up(sizeof(ProjJob) * (size_t)plan.njobs)) + first;
  // (chained: behind k_split_projection)
  const cudaError_t e = launch_chained(k_part_project, 2 * std::min(count, sms / 2), THREADS, SMEM_BYTES, st, true, 1, jobs, tiles, count, mats_dev, status_dev);
  if (e != cudaSuccess) { set_error(std::string("step projection: ") + cudaGetErrorString(e)); return FIRA_ERR_CUDA; }
  return FIRA_OK;
}

}  // namespace fira
