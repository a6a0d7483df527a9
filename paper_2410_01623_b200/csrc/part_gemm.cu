// Grouped products in fp32 precision of matrices stored as bf16 parts (part_gemm.cuh) for sm_100a.
//
// CTA pairs (clusters of two, one CTA per SM, persistent over a static tile list) compute 256 x 128 tiles
// with tcgen05.mma.cta_group::2.  A slab is 32 deep; one TMA box brings all parts of an operand's slab
// (the part index is the outermost dimension of its tensor map), so that a slab takes two TMA
// instructions per CTA although it holds up to six part tiles.  An operand that is contiguous along k
// comes as 64-byte rows (64-byte swizzle), one that is contiguous along its rows as 64-element chunks
// (128-byte swizzle): no transposed copy of anything is made.
//
// Tensor memory: the product of the leading parts alternates between two accumulators every PROMOTE of
// k, because MMAs add by truncation and a long chain of them drifts towards zero: the epilogue warps add
// each finished piece to fp32 sums in registers.  The small part products, 2^-8 and less of the result,
// have accumulators of their own, two that alternate between tiles.  4 x 128 columns in all.
//
// What bounds it: the tensor pipe, 12 MMAs of 256 x 128 x 16 per slab (768 cycles), as long as the
// products are long enough to hide the tile's end; shared-memory reads are 96 bytes per clock of 128.
//
// Warp roles: 0 producer (TMA), 1 MMA issuer (even CTA) and owner of the tensor memory, 2-9 epilogue (each
// lane quarter twice, 64 columns each).
#include <string.h>

#include <algorithm>
#include <atomic>
#include <functional>
#include <queue>

#include "part_slab.cuh"
#include "split_gemm.cuh"

namespace fira {

namespace {

constexpr int PG_MAX_STAGES = 12;
constexpr int PG_MAX_PAIRS = 127;               // (so many pairs of SMs at most)
constexpr int PG_PROMOTE = split::PROMOTE / PK; // slabs between two readings of the main accumulator
constexpr int PG_SLAB_BYTES = 216 * 1024;       // for the slabs in flight: 6 of three parts each, 10 of one and three
constexpr int PG_EPI_WARPS = 8;
constexpr int PG_THREADS = 32 * (2 + PG_EPI_WARPS);
constexpr int PG_TMEM = 512;

struct alignas(64) JobDev {
  CUtensorMap a, b;
  float* c;
  __nv_bfloat16* out;
  long long ldc, pitch, part_stride;
  int I, J;
  int shape;                                    // bits 0-1, 2-3: parts of A, B; 4: A transposed, 5: B transposed
};
static_assert(sizeof(JobDev) % 64 == 0, "tensor maps must stay 64-byte aligned");
struct TileDev { int job, i0, j0, nk; };

struct PgCtl {
  uint64_t full[PG_MAX_STAGES], empty[PG_MAX_STAGES];
  uint64_t main_full[2], main_empty[2];         // a piece of the main product is complete / has been read
  uint64_t small_empty[2];                      // the small products of a tile have been read
  uint32_t tmem_base;
  int abort_flag;
};
constexpr size_t PG_SMEM_BYTES = (size_t)PG_SLAB_BYTES + sizeof(PgCtl);
static_assert(PG_SMEM_BYTES <= 227 * 1024, "shared memory budget");

__device__ __forceinline__ TileDev load_tile(const TileDev* t) {
  const int4 v = __ldg(reinterpret_cast<const int4*>(t));
  return TileDev{v.x, v.y, v.z, v.w};
}

__device__ __forceinline__ void store32(void* p, const uint32_t (&v)[8]) {   // 32-byte aligned
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]),
               "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
}

// 64 columns of one row: as fp32, or split into parts.  Whole sectors where the row's pitch allows it.
__device__ __forceinline__ void store_result(const JobDev& jb, int i, int j, const float (&v)[64]) {
  if (jb.c) {
    float* c = jb.c + (long long)i * jb.ldc + j;
    const bool sectors = jb.ldc % 8 == 0 && reinterpret_cast<unsigned long long>(jb.c) % 32 == 0;
#pragma unroll
    for (int q = 0; q < 64; q += 8) {
      if (sectors && j + q + 8 <= jb.J) {
        uint32_t w[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) w[e] = __float_as_uint(v[q + e]);
        store32(c + q, w);
      } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) if (j + q + e < jb.J) c[q + e] = v[q + e];
      }
    }
  } else {
    __nv_bfloat16* o = jb.out + (long long)i * jb.pitch + j;      // (the pitch covers the last 64 columns)
#pragma unroll
    for (int q = 0; q < 64; q += 16) {
      if (j + q >= jb.J) break;
      uint32_t h[8], m[8], l[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) split::split3(v[q + 2 * e], v[q + 2 * e + 1], h[e], m[e], l[e]);
      store32(o + q, h);
      store32(o + jb.part_stride + q, m);
      store32(o + 2 * jb.part_stride + q, l);
    }
  }
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(PG_THREADS, 1)
k_part_gemm(const JobDev* __restrict__ jobs, const int* __restrict__ starts, const TileDev* __restrict__ tiles, int stages,
            int a_bytes, int stage_bytes, unsigned* __restrict__ status) {
  extern __shared__ __align__(1024) unsigned char smem[];
  PgCtl* ctl = reinterpret_cast<PgCtl*>(smem + PG_SLAB_BYTES);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = ptx::cluster_ctarank();
  const int first_tile = starts[blockIdx.x >> 1], end_tile = starts[(blockIdx.x >> 1) + 1];     // this pair's
  const bool smem_ok = (ptx::smem_u32(smem) & 1023u) == 0;
  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      ptx::mbar_init(ptx::smem_u32(&ctl->full[s]), 1);
      ptx::mbar_init(ptx::smem_u32(&ctl->empty[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      ptx::mbar_init(ptx::smem_u32(&ctl->main_full[b]), 1);
      ptx::mbar_init(ptx::smem_u32(&ctl->main_empty[b]), 2 * PG_EPI_WARPS);      // the epilogue warps of both CTAs
      ptx::mbar_init(ptx::smem_u32(&ctl->small_empty[b]), 2 * PG_EPI_WARPS);
    }
    ctl->abort_flag = smem_ok ? 0 : 1;
    ptx::fence_barrier_init();
  }
  if (warp == 1) {
    ptx::tmem_alloc_pair(ptx::smem_u32(&ctl->tmem_base), PG_TMEM);
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

  if (warp == 0) {
    if (lane == 0 && smem_ok) {
      int stage = 0; uint32_t phase = 0; bool ok = true;
      for (int t = first_tile; t < end_tile && ok; ++t) {
        const TileDev d = load_tile(tiles + t);
        const JobDev* jb = jobs + d.job;
        const int shape = jb->shape, pa = shape & 3, pb = (shape >> 2) & 3;
        const int i0 = d.i0 + PM / 2 * (int)rank, j0 = d.j0 + PN / 2 * (int)rank;
        for (int k = 0; k < d.nk; ++k) {
          if (!ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->empty[stage]), phase ^ 1u, abort_flag)) { ok = false; break; }
          const uint32_t fb = ptx::map_to_cta(ptx::smem_u32(&ctl->full[stage]), 0);
          const uint32_t sa = slabs + stage * stage_bytes, sb = sa + a_bytes;
          if (rank == 0) ptx::mbar_expect_tx(ptx::smem_u32(&ctl->full[stage]), 2 * (pa * A_PART + pb * B_PART));
          if (shape & 16) ptx::tma_load_4d_pair(sa, &jb->a, fb, 0, k * PK, i0 >> 6, 0);
          else ptx::tma_load_3d_pair(sa, &jb->a, fb, k * PK, i0, 0);
          if (shape & 32) ptx::tma_load_3d_pair(sb, &jb->b, fb, k * PK, j0, 0);
          else ptx::tma_load_4d_pair(sb, &jb->b, fb, 0, k * PK, j0 >> 6, 0);
          if (++stage == stages) { stage = 0; phase ^= 1u; }
        }
      }
      if (!ok && rank == 0) {   // give copies in flight a bounded time to land
        for (int s = 0; s < stages; ++s)
          for (uint32_t it = 0; it < (1u << 16); ++it)
            if (ptx::mbar_try_wait_cluster(ptx::smem_u32(&ctl->full[s]), (s < stage) ? phase : (phase ^ 1u))) break;
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && smem_ok && rank == 0) {
      int stage = 0; uint32_t phase = 0; bool ok = true;
      int piece = 0, tile = 0;                  // running numbers of the main accumulator's uses and of the tiles
      const uint32_t tmem = ctl->tmem_base;
      for (int t = first_tile; t < end_tile && ok; ++t) {
        const TileDev d = load_tile(tiles + t);
        const int shape = jobs[d.job].shape;
        const uint32_t small = tmem + 2 * PN + (tile & 1) * PN;
        if (!ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->small_empty[tile & 1]), ((tile >> 1) & 1) ^ 1u, abort_flag)) break;
        for (int k = 0; k < d.nk; ++k) {
          const int mb = piece & 1;
          const bool fresh = k % PG_PROMOTE == 0;
          if (fresh && !ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->main_empty[mb]), ((piece >> 1) & 1) ^ 1u, abort_flag)) { ok = false; break; }
          if (!ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->full[stage]), phase, abort_flag)) { ok = false; break; }
          ptx::tc_fence_after();
          issue_parts(shape, tmem + mb * PN, small, slabs + stage * stage_bytes, a_bytes, fresh, k == 0);
          ptx::umma_commit_pair(ptx::smem_u32(&ctl->empty[stage]), 3);
          if (++stage == stages) { stage = 0; phase ^= 1u; }
          if ((k + 1) % PG_PROMOTE == 0 || k + 1 == d.nk) {      // (covers the small products so far as well)
            ptx::umma_commit_pair(ptx::smem_u32(&ctl->main_full[mb]), 3);
            ++piece;
          }
        }
        ++tile;
      }
    }
  } else if (smem_ok) {
    const int quarter = warp & 3, c0 = ((warp - 2) >> 2) * 64;
    const uint32_t lanes = (uint32_t)(quarter * 32) << 16;
    const uint32_t tmem = ctl->tmem_base + lanes + c0;
    const uint32_t me[2] = {ptx::map_to_cta(ptx::smem_u32(&ctl->main_empty[0]), 0), ptx::map_to_cta(ptx::smem_u32(&ctl->main_empty[1]), 0)};
    const uint32_t se[2] = {ptx::map_to_cta(ptx::smem_u32(&ctl->small_empty[0]), 0), ptx::map_to_cta(ptx::smem_u32(&ctl->small_empty[1]), 0)};
    int piece = 0, tile = 0;
    bool ok = true;
    for (int t = first_tile; t < end_tile && ok; ++t) {
      const TileDev d = load_tile(tiles + t);
      const JobDev& jb = jobs[d.job];
      float sum[64];                            // this thread's row of the product, columns c0 .. c0 + 63
#pragma unroll
      for (int e = 0; e < 64; ++e) sum[e] = 0.f;
      const int npieces = (d.nk + PG_PROMOTE - 1) / PG_PROMOTE;
      for (int p = 0; p < npieces; ++p, ++piece) {
        const int mb = piece & 1;
        if (!ptx::mbar_wait_cluster(ptx::smem_u32(&ctl->main_full[mb]), (piece >> 1) & 1, abort_flag)) { ok = false; break; }
        ptx::tc_fence_after();
        add_columns(sum, tmem + mb * PN);
        if (lane == 0) ptx::mbar_arrive_cluster(me[mb]);
      }
      if (!ok) break;
      if ((jb.shape & 15) != 5) add_columns(sum, tmem + 2 * PN + (tile & 1) * PN);    // some operand has more than one part
      if (lane == 0) ptx::mbar_arrive_cluster(se[tile & 1]);
      ++tile;
      const int i = d.i0 + PM / 2 * (int)rank + 32 * quarter + lane;
      if (i < jb.I && d.j0 + c0 < jb.J) store_result(jb, i, d.j0 + c0, sum);
    }
  }
  // neither CTA may leave while its partner can still reach into its shared memory
  ptx::tc_fence_before();
  __syncthreads();
  ptx::cluster_sync_all();
  if (warp == 1) {
    __syncwarp();
    ptx::tc_fence_after();
    ptx::tmem_dealloc_pair(ctl->tmem_base, PG_TMEM);
  }
  if (threadIdx.x == 0 && ctl->abort_flag) atomicOr(status, DEV_STATUS_TIMEOUT);
}

long long depth_of(const PartGemm& g) { return g.a_t ? g.a.rows : g.a.cols; }

// The tiles of a row of tiles are neighbours (they share the rows of A in L2), forth and back in turn: where B is
// triangular their lengths differ, and every pair gets some of each.
void tiles_of(const PartGemm& g, int job, std::vector<TileDev>& out) {
  const long long I = g.a_t ? g.a.cols : g.a.rows, K = depth_of(g), J = g.b_t ? g.b.rows : g.b.cols;
  const int nj = (int)((J + PN - 1) / PN);
  for (int i0 = 0, row = 0; i0 < I; i0 += PM, ++row)
    for (int q = 0; q < nj; ++q) {
      const int j0 = (row % 2 ? nj - 1 - q : q) * PN;
      if (g.lower && j0 >= i0 + PM) continue;
      const long long k = g.upper_b ? std::min<long long>(K, j0 + PN) : K;
      out.push_back(TileDev{job, i0, j0, (int)((k + PK - 1) / PK)});
    }
}

}  // namespace

// SMs of the current device (0: error) once the kernel may use its shared memory there.
static int prepared_sms() {
  static std::atomic<int> sms_of_device[64];    // (the shared-memory limit is a per-device setting)
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess && (dev < 0 || dev >= 64)) e = cudaErrorInvalidDevice;
  if (e == cudaSuccess && (sms = sms_of_device[dev].load()) == 0) {
    e = cudaFuncSetAttribute(k_part_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PG_SMEM_BYTES);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) sms_of_device[dev].store(sms);
  }
  if (e != cudaSuccess) { set_error(std::string("part products: ") + cudaGetErrorString(e)); return 0; }
  return sms;
}

// Deals the tiles out to `pairs` CTA pairs, in order (neighbours run side by side), each to the pair with the least work
// so far; pair p gets those at starts[p] .. starts[p + 1] of the result.  A tile's end costs about as much as two slabs.
static std::vector<TileDev> deal(const std::vector<TileDev>& tiles, int pairs, std::vector<int>& starts) {
  typedef std::pair<long long, int> Load;
  std::priority_queue<Load, std::vector<Load>, std::greater<Load>> load;
  for (int p = 0; p < pairs; ++p) load.push({0, p});
  std::vector<std::vector<TileDev>> of((size_t)pairs);
  for (const TileDev& t : tiles) {
    const Load l = load.top();
    load.pop();
    of[l.second].push_back(t);
    load.push({l.first + t.nk + 2, l.second});
  }
  std::vector<TileDev> out;
  starts.assign(1, 0);
  for (const auto& v : of) {
    out.insert(out.end(), v.begin(), v.end());
    starts.push_back((int)out.size());
  }
  return out;
}

static size_t starts_bytes() { return align_up((PG_MAX_PAIRS + 1) * sizeof(int)); }

size_t part_gemm_table_bytes(const PartGemm* jobs, int njobs) {
  std::vector<TileDev> t;
  for (int q = 0; q < njobs; ++q) tiles_of(jobs[q], q, t);
  return align_up(sizeof(JobDev) * (size_t)njobs) + starts_bytes() + align_up(sizeof(TileDev) * t.size());
}

fira_status part_gemm_prepare(const PartGemm* jobs, int njobs, char* table_dev, size_t table_bytes, int* ntiles, cudaStream_t st) {
  std::vector<JobDev> jd((size_t)njobs);
  std::vector<TileDev> td;
  for (int q = 0; q < njobs; ++q) {
    const PartGemm& g = jobs[q];
    JobDev& j = jd[q];
    memset(&j, 0, sizeof(j));
    if (!encode_operand(&j.a, g.a, g.a_t, PM / 2) || !encode_operand(&j.b, g.b, !g.b_t, PN / 2)) return FIRA_ERR_CUDA;
    j.c = g.c; j.ldc = g.ldc;
    j.out = g.out.base; j.pitch = g.out.pitch; j.part_stride = g.out.part_stride;
    j.I = (int)(g.a_t ? g.a.cols : g.a.rows); j.J = (int)(g.b_t ? g.b.rows : g.b.cols);
    j.shape = g.a.parts | (g.b.parts << 2) | (g.a_t ? 16 : 0) | (g.b_t ? 32 : 0);
  }
  // the matrices with the longest products first: what is left over at the end of the list is short
  std::vector<int> order((size_t)njobs);
  for (int q = 0; q < njobs; ++q) order[q] = q;
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return depth_of(jobs[x]) > depth_of(jobs[y]); });
  for (int q : order) tiles_of(jobs[q], q, td);
  const int sms = prepared_sms();
  if (!sms) return FIRA_ERR_CUDA;
  *ntiles = (int)td.size();
  std::vector<int> starts;
  td = deal(td, std::min(*ntiles, sms / 2), starts);
  const size_t o_starts = align_up(sizeof(JobDev) * (size_t)njobs), o_tiles = o_starts + starts_bytes();
  if (starts.size() > PG_MAX_PAIRS + 1 || o_tiles + align_up(sizeof(TileDev) * td.size()) > table_bytes) {
    set_error("part products: table area too small"); return FIRA_ERR_WORKSPACE_TOO_SMALL;
  }
  cudaError_t e = cudaMemcpyAsync(table_dev, jd.data(), sizeof(JobDev) * jd.size(), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(table_dev + o_starts, starts.data(), sizeof(int) * starts.size(), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(table_dev + o_tiles, td.data(), sizeof(TileDev) * td.size(), cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) { set_error(std::string("part products, tables: ") + cudaGetErrorString(e)); return FIRA_ERR_CUDA; }
  return FIRA_OK;
}

fira_status part_gemm_run(const char* table_dev, int njobs, int ntiles, int a_parts, int b_parts, unsigned* status_dev, cudaStream_t st) {
  const int sms = prepared_sms();
  if (!sms) return FIRA_ERR_CUDA;
  if (ntiles == 0) return FIRA_OK;
  const int a_bytes = a_parts * A_PART, stage_bytes = a_bytes + b_parts * B_PART;
  const char* starts = table_dev + align_up(sizeof(JobDev) * (size_t)njobs);
  const cudaError_t e = launch_chained(
      k_part_gemm, 2 * std::min(ntiles, sms / 2), PG_THREADS, PG_SMEM_BYTES, st, true, 1, reinterpret_cast<const JobDev*>(table_dev), reinterpret_cast<const int*>(starts),
      reinterpret_cast<const TileDev*>(starts + starts_bytes()), std::min(PG_MAX_STAGES, PG_SLAB_BYTES / stage_bytes), a_bytes,
      stage_bytes, status_dev);
  if (e != cudaSuccess) { set_error(std::string("part product: ") + cudaGetErrorString(e)); return FIRA_ERR_CUDA; }
  return FIRA_OK;
}

}  // namespace fira
