// Tile product with fp32 precision on the tensor cores: a block of 256 threads computes a 128 x 128
// tile of C = A B with arbitrary element strides for both operands (one of an operand's two strides
// is 1), fp32 or bf16 elements.  Used by the fp32 step kernels and by the projection refresh.
//
// An fp32 number is the sum of three bf16 numbers, x = h + m + l, exactly (24 bits = 3 x 8): h = x
// rounded to bf16, m = x - h rounded, l what is left.  So A B is a sum of products of bf16 matrices,
// each exact in the tensor core's multipliers; of the nine the six (h h, h m, m h, h l, l h, m m) are
// taken, what is dropped (m l, l m, l l) is below 2^-26 |a| |b|, an eighth of an fp32 rounding.  A bf16
// operand has one part: three products against an fp32 one, one product against a bf16 one.
//
// The accumulators in tensor memory are fp32, but an MMA adds to them by truncation, and a long chain
// of truncations drifts towards zero.  Hence h h and the small products go to two accumulators, and h h
// is added to fp32 sums in registers (to nearest) every PROMOTE of k: at most 8 truncated additions of
// the main product follow one another (every product of the fp32-precision paths keeps to that).  Measured against
// fp64, relative to the result's norm, at k = 128 / 256 / 512 / 1024: 1.0e-7 throughout for Gaussian operands, 1.2e-7 to 1.4e-7
// for positive ones, against 2.0e-7 / 2.7e-7 / 3.7e-7 / 5.3e-7 and 1.7e-7 / 2.4e-7 / 3.3e-7 / 4.7e-7 of the chain of fp32
// multiply-adds on the CUDA cores that this replaces.  (One accumulator for all of k: 4.1e-7 and 6.8e-7 at 512, 8.8e-7
// and 1.8e-6 at 1024.)
//
// What bounds it: shared memory.  A k-slab of 32 is read once from global memory and split by all
// threads (about 3.5 integer-pipe instructions per element), written as 6 x 8 KiB and read 6 times 2 x
// 8 KiB by the MMAs, which is 1100 to 1200 cycles at 128 bytes per clock against 768 cycles of the
// tensor pipe; the same slab took 4096 cycles as FFMA.  Two blocks per SM: one block's epilogue and
// global latency overlap the other's products; two slabs of shared memory per block overlap its own.
#pragma once
#include "common.cuh"
#include "tc_ptx.cuh"

namespace fira {
namespace split {

constexpr int TILE = 128;                       // rows and columns of a tile
constexpr int BK = 32;                          // k per slab
constexpr int THREADS = 256;
constexpr int PROMOTE = 128;                    // k after which the main accumulator goes to registers
constexpr int STAGES = 2;
constexpr int UNITS = TILE * BK / 8 / THREADS;  // units (8 elements that are neighbours in memory) per thread
// Shared-memory layout of one bf16 part of an operand (no swizzle; 8 x 16-byte core matrices):
//   k contiguous in memory: unit (x, k / 8) at (k / 8) * K_LBO + x * 16
//   x contiguous in memory: unit (x / 8, k) at (x / 8) * X_SBO + k * 16
// The pads make the eight lanes of a 16-byte store phase hit different banks.
constexpr int K_LBO = TILE * 16 + 32;
constexpr int X_SBO = BK * 16 + 16;
constexpr int PART_BYTES = (TILE / 8) * X_SBO;
static_assert(PART_BYTES >= (BK / 8) * K_LBO, "both layouts fit a part");
constexpr int OPERAND_BYTES = 3 * PART_BYTES;
constexpr int STAGE_BYTES = 2 * OPERAND_BYTES;
constexpr int C_LD = TILE + 4;                  // row pitch (floats) of the finished tile in shared memory
static_assert(TILE * C_LD * 4 <= STAGES * STAGE_BYTES, "the finished tile takes the slabs' place");
constexpr int TMEM_COLS = 2 * TILE;             // main and small products

struct Ctl {
  uint64_t done[STAGES];                        // the MMAs that read a slab are done
  uint32_t tmem_base;
  int abort_flag;
  float red[THREADS / 32];
  float bias;                                   // (k_project)
};
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + (int)sizeof(Ctl);
static_assert(2 * (SMEM_BYTES + 1024) <= 228 * 1024, "two blocks per SM");

// x and y as three packed pairs of bf16.
__device__ __forceinline__ void split3(float x, float y, uint32_t& h, uint32_t& m, uint32_t& l) {
  const __nv_bfloat162 hp = __floats2bfloat162_rn(x, y);
  h = *reinterpret_cast<const uint32_t*>(&hp);
  x -= __uint_as_float(h << 16);
  y -= __uint_as_float(h & 0xffff0000u);
  const __nv_bfloat162 mp = __floats2bfloat162_rn(x, y);
  m = *reinterpret_cast<const uint32_t*>(&mp);
  x -= __uint_as_float(m << 16);
  y -= __uint_as_float(m & 0xffff0000u);
  const __nv_bfloat162 lp = __floats2bfloat162_rn(x, y);
  l = *reinterpret_cast<const uint32_t*>(&lp);
}

// Eight neighbouring elements in registers.
template <typename T> struct Frag;
template <> struct Frag<float> { float v[8]; };
template <> struct Frag<__nv_bfloat16> { uint4 u; };

// All eight, from an aligned address, unconditionally: a load in a branch is waited for at the branch's end.
__device__ __forceinline__ void load_frag(const float* p, Frag<float>& f) {
  const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
  f.v[0] = a.x; f.v[1] = a.y; f.v[2] = a.z; f.v[3] = a.w;
  f.v[4] = b.x; f.v[5] = b.y; f.v[6] = b.z; f.v[7] = b.w;
}
__device__ __forceinline__ void load_frag(const __nv_bfloat16* p, Frag<__nv_bfloat16>& f) {
  f.u = *reinterpret_cast<const uint4*>(p);
}
// n (>= 0) of the eight elements exist, the others are zeros.
__device__ __forceinline__ void load_frag(const float* p, int n, bool vec, Frag<float>& f) {
  if (vec && n >= 8) {
    load_frag(p, f);
  } else {
#pragma unroll
    for (int e = 0; e < 8; ++e) f.v[e] = e < n ? p[e] : 0.f;
  }
}
__device__ __forceinline__ void load_frag(const __nv_bfloat16* p, int n, bool vec, Frag<__nv_bfloat16>& f) {
  if (vec && n >= 8) {
    f.u = *reinterpret_cast<const uint4*>(p);
  } else if (n > 8) {
    // four or five aligned 4-byte words; the fifth also holds element 8, which exists
    const unsigned long long a = reinterpret_cast<unsigned long long>(p);
    const uint32_t* w = reinterpret_cast<const uint32_t*>(a & ~3ull);
    uint32_t x[5];
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = w[i];
    if (a & 2) {
      x[4] = w[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) x[i] = __byte_perm(x[i], x[i + 1], 0x5432);
    }
    f.u = make_uint4(x[0], x[1], x[2], x[3]);
  } else {
    const unsigned short* s = reinterpret_cast<const unsigned short*>(p);
    uint32_t x[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      x[i] = (2 * i < n ? (uint32_t)s[2 * i] : 0u) | (2 * i + 1 < n ? (uint32_t)s[2 * i + 1] << 16 : 0u);
    f.u = make_uint4(x[0], x[1], x[2], x[3]);
  }
}
__device__ __forceinline__ void store_parts(unsigned char* p, const Frag<float>& f, long long part_bytes = PART_BYTES) {
  uint32_t h[4], m[4], l[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) split3(f.v[2 * i], f.v[2 * i + 1], h[i], m[i], l[i]);
  *reinterpret_cast<uint4*>(p) = make_uint4(h[0], h[1], h[2], h[3]);
  *reinterpret_cast<uint4*>(p + part_bytes) = make_uint4(m[0], m[1], m[2], m[3]);
  *reinterpret_cast<uint4*>(p + 2 * part_bytes) = make_uint4(l[0], l[1], l[2], l[3]);
}
__device__ __forceinline__ void store_parts(unsigned char* p, const Frag<__nv_bfloat16>& f, long long = 0) {
  *reinterpret_cast<uint4*>(p) = f.u;
}

// Rows [x0, x0 + 128) of an operand Op(x, k) = base[x * sx + k * sk], zero outside X x K.
template <typename T>
struct Operand {
  static constexpr int PARTS = sizeof(T) == 4 ? 3 : 1;
  const T* base;
  long long ld;                                 // the stride that is not 1
  int X, K, x0;
  bool along_x, vec;
  Frag<T> f[UNITS];

  __device__ __forceinline__ Operand(const T* b, long long sx, long long sk, int X_, int K_, int x0_) {
    base = b; X = X_; K = K_; x0 = x0_;
    along_x = sx == 1;
    ld = along_x ? sk : sx;
    vec = ld * (long long)sizeof(T) % 16 == 0 && reinterpret_cast<unsigned long long>(b) % 16 == 0;
  }
  __device__ __forceinline__ void coords(int u, int& x, int& k) const {
    const int e = threadIdx.x + THREADS * u;
    if (along_x) { x = e % (TILE / 8) * 8; k = e / (TILE / 8); } else { k = e % (BK / 8) * 8; x = e / (BK / 8); }
  }
  // Whether every slab's loads are whole aligned units; rows past the matrix then read its last ones again, for rows of the
  // result that nobody looks at.
  __device__ __forceinline__ bool regular() const { return vec && (!along_x || X % 8 == 0) && K % BK == 0; }
  template <bool REGULAR>
  __device__ __forceinline__ void load(int k0) {
#pragma unroll
    for (int u = 0; u < UNITS; ++u) {
      int x, k;
      coords(u, x, k);
      x += x0; k += k0;
      if (REGULAR) {
        x = min(x, along_x ? X - 8 : X - 1);
        load_frag(base + (along_x ? (long long)k * ld + x : (long long)x * ld + k), f[u]);
        continue;
      }
      const int n = along_x ? (k < K ? X - x : 0) : (x < X ? K - k : 0);
      load_frag(base + (along_x ? (long long)k * ld + x : (long long)x * ld + k), n, vec, f[u]);
    }
  }
  __device__ __forceinline__ void store(unsigned char* part) const {
#pragma unroll
    for (int u = 0; u < UNITS; ++u) {
      int x, k;
      coords(u, x, k);
      store_parts(part + (along_x ? (x / 8) * X_SBO + k * 16 : (k / 8) * K_LBO + x * 16), f[u]);
    }
  }
};

// The operand a N - c_x R (rows x, k contiguous), formed between load and store.
struct CombinedOperand {
  static constexpr int PARTS = 3;
  static constexpr bool along_x = false;
  Operand<float> n, r;
  float a, c[UNITS];

  // c_x = c factor[x]
  __device__ __forceinline__ CombinedOperand(const float* N, const float* R, long long ld, int X, int K, int x0,
                                             const float* factor, float a_, float c_)
      : n(N, ld, 1, X, K, x0), r(R, ld, 1, X, K, x0), a(a_) {
    n.along_x = r.along_x = false;              // (a pitch of 1 would count as x contiguous)
    n.ld = r.ld = ld;
#pragma unroll
    for (int u = 0; u < UNITS; ++u) {
      int x, k;
      n.coords(u, x, k);
      c[u] = x0 + x < X ? c_ * factor[x0 + x] : 0.f;
    }
  }
  __device__ __forceinline__ bool regular() const { return n.regular() && r.regular(); }
  template <bool REGULAR>
  __device__ __forceinline__ void load(int k0) {
    n.template load<REGULAR>(k0);
    r.template load<REGULAR>(k0);
  }
  __device__ __forceinline__ void store(unsigned char* part) const {
#pragma unroll
    for (int u = 0; u < UNITS; ++u) {
      int x, k;
      n.coords(u, x, k);
      Frag<float> f;
#pragma unroll
      for (int e = 0; e < 8; ++e) f.v[e] = a * n.f[u].v[e] - c[u] * r.f[u].v[e];
      store_parts(part + (k / 8) * K_LBO + x * 16, f);
    }
  }
};

// Barriers and tensor memory of the block; every thread calls it once.
__device__ __forceinline__ void begin(Ctl* ctl) {
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) ptx::mbar_init(ptx::smem_u32(&ctl->done[s]), 1);
    ctl->abort_flag = 0;
    ptx::fence_barrier_init();
  }
  if (threadIdx.x < 32) {
    ptx::tmem_alloc(ptx::smem_u32(&ctl->tmem_base), TMEM_COLS);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
}
__device__ __forceinline__ void end(Ctl* ctl, unsigned* status) {
  ptx::tc_fence_before();
  __syncthreads();
  if (threadIdx.x < 32) {
    __syncwarp();
    ptx::tc_fence_after();
    ptx::tmem_dealloc(ctl->tmem_base, TMEM_COLS);
  }
  if (threadIdx.x == 0 && ctl->abort_flag) atomicOr(status, DEV_STATUS_TIMEOUT);
}

// MMAs of one slab (A's and B's place), issued by one thread: `steps` of 16 along k, the main product into column 0 of the
// block's tensor memory, the small ones behind it.
template <int PA, int PB, bool A_X, bool B_X>
__device__ __forceinline__ void issue_slab(uint32_t tmem, uint32_t slab_a, uint32_t slab_b, int n, int steps, bool first, bool fresh_main) {
  const uint32_t idesc = ptx::make_idesc_bf16(TILE, n, A_X, B_X);
  constexpr uint64_t along_x = ptx::smem_desc_constant(ptx::LAYOUT_PLAIN, 128, X_SBO);
  constexpr uint64_t along_k = ptx::smem_desc_constant(ptx::LAYOUT_PLAIN, K_LBO, 128);
  constexpr int a_step = (A_X ? 256 : 2 * K_LBO) / 16, b_step = (B_X ? 256 : 2 * K_LBO) / 16;
  slab_a &= 0x3ffff; slab_b &= 0x3ffff;         // (in a cluster the address carries the block's rank above the descriptor's field)
  uint64_t a = (A_X ? along_x : along_k) + (slab_a >> 4), b = (B_X ? along_x : along_k) + (slab_b >> 4);
  uint32_t acc_main = !fresh_main, acc = !first;
  for (int k = 0; k < steps; ++k, a += a_step, b += b_step) {
    ptx::umma_bf16(tmem, a, b, idesc, acc_main);
#pragma unroll
    for (int s = 2; s >= 1; --s)                // i + j = 2, then 1: the smallest first
#pragma unroll
      for (int i = 0; i <= s; ++i)
        if (i < PA && s - i < PB) {
          ptx::umma_bf16(tmem + TILE, a + i * (PART_BYTES / 16), b + (s - i) * (PART_BYTES / 16), idesc, acc);
          acc = 1;
        }
    acc_main = 1;
  }
}
template <int PA, int PB>
__device__ __forceinline__ void issue_slab(uint32_t tmem, uint32_t slab, bool a_x, bool b_x, int n, int steps, bool first, bool fresh_main) {
  const uint32_t slab_b = slab + OPERAND_BYTES;
  if (a_x) {
    if (b_x) issue_slab<PA, PB, true, true>(tmem, slab, slab_b, n, steps, first, fresh_main);
    else issue_slab<PA, PB, true, false>(tmem, slab, slab_b, n, steps, first, fresh_main);
  } else {
    if (b_x) issue_slab<PA, PB, false, true>(tmem, slab, slab_b, n, steps, first, fresh_main);
    else issue_slab<PA, PB, false, false>(tmem, slab, slab_b, n, steps, first, fresh_main);
  }
}

// The slabs of tile_product: loads one slab ahead, splits, issues; sum: pieces of the main product.
template <bool LONG_K, bool REGULAR, class A, class B, class F>
__device__ __forceinline__ void product_slabs(A& a, B& b, int K, int n, unsigned char* slabs, Ctl* ctl, float (&sum)[LONG_K ? TILE / 2 : 1], const F& meanwhile) {
  const int ns = (K + BK - 1) / BK;
  const int warp = threadIdx.x >> 5, c0 = (warp >> 2) * (TILE / 2);
  const uint32_t tmem = ctl->tmem_base;
  const uint32_t lane_col = tmem + ((uint32_t)((warp & 3) * 32) << 16) + c0;
  bool fresh = true;
  a.template load<REGULAR>(0);
  b.template load<REGULAR>(0);
  meanwhile();
  for (int s = 0; s < ns; ++s) {
    unsigned char* slab = slabs + (s % STAGES) * STAGE_BYTES;
    const uint32_t done = ptx::smem_u32(&ctl->done[s % STAGES]);
    if (s >= STAGES) ptx::mbar_wait(done, (s / STAGES - 1) & 1, &ctl->abort_flag);
    a.store(slab);
    b.store(slab + OPERAND_BYTES);
    ptx::fence_proxy_async_smem();
    const int next = min(s + 1, ns - 1) * BK;   // (the last slab once more, unused)
    a.template load<REGULAR>(next);
    b.template load<REGULAR>(next);
    ptx::tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0) {
      ptx::tc_fence_after();
      issue_slab<A::PARTS, B::PARTS>(tmem, ptx::smem_u32(slab), a.along_x, b.along_x, n,
                                     min(BK, K - s * BK + 15) / 16, s == 0, fresh);
      ptx::umma_commit(done);
    }
    fresh = false;
    if (LONG_K && (s + 1) % (PROMOTE / BK) == 0 && s + 1 < ns) {
      ptx::mbar_wait(done, (s / STAGES) & 1, &ctl->abort_flag);
      ptx::tc_fence_after();
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (c0 + 32 * h < n) {
          uint32_t v[32];
          __syncwarp();
          ptx::tmem_ld_32x32b_x32(lane_col + 32 * h, v);
          ptx::tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 32; ++i) sum[LONG_K ? 32 * h + i : 0] += __uint_as_float(v[i]);
        }
      fresh = true;
    }
  }
}

// The tile A B over k < K into shared memory, row x of A at C[x * C_LD]; ends with a block barrier.
// cols: columns of the tile that are wanted (the others hold garbage).  C overlays the slabs.
// Returns false if a wait ran out (bounded as in tc_ptx.cuh); all threads take the same path even then.
// meanwhile: called by every thread while its first loads are on their way.
struct Nothing { __device__ __forceinline__ void operator()() const {} };
template <bool LONG_K, class A, class B, class F = Nothing>
__device__ __forceinline__ bool tile_product(A& a, B& b, int K, int cols, unsigned char* slabs, Ctl* ctl, const F& meanwhile = F()) {
  constexpr bool SMALL = A::PARTS > 1 || B::PARTS > 1;
  const int n = (min(cols, TILE) + 15) / 16 * 16;
  const int ns = (K + BK - 1) / BK;
  const int warp = threadIdx.x >> 5;
  const uint32_t lane_col = ctl->tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (warp >> 2) * (TILE / 2);
  const int c0 = (warp >> 2) * (TILE / 2);      // this thread: row 32 (warp % 4) + lane, columns c0 .. c0 + 63
  float sum[LONG_K ? TILE / 2 : 1];
  if (LONG_K) {
#pragma unroll
    for (int i = 0; i < TILE / 2; ++i) sum[LONG_K ? i : 0] = 0.f;
  }
  if (a.regular() && b.regular()) product_slabs<LONG_K, true>(a, b, K, n, slabs, ctl, sum, meanwhile);
  else product_slabs<LONG_K, false>(a, b, K, n, slabs, ctl, sum, meanwhile);
  // all MMAs: the last commit covers the earlier ones; nobody overwrites the slabs before everybody has seen it
  const int last = ns - 1;
  const bool ok = ptx::mbar_wait(ptx::smem_u32(&ctl->done[last % STAGES]), (last / STAGES) & 1, &ctl->abort_flag);
  if (__syncthreads_or(!ok || *(volatile int*)&ctl->abort_flag)) return false;
  ptx::tc_fence_after();
  float* C = reinterpret_cast<float*>(slabs) + (32 * (warp & 3) + (threadIdx.x & 31)) * C_LD + c0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {                 // 16 columns at a time
    if (c0 + 16 * q >= n) break;
    uint32_t v[16], w[16];
    __syncwarp();
    ptx::tmem_ld_32x32b_x16(lane_col + 16 * q, v);
    if (SMALL) ptx::tmem_ld_32x32b_x16(lane_col + TILE + 16 * q, w);
    ptx::tmem_ld_wait();
#pragma unroll
    for (int i = 0; i < 16; i += 4) {
      float o[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        o[e] = __uint_as_float(v[i + e]);
        if (LONG_K) o[e] += sum[LONG_K ? 16 * q + i + e : 0];
        if (SMALL) o[e] += __uint_as_float(w[i + e]);
      }
      *reinterpret_cast<float4*>(C + 16 * q + i) = make_float4(o[0], o[1], o[2], o[3]);
    }
  }
  __syncthreads();
  return true;
}

}  // namespace split
}  // namespace fira
