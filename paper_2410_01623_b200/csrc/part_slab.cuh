// Slabs of bf16 parts for CTA pairs: shared by the part products (part_gemm.cu) and the step's products with the
// projection (part_back.cu).  A slab is 32 deep; one TMA box brings all parts of an operand's slab (the part index is the
// outermost dimension of its tensor map), so that a slab takes two TMA instructions per CTA although it holds up to six
// part tiles.
#pragma once
#include "part_gemm.cuh"
#include "tc_ptx.cuh"
#include "tma_encode.cuh"

namespace fira {

constexpr int PM = 256, PN = 128, PK = 32;      // tile of a CTA pair, depth of a slab
constexpr int A_PART = PM / 2 * PK * 2;         // bytes of one part of a slab in one CTA: 8 KiB
constexpr int B_PART = PN / 2 * PK * 2;         // 4 KiB

// MMAs of one slab.  An operand along its rows: 64-element chunks of 32 k-rows (4 KiB), 16 k-rows of 128 bytes per
// step; along k: 64-byte rows.
template <int PA, int PB, bool A_MN, bool B_MN>
__device__ __forceinline__ void issue_slab(uint32_t main, uint32_t small, uint32_t slab, int a_bytes, bool fresh, bool first) {
  constexpr uint64_t mn = ptx::smem_desc_constant(ptx::LAYOUT_SW128, PK * 128, 1024);
  constexpr uint64_t km = ptx::smem_desc_constant(ptx::LAYOUT_SW64, 0, 512);
  const uint32_t idesc = ptx::make_idesc_bf16(PM, PN, A_MN, B_MN);
  uint64_t a = (A_MN ? mn : km) + (slab >> 4), b = (B_MN ? mn : km) + ((slab + a_bytes) >> 4);
  uint32_t acc = !first;
#pragma unroll
  for (int s = 0; s < PK / 16; ++s, a += (A_MN ? 2048 : 32) / 16, b += (B_MN ? 2048 : 32) / 16) {
    ptx::umma_bf16_pair(main, a, b, idesc, s ? 1u : !fresh);
#pragma unroll
    for (int q = 2; q >= 1; --q)
#pragma unroll
      for (int p = 0; p <= q; ++p)
        if (p < PA && q - p < PB) {
          ptx::umma_bf16_pair(small, a + p * (A_PART / 16), b + (q - p) * (B_PART / 16), idesc, acc);
          acc = 1u;
        }
  }
}
template <int PA, int PB>
__device__ __forceinline__ void issue_slab(int shape, uint32_t main, uint32_t small, uint32_t slab, int a_bytes, bool fresh, bool first) {
  if (shape & 16) {
    if (shape & 32) issue_slab<PA, PB, true, false>(main, small, slab, a_bytes, fresh, first);
    else issue_slab<PA, PB, true, true>(main, small, slab, a_bytes, fresh, first);
  } else {
    if (shape & 32) issue_slab<PA, PB, false, false>(main, small, slab, a_bytes, fresh, first);
    else issue_slab<PA, PB, false, true>(main, small, slab, a_bytes, fresh, first);
  }
}
__device__ __forceinline__ void issue_parts(int shape, uint32_t main, uint32_t small, uint32_t slab, int a_bytes, bool fresh, bool first) {
  if ((shape & 15) == 15) issue_slab<3, 3>(shape, main, small, slab, a_bytes, fresh, first);
  else if ((shape & 15) == 13) issue_slab<1, 3>(shape, main, small, slab, a_bytes, fresh, first);
  else if ((shape & 15) == 7) issue_slab<3, 1>(shape, main, small, slab, a_bytes, fresh, first);
  else issue_slab<1, 1>(shape, main, small, slab, a_bytes, fresh, first);
}

// sum += 64 columns of this thread's accumulator row.
__device__ __forceinline__ void add_columns(float (&sum)[64], uint32_t taddr) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t v[32];
    __syncwarp();
    ptx::tmem_ld_32x32b_x32(taddr + 32 * h, v);
    ptx::tmem_ld_wait();
#pragma unroll
    for (int e = 0; e < 32; ++e) sum[32 * h + e] += __uint_as_float(v[e]);
  }
  ptx::tc_fence_before();
  __syncwarp();
}

// Tensor map of an operand: rows_contiguous: its rows (i of A, j of B) are contiguous in memory.
inline bool encode_operand(CUtensorMap* map, const PartMatrix& p, bool rows_contiguous, int rows_box) {
  const unsigned long long pitch = p.pitch * 2, part = p.part_stride * 2;
  if (rows_contiguous) {
    const unsigned long long extent[4] = {64, (unsigned long long)p.rows, (unsigned long long)(p.pitch / 64), (unsigned long long)p.parts};
    const unsigned long long stride[3] = {pitch, 128, part};
    const unsigned box[4] = {64, PK, (unsigned)rows_box / 64, (unsigned)p.parts};
    return encode_tiled(map, p.base, false, 4, extent, stride, box, 128);
  }
  const unsigned long long extent[3] = {(unsigned long long)p.cols, (unsigned long long)p.rows, (unsigned long long)p.parts};
  const unsigned long long stride[2] = {pitch, part};
  const unsigned box[3] = {PK, (unsigned)rows_box, (unsigned)p.parts};
  return encode_tiled(map, p.base, false, 3, extent, stride, box, 64);
}

}  // namespace fira
