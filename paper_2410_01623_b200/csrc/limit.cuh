// The limiter (Eq. 12 in Algorithm 1's form) inside kernels whose blocks hold a matrix's residual while they wait for its norm.
#pragma once
#include "common.cuh"
#include "tc_ptx.cuh"

namespace fira {

// What a matrix's tiles need to know of its norm: lambda, times the matrix's one factor if it has one.  By one warp of every block
// (or pair) that has a tile of it, all of them with the same result: they wait for the shares themselves, marked words (SHARE: a float or
// a double per tile, of the width that the tile's own sums have been added in), which a kernel before has zeroed.  (Counting the tiles and having the last
// one publish lambda took 8 us in place of 3: two trips through L2 and two fences more.)
struct Limit { double sum; float kmat, norm, lambda; };

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// prev: the norm remembered before the step.
template <typename SHARE>
__device__ __forceinline__ bool wait_limit(const unsigned long long* shares, int tiles, const MatDev& mt, float prev, const Hyper& hp, volatile int* abort_flag, Limit& out) {
  const int lane = threadIdx.x & 31;
  out.kmat = 1.f;
  if (hp.mode & HYPER_MATRIX_SCALING) {          // Eq. 9: the tiles have worked with factor 1
    double nn = 0.0, rn = 0.0;
#pragma unroll 8
    for (int i = lane; i < mt.l; i += 32) { nn += (double)__ldcg(mt.aux + i); rn += (double)__ldcg(mt.aux + mt.l + i); }
    out.kmat = (float)(sqrt(warp_sum(nn)) / (sqrt(warp_sum(rn)) + (double)hp.eps));
  }
  for (uint32_t it = 0;; ++it) {
    bool there = true;
    double acc = 0.0;
    for (int i = lane; i < tiles; i += 32) {
      SHARE v;
      there = ptx::get_marked(shares + i * (sizeof(SHARE) / sizeof(float)), &v) && there;
      acc += (double)v;
    }
    if (__all_sync(0xffffffffu, there)) { out.sum = warp_sum(acc); break; }
    __nanosleep(it < 64 ? 32 : 256);
    const bool stop = it == (1u << 21) || ((it & 63u) == 63u && *abort_flag);
    if (__any_sync(0xffffffffu, stop)) { *abort_flag = 1; return false; }
  }
  const bool residual = !(hp.mode & HYPER_NO_RESIDUAL);
  out.norm = residual ? out.kmat * (float)sqrt(out.sum > 0.0 ? out.sum : 0.0) : 0.f;
  out.lambda = 1.f;
  if (residual && prev >= 0.f && !isinf(hp.gamma)) {
    const float ratio = out.norm / (prev + hp.eps);
    out.lambda = hp.gamma / fmaxf(ratio, hp.gamma);
  }
  return true;
}
// The matrix's state and diagnostics (as k_finalize leaves them), by one of them.  (No more than that: who is
// late with one tile is late with the next, so that microseconds add up over the matrices.  The next step's bias factor, in double,
// made the kernel take 281 us where it took 166 without.)
__device__ __forceinline__ void store_limit(const MatDev& mt, const Hyper& hp, const Limit& lim, unsigned* status) {
  const int lane = threadIdx.x & 31;
  float kmin = lim.kmat, kmax = lim.kmat;
  if (!(hp.mode & HYPER_MATRIX_SCALING)) {
    kmin = INFINITY; kmax = -INFINITY;
    const int quads = mt.l / 4;                  // (the table is 256-byte aligned)
    for (int q = lane; q < quads; q += 32 * 8) {
      float4 v[8];                               // loads in flight together
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = __ldcg(reinterpret_cast<const float4*>(mt.kvec) + min(q + 32 * e, quads - 1));
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        kmin = fminf(kmin, fminf(fminf(v[e].x, v[e].y), fminf(v[e].z, v[e].w)));
        kmax = fmaxf(kmax, fmaxf(fmaxf(v[e].x, v[e].y), fmaxf(v[e].z, v[e].w)));
      }
    }
    if (4 * quads + lane < mt.l) {
      const float k = __ldcg(mt.kvec + 4 * quads + lane);
      kmin = fminf(kmin, k); kmax = fmaxf(kmax, k);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      kmin = fminf(kmin, __shfl_xor_sync(0xffffffffu, kmin, o));
      kmax = fmaxf(kmax, __shfl_xor_sync(0xffffffffu, kmax, o));
    }
  }
  if (lane == 0) {
    const bool residual = !(hp.mode & HYPER_NO_RESIDUAL);
    MatScalars* sc = mt.sc;
    sc->norm_scaled = lim.norm;
    sc->lambda = lim.lambda;
    if (residual) {
      if (!isfinite((float)lim.sum) || !isfinite(kmax)) atomicOr(status, DEV_STATUS_NONFINITE);
      sc->prev_norm = lim.lambda * lim.norm;
    }
    sc->k_min = residual ? kmin : 0.f;
    sc->k_max = residual ? kmax : 0.f;
    sc->t = sc->t + 1;
  }
}

}  // namespace fira
