// U = L^-T of C = L L^T (r x r, fp32, the lower triangle of C given), for all matrices of a chunk at once.
// Included by refresh.cu inside its namespace.
//
// Blocked over columns of NB = 128, three launches per block column J, each over every matrix:
//   k_factor_block   one block per matrix: factors C[J, J] and inverts the factor in registers; U[J, J]
//   k_factor_tiles   phase 0: the panel, L[I, J] = C[I, J] U[J, J] for the rows I below (in place), and the
//                    first half of U's block column, U[a, J] = sum_k U[a, k] L[J, k]^T over k < J
//                    phase 1: the trailing matrix, C[I, K] -= L[I, J] L[K, J]^T, and the second half of
//                    U's block column, U[a, J] = -U[a, J] U[J, J]
// The tiles are the 128 x 128 tile products of split_gemm.cuh (fp32 precision on the tensor cores), one block each; a
// tile that is written in place reads nothing else than itself of what it writes.  Factor and inverse
// grow together, so the inverse costs no launches of its own.
//
// C is used up (its lower triangle becomes L off the diagonal blocks).  What of U is below the diagonal is not
// written: it has to be zero where a product reads it.  Finished entries of U are also left in the form that the
// application's products read (InverseOut).
// A non-positive or non-finite pivot is replaced and flagged.  Matrices whose r does not reach the
// block column do nothing.
//
// Measured on 75 matrices with r = 1024: see k_factor_block and k_factor_tiles.
constexpr int NB = split::TILE;
constexpr int PANEL = 8;                        // columns that k_factor_block eliminates at a time
constexpr int PP = PANEL + 4;                   // pitch of a panel's rows in shared memory
constexpr int FI = 8, FJ = 4;                   // tile (rows and columns) of a thread
// Row i of a panel in shared memory: rows i, i + 4, ... are neighbours, which the threads of a row of tiles read
// together; with the pitch above eight of them hit different banks.
__device__ __forceinline__ int panel_row(int i) { return (i % FJ * (NB / FJ) + i / FJ) * PP; }
constexpr int FACTOR_TILES = (NB / FI) * (NB / FI + 1);         // that reach into a lower triangle
constexpr int FACTOR_THREADS = (FACTOR_TILES + 31) / 32 * 32;

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }

// U = L^-T in every form that products read: fp32, and as parts or (on the tensor-core path) as bf16 with its remainder.
struct InverseOut {
  float* u;
  __nv_bfloat16* hi;                            // the second form lies `second` behind it, the third as far behind that
  long long second, pitch;
  int r, third;
  __device__ __forceinline__ explicit InverseOut(const RefreshMat& m) {
    u = m.U; r = m.r; third = !m.tc;
    hi = m.tc ? m.Ub[0] : m.Up.base;
    pitch = m.tc ? m.r : m.Up.pitch;
    second = m.tc ? m.Ub[1] - m.Ub[0] : m.Up.part_stride;
  }
  // n (<= 4) neighbours of row i from column j; vec: all four, from an aligned place.
  __device__ __forceinline__ void put(int i, int j, const float (&v)[4], int n, bool vec) const {
    float* f = u + (long long)i * r + j;
    __nv_bfloat16 *a = hi + i * pitch + j, *b = a + second, *c = b + second;
    uint32_t h[2], m[2], l[2];
    split::split3(v[0], v[1], h[0], m[0], l[0]);
    split::split3(v[2], v[3], h[1], m[1], l[1]);
    if (vec) {
      *reinterpret_cast<float4*>(f) = make_float4(v[0], v[1], v[2], v[3]);
      *reinterpret_cast<uint2*>(a) = make_uint2(h[0], h[1]);
      *reinterpret_cast<uint2*>(b) = make_uint2(m[0], m[1]);
      if (third) *reinterpret_cast<uint2*>(c) = make_uint2(l[0], l[1]);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (e < n) {
          f[e] = v[e];
          reinterpret_cast<unsigned short*>(a)[e] = (unsigned short)(h[e / 2] >> (16 * (e & 1)));
          reinterpret_cast<unsigned short*>(b)[e] = (unsigned short)(m[e / 2] >> (16 * (e & 1)));
          if (third) reinterpret_cast<unsigned short*>(c)[e] = (unsigned short)(l[e / 2] >> (16 * (e & 1)));
        }
    }
  }
};

// Diagonal block J0 / NB of every matrix: U = L^-T of the block C = L L^T.
//
// The lower triangle lives in registers, 8 x 4 entries per thread, eliminated in panels of 8 columns.  Where a column has
// been eliminated, its place takes the inverse's (T, the identity under the same row operations): one triangle
// holds both, and one update serves both, a(i, j) -= sum_k Q[i][k] Q[j][k] with
//   Q[i] = row i of L in the panel's columns            for rows below the panel,
//   Q[j] = column j of the inverse in the panel's rows  for columns up to the panel's end,
// both of which come out of the same forward substitution with the panel's diagonal 8 x 8 block.  That block's own
// factorisation is a chain of 8 pivots (root, reciprocal, product, difference); each of the 128 threads that
// substitute a row or column works it out for itself, which costs no exchange.
//
// Bound by the chain of 128 pivots, about 60 cycles each, and two block barriers per panel.  Measured (56 to 109
// matrices): 33 us; a blocked factorisation in shared memory with the chain in one warp (285 cycles per pivot)
// took 51.
__global__ void __launch_bounds__(FACTOR_THREADS)
k_factor_block(const RefreshMat* __restrict__ rm, int J0, float shift_rel, unsigned* __restrict__ status) {
  __shared__ __align__(16) float in[NB * PP], Q[NB * PP], diag[PANEL * PANEL];
  __shared__ float red[FACTOR_THREADS / 32];
  const RefreshMat& m = rm[blockIdx.x];
  const int r = m.r, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  ptx::grid_wait();
  ptx::grid_launch_next();
  if (J0 >= r) return;
  const int nb = min(NB, r - J0);
  const float* C = m.C + (long long)J0 * r + J0;
  float mean_diag;
  if (J0 == 0) {                                // trace(C) / r sets the shift and the pivot floor of all blocks
    float tr = 0.f;
    for (int i = tid; i < r; i += FACTOR_THREADS) tr += m.C[(long long)i * r + i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(0xffffffffu, tr, o);
    if (lane == 0) red[warp] = tr;
    __syncthreads();
    tr = 0.f;
    for (int w = 0; w < FACTOR_THREADS / 32; ++w) tr += red[w];
    mean_diag = tr / (float)r;
    if (tid == 0) m.info[0] = mean_diag;
  } else {
    mean_diag = m.info[0];
  }
  const float shift = shift_rel * mean_diag, floor_pivot = fmaxf(1e-30f, 1e-12f * mean_diag);
  const bool vec = r % 4 == 0;
  const InverseOut out(m);
  // this thread's tile: row of tiles ti, column tj <= 2 ti + 1, numbered row by row
  int ti = 0;
  while ((ti + 1) * (ti + 2) <= tid) ++ti;
  const int tj = tid - ti * (ti + 1);
  const bool mine = tid < FACTOR_TILES;
  const int i0 = FI * ti, j0 = FJ * tj;
  float a[FI][FJ];
#pragma unroll
  for (int x = 0; x < FI; ++x) {
    const int i = i0 + x;
    if (mine && vec && i < nb && j0 + 4 <= nb) {
      const float4 u = __ldcg(reinterpret_cast<const float4*>(C + (long long)i * r + j0));
      a[x][0] = u.x; a[x][1] = u.y; a[x][2] = u.z; a[x][3] = u.w;
    } else {
#pragma unroll
      for (int y = 0; y < FJ; ++y) a[x][y] = mine && i < nb && j0 + y < nb ? __ldcg(C + (long long)i * r + j0 + y) : 0.f;
    }
#pragma unroll
    for (int y = 0; y < FJ; ++y) {              // the lower triangle, shifted; past the matrix the identity's
      if (j0 + y > i) a[x][y] = 0.f;
      else if (j0 + y == i) a[x][y] = i < nb ? a[x][y] + shift : 1.f;
    }
  }
  bool bad = false;
#pragma unroll 1
  for (int c0 = 0; c0 < NB; c0 += PANEL) {
    const int q = c0 / FI, k0 = j0 - c0;        // the panel: row of tiles q, tile columns 2 q and 2 q + 1
    if (mine && ti == q) {
      if (k0 >= 0) {
#pragma unroll
        for (int x = 0; x < FI; ++x) *reinterpret_cast<float4*>(diag + x * PANEL + k0) = make_float4(a[x][0], a[x][1], a[x][2], a[x][3]);
      } else {                                  // the panel's rows of T
#pragma unroll
        for (int y = 0; y < FJ; ++y) {
          float* p = in + panel_row(j0 + y);
          *reinterpret_cast<float4*>(p) = make_float4(a[0][y], a[1][y], a[2][y], a[3][y]);
          *reinterpret_cast<float4*>(p + 4) = make_float4(a[4][y], a[5][y], a[6][y], a[7][y]);
        }
      }
    } else if (mine && ti > q && (k0 == 0 || k0 == FJ)) {        // rows below: the panel's columns of C
#pragma unroll
      for (int x = 0; x < FI; ++x) {
        *reinterpret_cast<float4*>(in + panel_row(i0 + x) + k0) = make_float4(a[x][0], a[x][1], a[x][2], a[x][3]);
#pragma unroll
        for (int y = 0; y < FJ; ++y) a[x][y] = 0.f;              // from here on T's
      }
    }
    __syncthreads();
    float v[PANEL];
    const int own = tid - c0;                   // a column of the panel itself starts as the identity's
    if (tid < NB) {
      float d[PANEL][PANEL];
#pragma unroll
      for (int i = 0; i < PANEL; ++i)
#pragma unroll
        for (int k = 0; k < PANEL; k += 4) {
          if (k > i) continue;
          const float4 u = ld4(diag + i * PANEL + k);
          d[i][k] = u.x; d[i][k + 1] = u.y; d[i][k + 2] = u.z; d[i][k + 3] = u.w;
        }
#pragma unroll
      for (int k = 0; k < PANEL; k += 4) {
        const float4 u = ld4(in + panel_row(tid) + k);
        v[k] = u.x; v[k + 1] = u.y; v[k + 2] = u.z; v[k + 3] = u.w;
      }
      if (own >= 0 && own < PANEL) {
#pragma unroll
        for (int k = 0; k < PANEL; ++k) v[k] = k == own ? 1.f : 0.f;
      }
#pragma unroll
      for (int k = 0; k < PANEL; ++k) {
        // (a pivot that is not a positive finite number becomes the bound it misses; padding's are 1)
        const float pv = fminf(fmaxf(d[k][k], c0 + k < nb ? floor_pivot : 0.f), 3.4e38f);
        bad |= pv != d[k][k];
        float s;
        asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"(pv));
        s = s * (1.5f - 0.5f * pv * s * s);     // one Newton step: to working precision
        v[k] *= s;
#pragma unroll
        for (int i = k + 1; i < PANEL; ++i) {
          d[i][k] *= s;
          v[i] = fmaf(-d[i][k], v[k], v[i]);
#pragma unroll
          for (int j = k + 1; j <= i; ++j) d[i][j] = fmaf(-d[i][k], d[j][k], d[i][j]);
        }
      }
#pragma unroll
      for (int k = 0; k < PANEL; k += 4) *reinterpret_cast<float4*>(Q + panel_row(tid) + k) = make_float4(v[k], v[k + 1], v[k + 2], v[k + 3]);
    }
    __syncthreads();
    if (tid < NB && own < PANEL && tid < nb) {  // rows c0 ... of the inverse are final: U's row `tid`
#pragma unroll
      for (int k = 0; k < PANEL; k += 4) {
        const float w[4] = {v[k], v[k + 1], v[k + 2], v[k + 3]};
        out.put(J0 + tid, J0 + c0 + k, w, nb - c0 - k, vec && c0 + k + 4 <= nb);
      }
    }
    if (mine && ti > q) {
#pragma unroll
      for (int k = 0; k < PANEL; k += 4) {
        float4 x[FI], y[FJ];
#pragma unroll
        for (int e = 0; e < FI; ++e) x[e] = ld4(Q + panel_row(i0 + e) + k);
#pragma unroll
        for (int f = 0; f < FJ; ++f) y[f] = ld4(Q + panel_row(j0 + f) + k);
#pragma unroll
        for (int e = 0; e < FI; ++e)
#pragma unroll
          for (int f = 0; f < FJ; ++f)
            a[e][f] = fmaf(-x[e].w, y[f].w, fmaf(-x[e].z, y[f].z, fmaf(-x[e].y, y[f].y, fmaf(-x[e].x, y[f].x, a[e][f]))));
      }
    }
  }
  if (bad) atomicOr(status, DEV_STATUS_NONFINITE);
}

// dst[i][j] (+)= sign * the finished tile, rows x cols of it, pitch r.
template <bool ACCUMULATE>
__device__ __forceinline__ void write_tile(float* dst, int r, int rows, int cols, const float* C, float sign) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (r % 4 == 0 && cols % 4 == 0) {
#pragma unroll 4
    for (int i = warp; i < rows; i += split::THREADS / 32)
      if (4 * lane < cols) {
        float4 v = *reinterpret_cast<const float4*>(C + i * split::C_LD + 4 * lane);
        float4* p = reinterpret_cast<float4*>(dst + (long long)i * r + 4 * lane);
        const float4 o = ACCUMULATE ? *p : make_float4(0.f, 0.f, 0.f, 0.f);
        *p = make_float4(o.x + sign * v.x, o.y + sign * v.y, o.z + sign * v.z, o.w + sign * v.w);
      }
  } else {
    for (int i = warp; i < rows; i += split::THREADS / 32)
      for (int j = lane; j < cols; j += 32) {
        float* p = dst + (long long)i * r + j;
        *p = (ACCUMULATE ? *p : 0.f) + sign * C[i * split::C_LD + j];
      }
  }
}

__global__ void __launch_bounds__(split::THREADS, 2)
k_factor_tiles(const RefreshMat* __restrict__ rm, int J, int phase, int tiles_per_matrix, unsigned* __restrict__ status) {
  extern __shared__ __align__(128) unsigned char smem[];
  split::Ctl* ctl = reinterpret_cast<split::Ctl*>(smem + split::STAGES * split::STAGE_BYTES);
  const RefreshMat& m = rm[blockIdx.x / tiles_per_matrix];
  int t = blockIdx.x % tiles_per_matrix;
  const int r = m.r, blocks = (r + NB - 1) / NB, below = blocks - 1 - J, J0 = J * NB;
  ptx::grid_wait();
  ptx::grid_launch_next();
  if (J >= blocks) return;
  const int nj = min(NB, r - J0);
  const int ours = phase == 0 ? below : below * (below + 1) / 2;    // tiles of the factor; then J tiles of the inverse
  if (t >= ours + J) return;
  split::begin(ctl);
  const float* Cs = reinterpret_cast<const float*>(smem);
  float* C = m.C;
  float* U = m.U;
  const long long ld = r;
  float* ujj = U + J0 * ld + J0;
  if (t < ours && phase == 0) {
    const int I0 = (J + 1 + t) * NB;
    float* c = C + I0 * ld + J0;
    split::Operand<float> a(c, ld, 1, r - I0, nj, 0), b(ujj, 1, ld, nj, nj, 0);
    if (split::tile_product<false>(a, b, nj, nj, smem, ctl)) write_tile<false>(c, r, min(NB, r - I0), nj, Cs, 1.f);
  } else if (t < ours) {
    int ti = 0;
    while (t > ti) { t -= ti + 1; ++ti; }       // block row ti, block column t <= ti below the panel
    const int I0 = (J + 1 + ti) * NB, K0 = (J + 1 + t) * NB;
    split::Operand<float> a(C + I0 * ld + J0, ld, 1, r - I0, nj, 0), b(C + K0 * ld + J0, ld, 1, r - K0, nj, 0);
    if (split::tile_product<false>(a, b, nj, r - K0, smem, ctl))
      write_tile<true>(C + I0 * ld + K0, r, min(NB, r - I0), min(NB, r - K0), Cs, -1.f);
  } else {
    const int A0 = (t - ours) * NB;
    float* u = U + A0 * ld + J0;
    if (phase == 0) {
      split::Operand<float> a(U + A0 * ld + A0, ld, 1, NB, J0 - A0, 0), b(C + J0 * ld + A0, ld, 1, nj, J0 - A0, 0);
      if (split::tile_product<true>(a, b, J0 - A0, nj, smem, ctl)) write_tile<false>(u, r, NB, nj, Cs, 1.f);
    } else {
      split::Operand<float> a(u, ld, 1, NB, nj, 0), b(ujj, 1, ld, nj, nj, 0);
      if (split::tile_product<false>(a, b, nj, nj, smem, ctl)) {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n = min(4, nj - 4 * lane);
        const InverseOut out(m);
#pragma unroll 4
        for (int i = warp; i < NB; i += split::THREADS / 32)
          if (n > 0) {
            const float4 v = *reinterpret_cast<const float4*>(Cs + i * split::C_LD + 4 * lane);
            const float w[4] = {-v.x, -v.y, -v.z, -v.w};
            out.put(A0 + i, J0 + 4 * lane, w, n, r % 4 == 0 && n == 4);
          }
      }
    }
  }
  split::end(ctl, status);
}

// Enqueues all of it; rmax: the largest r of the chunk.
cudaError_t factor_and_invert(const RefreshMat* rm_dev, int nm, int rmax, float shift_rel, unsigned* status_dev, cudaStream_t st) {
  static std::atomic<bool> ready[64];           // (the shared-memory limit is a per-device setting)
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess && (dev < 0 || dev >= 64)) e = cudaErrorInvalidDevice;
  if (e == cudaSuccess && !ready[dev].load()) {
    e = cudaFuncSetAttribute(k_factor_tiles, cudaFuncAttributeMaxDynamicSharedMemorySize, split::SMEM_BYTES);
    if (e == cudaSuccess) ready[dev].store(true);
  }
  if (e != cudaSuccess) return e;
  const int blocks = (rmax + NB - 1) / NB;
  for (int J = 0; J < blocks; ++J) {
    if (e == cudaSuccess) e = launch_chained(k_factor_block, nm, FACTOR_THREADS, 0, st, true, 1, rm_dev, J * NB, shift_rel, status_dev);
    for (int phase = 0; phase < 2; ++phase) {
      const int below = blocks - 1 - J, tiles = (phase == 0 ? below : below * (below + 1) / 2) + J;
      if (tiles && e == cudaSuccess)
        e = launch_chained(k_factor_tiles, nm * tiles, split::THREADS, split::SMEM_BYTES, st, true, 1, rm_dev, J, phase, tiles, status_dev);
    }
  }
  return e;
}
