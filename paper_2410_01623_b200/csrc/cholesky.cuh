// U = L^-T of C = L L^T (r x r, fp32, the lower triangle of C given), for all matrices of a chunk at once.
// Included by refresh.cu inside its namespace.
//
// Blocked over columns of NB = 128, three launches per block column J, each over every matrix:
//   k_factor_block   one block per matrix: factors C[J, J] and inverts the factor in shared memory; U[J, J]
//   k_factor_tiles   phase 0: the panel, L[I, J] = C[I, J] U[J, J] for the rows I below (in place), and the
//                    first half of U's block column, U[a, J] = sum_k U[a, k] L[J, k]^T over k < J
//                    phase 1: the trailing matrix, C[I, K] -= L[I, J] L[K, J]^T, and the second half of
//                    U's block column, U[a, J] = -U[a, J] U[J, J]
// The tiles are the 128 x 128 tile products of split_gemm.cuh (fp32 precision on the tensor cores), one block each; a
// tile that is written in place reads nothing else than itself of what it writes.  Factor and inverse
// grow together, so the inverse costs no launches of its own.
//
// C is used up (its lower triangle becomes L off the diagonal blocks).  U's blocks below the diagonal are not
// written: they have to be zero where a product reads them.
// A non-positive or non-finite pivot is replaced and flagged.  Matrices whose r does not reach the
// block column do nothing.
//
// Measured on 75 matrices with r = 1024: see k_factor_block and k_factor_tiles.
constexpr int NB = split::TILE;
constexpr int SB = 32;                          // sub-blocks of k_factor_block
constexpr int FP = NB + 4;                      // pitch: 16-byte rows, eight neighbouring rows in different banks
constexpr int FACTOR_THREADS = 256;
constexpr int FACTOR_SMEM = 2 * NB * FP * 4;

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }

// Eight steps of factor_subblock on rows whose last W entries are still to be done.  a: lane i's row i, moved left by
// one entry per step, so that the loop body is the same for every step (unrolled over all 32 steps one warp waits for
// its instructions: 20 us per sub-block instead of 4); t: lane j's column j of the identity on its way to the inverse,
// moved the same way.  Both take the entries of the factor's column below the pivot from `column` (the first of them,
// on which the next pivot waits, by a shuffle).
template <int W>
__device__ __forceinline__ void factor_steps(float (&a)[SB], float (&t)[SB], int k0, float* S, float* X, float* column,
                                             int n, float floor_pivot, bool& bad) {
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (int k = k0; k < k0 + 8; ++k) {
    float pv = __shfl_sync(0xffffffffu, a[0], k);
    if (k < n && !(pv > floor_pivot && pv < INFINITY)) { bad = true; pv = floor_pivot; }
    float s = rsqrtf(pv);
    s = s * (1.5f - 0.5f * pv * s * s);         // one Newton step: to working precision
    const float l = lane == k ? pv * s : a[0] * s, x = t[0] * s;
    float* c = column + (k & 1) * SB;           // (two in turn: nobody is more than a step behind)
    if (lane > k) c[lane - k - 1] = l;
    S[lane * FP + k] = lane >= k ? l : 0.f;
    X[k * FP + lane] = x;
    const float next = __shfl_sync(0xffffffffu, l, k + 1);
    a[0] = a[1] - l * next;
    t[0] = t[1] - next * x;
    __syncwarp();
#pragma unroll
    for (int j = 0; j < W; j += 4) {            // (entries past the row's end never come to the front)
      const float4 v = ld4(c + j);
      const float w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (j + q > 0 && j + q < W - 1) {
          a[j + q] = a[j + q + 1] - l * w[q];
          t[j + q] = t[j + q + 1] - w[q] * x;
        }
    }
  }
}

// One warp: Cholesky factor of the SB x SB block at S (pitch FP) in place and its inverse at X.
// n of its rows are the matrix's, the others the identity's.
__device__ __forceinline__ void factor_subblock(float* S, float* X, float* column, int n, float floor_pivot, bool& bad) {
  const int lane = threadIdx.x & 31;
  float a[SB], t[SB];
#pragma unroll
  for (int j = 0; j < SB; j += 4) {
    const float4 v = ld4(S + lane * FP + j);
    a[j] = v.x; a[j + 1] = v.y; a[j + 2] = v.z; a[j + 3] = v.w;
#pragma unroll
    for (int q = 0; q < 4; ++q) t[j + q] = j + q == lane ? 1.f : 0.f;
  }
  __syncwarp();
  factor_steps<32>(a, t, 0, S, X, column, n, floor_pivot, bad);
  factor_steps<24>(a, t, 8, S, X, column, n, floor_pivot, bad);
  factor_steps<16>(a, t, 16, S, X, column, n, floor_pivot, bad);
  factor_steps<8>(a, t, 24, S, X, column, n, floor_pivot, bad);
}

// Products in shared memory (pitch FP), NX blocks of 32 x 32, four neighbours of a row of every block per thread.
//   by_rows:  acc[x][y] = sum_k P[row + 32 x][k] Q[col + 8 y][k]      (col = lane % 8)
//   otherwise acc[x][y] = sum_k P[row][k] Q[k][32 x + 4 col + y]
// Four of k at a time, all loads 16 bytes and free of bank conflicts: for three blocks 7 or 13 of them for 48
// multiply-adds.
template <int NX, bool BY_ROWS>
__device__ __forceinline__ void small_product(float (&acc)[3][4], const float* P, const float* Q, int depth) {
  const int col = threadIdx.x & 7, row = threadIdx.x >> 3;
#pragma unroll
  for (int x = 0; x < NX; ++x)
#pragma unroll
    for (int y = 0; y < 4; ++y) acc[x][y] = 0.f;
#pragma unroll 2
  for (int k = 0; k < depth; k += 4) {
    if (BY_ROWS) {
      float4 p[NX], q[4];
#pragma unroll
      for (int x = 0; x < NX; ++x) p[x] = ld4(P + (row + 32 * x) * FP + k);
#pragma unroll
      for (int y = 0; y < 4; ++y) q[y] = ld4(Q + (col + 8 * y) * FP + k);
#pragma unroll
      for (int x = 0; x < NX; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y)
          acc[x][y] = fmaf(p[x].w, q[y].w, fmaf(p[x].z, q[y].z, fmaf(p[x].y, q[y].y, fmaf(p[x].x, q[y].x, acc[x][y]))));
    } else {
      const float4 p = ld4(P + row * FP + k);
      const float pk[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
      for (int x = 0; x < NX; ++x)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float4 q = ld4(Q + (k + u) * FP + 32 * x + 4 * col);
          acc[x][0] = fmaf(pk[u], q.x, acc[x][0]);
          acc[x][1] = fmaf(pk[u], q.y, acc[x][1]);
          acc[x][2] = fmaf(pk[u], q.z, acc[x][2]);
          acc[x][3] = fmaf(pk[u], q.w, acc[x][3]);
        }
    }
  }
}
template <bool BY_ROWS>
__device__ __forceinline__ void small_product(int nx, float (&acc)[3][4], const float* P, const float* Q, int depth) {
  if (nx == 3) small_product<3, BY_ROWS>(acc, P, Q, depth);
  else if (nx == 2) small_product<2, BY_ROWS>(acc, P, Q, depth);
  else if (nx == 1) small_product<1, BY_ROWS>(acc, P, Q, depth);
}

// Diagonal block J0 / NB of every matrix.  Bound by the chain of 128 pivots, which one warp runs through.
__global__ void __launch_bounds__(FACTOR_THREADS)
k_factor_block(const RefreshMat* __restrict__ rm, int J0, float shift_rel, unsigned* __restrict__ status) {
  extern __shared__ __align__(16) float fsm[];
  __shared__ float red[FACTOR_THREADS / 32];
  __shared__ __align__(16) float column[2 * SB];
  float* S = fsm;                               // the block, later its factor
  float* X = fsm + NB * FP;                     // the factor's inverse
  const RefreshMat& m = rm[blockIdx.x];
  const int r = m.r, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
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
  // eight groups of four entries per thread at a time, their loads before their stores to shared memory
  const bool vec = r % 4 == 0;
#pragma unroll 1
  for (int h = 0; h < NB * NB / 4; h += 8 * FACTOR_THREADS) {
    float v[8][4];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int e = h + q * FACTOR_THREADS + tid, i = e / (NB / 4), j = e % (NB / 4) * 4;
      if (vec && i < nb && j < nb) {
        const float4 u = __ldcg(reinterpret_cast<const float4*>(C + (long long)i * r + j));
        v[q][0] = u.x; v[q][1] = u.y; v[q][2] = u.z; v[q][3] = u.w;
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) v[q][c] = i < nb && j + c < nb ? __ldcg(C + (long long)i * r + j + c) : (i == j + c ? 1.f : 0.f);
      }
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int e = h + q * FACTOR_THREADS + tid, i = e / (NB / 4), j = e % (NB / 4) * 4;
#pragma unroll
      for (int c = 0; c < 4; ++c) {             // the lower triangle, shifted
        if (j + c > i) v[q][c] = 0.f;
        else if (j + c == i && i < nb) v[q][c] += shift;
      }
      *reinterpret_cast<float4*>(S + i * FP + j) = make_float4(v[q][0], v[q][1], v[q][2], v[q][3]);
      *reinterpret_cast<float4*>(X + i * FP + j) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  __syncthreads();
  bool bad = false;
  const int col = tid & 7, row = tid >> 3;
  for (int b = 0; b < NB; b += SB) {
    if (warp == 0) factor_subblock(S + b * FP + b, X + b * FP + b, column, nb - b, floor_pivot, bad);
    __syncthreads();
    const int lo = b + SB, below = (NB - lo) / SB;
    float acc[3][4];
    // rows below: S[i][b + j] <- sum_k S[i][b + k] X[b + j][b + k]
    small_product<true>(below, acc, S + lo * FP + b, X + b * FP + b, SB);
    __syncthreads();
#pragma unroll
    for (int x = 0; x < 3; ++x)
#pragma unroll
      for (int y = 0; y < 4; ++y)
        if (x < below) S[(lo + row + 32 * x) * FP + b + col + 8 * y] = acc[x][y];
    // X[b + j][i] = -sum_k X[b + j][b + k] T[k][i] with T[j][i] = sum_k S[b + j][k] X[k][i], over the columns
    // i < b; T takes the place of the row block of S that it is made of
    small_product<false>(b / SB, acc, S + b * FP, X, b);
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 3; ++c)
      if (c * SB < b) *reinterpret_cast<float4*>(S + (b + row) * FP + c * SB + 4 * col) = make_float4(acc[c][0], acc[c][1], acc[c][2], acc[c][3]);
    // the rest of the block: S[i][j] -= sum_k S[i][b + k] S[j][b + k], 32 columns at a time
    for (int c = 0; c < below; ++c) {
      small_product<true>(below, acc, S + lo * FP + b, S + (lo + SB * c) * FP + b, SB);
#pragma unroll
      for (int x = 0; x < 3; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) {
          const int i = lo + row + 32 * x, j = lo + SB * c + col + 8 * y;
          if (x < below && j <= i) S[i * FP + j] -= acc[x][y];
        }
    }
    __syncthreads();
    small_product<false>(b / SB, acc, X + b * FP + b, S + b * FP, SB);
#pragma unroll
    for (int c = 0; c < 3; ++c)
      if (c * SB < b) *reinterpret_cast<float4*>(X + (b + row) * FP + c * SB + 4 * col) = make_float4(-acc[c][0], -acc[c][1], -acc[c][2], -acc[c][3]);
    __syncthreads();
  }
  if (bad && lane == 0) atomicOr(status, DEV_STATUS_NONFINITE);
  float* out = m.U + (long long)J0 * r + J0;    // U = X^T: a lane is a row of X
  for (int e = warp; e < (NB / 32) * (NB / 4); e += FACTOR_THREADS / 32) {
    const int j = (e % (NB / 32)) * 32 + lane, k = (e / (NB / 32)) * 4;
    const float4 v = ld4(X + j * FP + k);
    const float w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (j < nb && k + q < nb) out[(long long)(k + q) * r + j] = w[q];
  }
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
      if (split::tile_product<false>(a, b, nj, nj, smem, ctl)) write_tile<false>(u, r, NB, nj, Cs, -1.f);
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
    e = cudaFuncSetAttribute(k_factor_block, cudaFuncAttributeMaxDynamicSharedMemorySize, FACTOR_SMEM);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_factor_tiles, cudaFuncAttributeMaxDynamicSharedMemorySize, split::SMEM_BYTES);
    if (e == cudaSuccess) ready[dev].store(true);
  }
  if (e != cudaSuccess) return e;
  const int blocks = (rmax + NB - 1) / NB;
  for (int J = 0; J < blocks; ++J) {
    k_factor_block<<<nm, FACTOR_THREADS, FACTOR_SMEM, st>>>(rm_dev, J * NB, shift_rel, status_dev);
    for (int phase = 0; phase < 2; ++phase) {
      const int below = blocks - 1 - J, tiles = (phase == 0 ? below : below * (below + 1) / 2) + J;
      if (tiles) k_factor_tiles<<<nm * tiles, split::THREADS, split::SMEM_BYTES, st>>>(rm_dev, J, phase, tiles, status_dev);
    }
  }
  return cudaSuccess;
}
