// Projection refresh (Eq. 7): an orthonormal basis of the dominant rank-r singular
// subspace of G, by blocked subspace iteration on the device.
//
// With A = G seen as a d x l matrix (d = projected extent):
//   Z <- Gaussian (l x r);  Y <- orth(A Z)
//   repeat `iters` times:   Z <- orth(A^T Y);  Y <- orth(A Z)
//   projection <- Y  (d x r)
// orth() is CholeskyQR: C = Y^T Y, C = L L^T, Y <- Y L^-T, once for the intermediate
// iterates and twice for the basis that is kept.  It changes the basis, never the
// spanned subspace, so a small diagonal shift in the first pass (which keeps the
// factorisation defined for ill-conditioned Y) costs no accuracy of the subspace.
// The paper calls a library SVD here; the iteration converges to the same subspace
// at the rate (sigma_{r+1}/sigma_r)^2 per round.
//
// Products.  bf16 matrices of tensor-core size with TMA-readable rows use the step's projection kernel in
// its plain-output mode (fp32 accumulation in tensor memory):
//   * A Z and A^T Y: G is exact in bf16; the iterate is rounded to bf16, and in the last round it is
//     split into a bf16 high part and a bf16 remainder (two k-segments), so that the basis that is
//     kept carries no bf16 rounding of the iterate;
//   * the Gram product Y^T Y and the application of the inverse factor Y <- Y L^-T: for the basis
//     that is kept both operands are fp32 matrices split into two bf16 parts, three k-segments
//     (hi hi + hi lo + lo hi), which is good to about 2^-16: enough for CholeskyQR, whose second pass
//     removes what the first left; for the intermediate iterates plain bf16 operands (one segment):
//     the next product rounds the iterate to bf16 anyway, and all it asks is a well-conditioned one.
// Every other matrix (fp32, odd pitches, small or odd ranks) is iterated in fp32 precision: G, Y, Z and L^-T
// are kept as bf16 parts (three, or one for a bf16 G) and multiplied by the part products of
// part_gemm.cu, which also leave their results as parts; only the Gram matrix is needed as fp32.  On the
// CUDA cores these products were 90 % of the refresh of a list with odd-width matrices.
// The Cholesky factorisation and L^-T (r x r, fp32 precision): cholesky.cuh.
//
// Random numbers: Philox4x32-10 (Salmon et al., "Parallel random numbers: as easy
// as 1, 2, 3", SC'11), keyed by the caller's seed, turned into normals by the
// Box-Muller transform.
#include <string.h>

#include <algorithm>
#include <atomic>

#include "context.cuh"
#include "part_gemm.cuh"
#include "split_gemm.cuh"
#include "step_tc.cuh"

namespace fira {

namespace {

struct RefreshMat {
  const void* G;
  void* P;
  float* C;   // r x r
  float* U;   // r x r: L^-T
  // matrices iterated in fp32 precision: everything as bf16 parts; the two buffers of an iterate hold it
  // before and after its orthonormalisation
  PartMatrix Gp, Y0, Y1, Z0, Z1, Up;
  // matrices whose products run on the step's projection kernel (tc): bf16 roundings [0] and remainders [1]
  // of Y and Z before (index 0) and after (1) their orthonormalisation and of U.  Y[0] also has room for the kept
  // basis in fp32.
  __nv_bfloat16* Y[2][2];
  __nv_bfloat16* Z[2][2];
  __nv_bfloat16* Ub[2];
  float* out32;        // optional copy of the kept basis in fp32, before it is rounded for storage
  float* info;         // a few floats of the Cholesky factorisation (pivot floor)
  int tc;
  long long ld;
  int d, l, r;
  int left, bf16;
  unsigned long long key;
};

// ------------------------------------------------------------------ Philox4x32-10
__device__ __forceinline__ void philox4x32_10(unsigned c0, unsigned c1, unsigned c2, unsigned c3,
                                              unsigned k0, unsigned k1, unsigned (&out)[4]) {
  const unsigned M0 = 0xD2511F53u, M1 = 0xCD9E8D57u, W0 = 0x9E3779B9u, W1 = 0xBB67AE85u;
#pragma unroll
  for (int round = 0; round < 10; ++round) {
    const unsigned hi0 = __umulhi(M0, c0), lo0 = M0 * c0;
    const unsigned hi1 = __umulhi(M1, c2), lo1 = M1 * c2;
    const unsigned n0 = hi1 ^ c1 ^ k0, n1 = lo1, n2 = hi0 ^ c3 ^ k1, n3 = lo0;
    c0 = n0; c1 = n1; c2 = n2; c3 = n3;
    k0 += W0; k1 += W1;
  }
  out[0] = c0; out[1] = c1; out[2] = c2; out[3] = c3;
}

__global__ void __launch_bounds__(256)
k_gauss(const RefreshMat* __restrict__ rm) {
  const RefreshMat m = rm[blockIdx.y];
  const long long total = (long long)m.l * m.r;
  const long long quads = (total + 3) / 4;
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < quads;
       q += (long long)gridDim.x * blockDim.x) {
    unsigned o[4];
    philox4x32_10((unsigned)q, (unsigned)(q >> 32), 0u, 0u, (unsigned)m.key, (unsigned)(m.key >> 32), o);
    // two Box-Muller pairs; the radius uniforms lie in (0, 1]
    const float u0 = ((float)(o[0] >> 8) + 1.0f) * (1.0f / 16777216.0f);
    const float u1 = (float)(o[1] >> 8) * (1.0f / 16777216.0f);
    const float u2 = ((float)(o[2] >> 8) + 1.0f) * (1.0f / 16777216.0f);
    const float u3 = (float)(o[3] >> 8) * (1.0f / 16777216.0f);
    const float ra = sqrtf(-2.0f * logf(u0)), rb = sqrtf(-2.0f * logf(u2));
    float s0, c0, s1, c1;
    sincospif(2.0f * u1, &s0, &c0);
    sincospif(2.0f * u3, &s1, &c1);
    const float v[4] = {ra * c0, ra * s0, rb * c1, rb * s1};
    for (int e = 0; e < 4; ++e) {
      const long long idx = q * 4 + e;
      if (idx >= total) break;
      if (m.tc) {
        const __nv_bfloat16 h = __float2bfloat16_rn(v[e]);
        m.Z[1][0][idx] = h;
        m.Z[1][1][idx] = __float2bfloat16_rn(v[e] - __bfloat162float(h));
        continue;
      }
      uint32_t h, mid, lo;
      split::split3(v[e], 0.f, h, mid, lo);
      __nv_bfloat16_raw* o = reinterpret_cast<__nv_bfloat16_raw*>(m.Z1.base) + idx / m.r * m.Z1.pitch + idx % m.r;
      o[0].x = (unsigned short)h; o[m.Z1.part_stride].x = (unsigned short)mid; o[2 * m.Z1.part_stride].x = (unsigned short)lo;
    }
  }
}

// ------------------------------------------------------------------ parts
// G as parts, once.  Eight neighbours per thread; the columns between its width and its pitch become zeros.
template <typename T>
__device__ __forceinline__ void to_parts(const T* src, long long ld, const PartMatrix& p) {
  const bool vec = ld * (long long)sizeof(T) % 16 == 0 && reinterpret_cast<unsigned long long>(src) % 16 == 0;
  const long long per_row = p.pitch / 8, units = p.rows * per_row;
  for (long long u = (long long)blockIdx.x * blockDim.x + threadIdx.x; u < units; u += (long long)gridDim.x * blockDim.x) {
    const long long i = u / per_row, j = u % per_row * 8;
    split::Frag<T> f;
    split::load_frag(src + i * ld + j, (int)(p.cols - j), vec, f);
    split::store_parts(reinterpret_cast<unsigned char*>(p.base + i * p.pitch + j), f, p.part_stride * 2);
  }
}
__global__ void __launch_bounds__(256)
k_to_parts(const RefreshMat* __restrict__ rm) {
  const RefreshMat& m = rm[blockIdx.y];
  if (m.tc) return;
  if (m.bf16) to_parts((const __nv_bfloat16*)m.G, m.ld, m.Gp);
  else to_parts((const float*)m.G, m.ld, m.Gp);
}

#include "cholesky.cuh"

__global__ void __launch_bounds__(256)
k_store_projection(const RefreshMat* __restrict__ rm) {
  const RefreshMat& m = rm[blockIdx.y];
  const long long total = (long long)m.d * m.r;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    float y;
    if (m.tc) {
      y = reinterpret_cast<const float*>(m.Y[0][0])[i];
    } else {                                   // the sum of the parts is the fp32 number they were made of
      const __nv_bfloat16* p = m.Y0.base + i / m.r * m.Y0.pitch + i % m.r;
      y = __bfloat162float(p[0]) + (__bfloat162float(p[m.Y0.part_stride]) + __bfloat162float(p[2 * m.Y0.part_stride]));
    }
    if (m.bf16) ((__nv_bfloat16*)m.P)[i] = __float2bfloat16_rn(y);
    else ((float*)m.P)[i] = y;
    if (m.out32) m.out32[i] = y;
  }
}

// U <- 0 in all its forms, once: what is below the diagonal is never written.
__global__ void __launch_bounds__(256)
k_clear_inverse(const RefreshMat* __restrict__ rm) {
  const RefreshMat& m = rm[blockIdx.y];
  const long long total = (long long)m.r * m.r, first = (long long)blockIdx.x * blockDim.x + threadIdx.x, step = (long long)gridDim.x * blockDim.x;
  for (long long i = first; i < total; i += step) m.U[i] = 0.f;
  uint4* p = reinterpret_cast<uint4*>(m.tc ? m.Ub[0] : m.Up.base);      // (two or three forms, one behind the other)
  const long long units = (m.tc ? 2 * total : 3 * m.Up.part_stride) / 8;
  for (long long i = first; i < units; i += step) p[i] = make_uint4(0u, 0u, 0u, 0u);
}

// descriptor tables of a chunk: per-matrix entries plus alignment slack
constexpr size_t TABLE_PER_MATRIX = 1024;
constexpr size_t TABLE_SLACK = 16 * 1024;
static_assert(sizeof(RefreshMat) <= TABLE_PER_MATRIX, "table allowance");

}  // namespace

// bf16 matrices that TMA can read in place: their products run on the tensor cores
static bool refresh_on_tc(const fira_matrix_desc& d) {
  return d.dtype == FIRA_BF16 && tc_supported(d) && tc_rows_aligned(d);   // the refresh only reads G
}

// The tensor-core jobs of one matrix.  Y and Z exist twice (before and after their orthonormalisation), as bf16 and,
// where the next product asks for it, with the bf16 remainder.  The Gram products and the applications of L^-T: with split
// operands (three k-segments) for the basis that is kept, with plain bf16 operands (one segment) for the
// intermediate iterates, which the next product rounds to bf16 anyway and which only have to stay well conditioned.
enum { JOB_AZ = 0, JOB_AZ_SPLIT, JOB_ATY, JOB_ATY_SPLIT, JOB_GRAM_Y, JOB_GRAM_Y_SPLIT, JOB_GRAM_Y2_SPLIT, JOB_GRAM_Z,
       JOB_GRAM_Z_SPLIT, JOB_APPLY_Y, JOB_APPLY_Y_LO, JOB_APPLY_Y_SPLIT, JOB_APPLY_Y2_SPLIT, JOB_APPLY_Z, JOB_APPLY_Z_SPLIT,
       JOB_KINDS };

static TcGemmJob refresh_job(const RefreshMat& m, int kind) {
  TcGemmJob j;
  memset(&j, 0, sizeof(j));
  j.r = m.r;
  auto with_g = [&](bool az, __nv_bfloat16* const (&b)[2], __nv_bfloat16* const (&out)[2], bool split) {
    j.G = m.G; j.ld = m.ld;
    j.m = m.left ? m.d : m.l; j.n = m.left ? m.l : m.d;
    j.mn_major = az ? !m.left : m.left;    // A Z: rows d, k = l;  A^T Y: rows l, k = d
    j.B = b[0]; j.hi = out[0];
    if (split) { j.B_lo = b[1]; j.lo = out[1]; j.nseg = 2; j.asel = 0u; j.bsel = 2u; }   // A hi, A lo(iterate)
  };
  auto segments = [&](__nv_bfloat16* const (&a)[2], __nv_bfloat16* const (&b)[2], bool split) {
    j.G = a[0]; j.B = b[0];
    if (split) { j.G_lo = a[1]; j.B_lo = b[1]; j.nseg = 3; j.asel = 4u; j.bsel = 2u; }   // hi hi, hi lo, lo hi
  };
  auto gram = [&](__nv_bfloat16* const (&x)[2], int rows, bool split) {    // C[i][j] = sum_k X[k][i] X[k][j]: "G" = X as [k][i]
    j.m = rows; j.n = j.r; j.ld = j.r; j.mn_major = 1; j.C = m.C; j.lower = 1;
    segments(x, x, split);
  };
  auto apply = [&](__nv_bfloat16* const (&x)[2], int rows, __nv_bfloat16* const (&out)[2], bool split, bool with_lo) {
    j.m = rows; j.n = j.r; j.ld = j.r; j.mn_major = 0; j.upper_b = 1;      // X[i][j] = sum_k X[i][k] U[k][j]: "G" = X as [i][k]
    segments(x, m.Ub, split);
    j.hi = out[0]; j.lo = with_lo ? out[1] : nullptr;
  };
  switch (kind) {
    case JOB_AZ: with_g(true, m.Z[1], m.Y[0], false); break;
    case JOB_AZ_SPLIT: with_g(true, m.Z[1], m.Y[0], true); break;
    case JOB_ATY: with_g(false, m.Y[1], m.Z[0], false); break;
    case JOB_ATY_SPLIT: with_g(false, m.Y[1], m.Z[0], true); break;
    case JOB_GRAM_Y: gram(m.Y[0], m.d, false); break;
    case JOB_GRAM_Y_SPLIT: gram(m.Y[0], m.d, true); break;
    case JOB_GRAM_Y2_SPLIT: gram(m.Y[1], m.d, true); break;
    case JOB_GRAM_Z: gram(m.Z[0], m.l, false); break;
    case JOB_GRAM_Z_SPLIT: gram(m.Z[0], m.l, true); break;
    case JOB_APPLY_Y: apply(m.Y[0], m.d, m.Y[1], false, false); break;
    case JOB_APPLY_Y_LO: apply(m.Y[0], m.d, m.Y[1], false, true); break;   // the last plain one: a split product follows
    case JOB_APPLY_Y_SPLIT: apply(m.Y[0], m.d, m.Y[1], true, true); break;
    case JOB_APPLY_Y2_SPLIT:                                               // the kept basis, in fp32
      apply(m.Y[1], m.d, m.Y[0], true, false);
      j.hi = nullptr; j.C = reinterpret_cast<float*>(m.Y[0][0]);
      break;
    case JOB_APPLY_Z: apply(m.Z[0], m.l, m.Z[1], false, false); break;
    default: apply(m.Z[0], m.l, m.Z[1], true, true); break;
  }
  return j;
}

// The part products of a matrix that is iterated in fp32 precision.
enum { PART_AZ = 0, PART_ATY, PART_GRAM_Y, PART_APPLY_Y, PART_GRAM_Y2, PART_APPLY_Y2, PART_GRAM_Z, PART_APPLY_Z, PART_KINDS };

static PartGemm part_job(const RefreshMat& m, int kind) {
  PartGemm g;
  auto gram = [&](const PartMatrix& x) { g.a = g.b = x; g.a_t = true; g.c = m.C; g.ldc = m.r; g.lower = true; };
  auto apply = [&](const PartMatrix& x, const PartMatrix& y) { g.a = x; g.b = m.Up; g.upper_b = true; g.out = y; };
  switch (kind) {
    case PART_AZ: g.a = m.Gp; g.a_t = !m.left; g.b = m.Z1; g.out = m.Y0; break;
    case PART_ATY: g.a = m.Gp; g.a_t = m.left; g.b = m.Y1; g.out = m.Z0; break;
    case PART_GRAM_Y: gram(m.Y0); break;
    case PART_APPLY_Y: apply(m.Y0, m.Y1); break;
    case PART_GRAM_Y2: gram(m.Y1); break;
    case PART_APPLY_Y2: apply(m.Y1, m.Y0); break;
    case PART_GRAM_Z: gram(m.Z0); break;
    default: apply(m.Z0, m.Z1); break;
  }
  return g;
}

// The matrix's buffers, carved from base (null: only their sizes count); *end_out: what follows.
static RefreshMat carve_refresh(const fira_matrix_desc& dsc, char* base, size_t* bytes_out) {
  RefreshMat m{};
  size_t off = 0;
  auto take = [&](size_t bytes) { char* p = base ? base + off : nullptr; off += align_up(bytes); return p; };
  m.ld = dsc.ld ? dsc.ld : dsc.n;
  m.d = std::min(dsc.m, dsc.n); m.l = std::max(dsc.m, dsc.n); m.r = dsc.r;
  m.left = dsc.m <= dsc.n; m.bf16 = dsc.dtype == FIRA_BF16;
  m.tc = refresh_on_tc(dsc) ? 1 : 0;
  const size_t d = m.d, l = m.l, r = m.r;
  m.C = (float*)take(r * r * 4);
  m.U = (float*)take(r * r * 4);
  m.info = (float*)take(256);
  if (m.tc) {
    auto pair = [&](__nv_bfloat16* (&p)[2], size_t elements) {       // one buffer: together they hold as many floats
      p[0] = (__nv_bfloat16*)take(elements * 4);
      p[1] = p[0] ? p[0] + elements : nullptr;
    };
    for (int i = 0; i < 2; ++i) { pair(m.Y[i], d * r); pair(m.Z[i], l * r); }
    pair(m.Ub, r * r);
  } else {
    auto parts = [&](long long rows, long long cols, int n) { return part_matrix(take(part_matrix_bytes(rows, cols, n)), rows, cols, n); };
    m.Gp = parts(dsc.m, dsc.n, m.bf16 ? 1 : 3);
    m.Y0 = parts(d, r, 3); m.Y1 = parts(d, r, 3);
    m.Z0 = parts(l, r, 3); m.Z1 = parts(l, r, 3);
    m.Up = parts(r, r, 3);
  }
  *bytes_out = off;
  return m;
}

static size_t refresh_data_bytes(const fira_matrix_desc& d) {
  size_t b = 0;
  const RefreshMat m = carve_refresh(d, nullptr, &b);
  if (m.tc)
    for (int k = 0; k < JOB_KINDS; ++k) { const TcGemmJob j = refresh_job(m, k); b += tc_gemm_table_bytes(&j, 1); }
  else
    for (int k = 0; k < PART_KINDS; ++k) { const PartGemm g = part_job(m, k); b += part_gemm_table_bytes(&g, 1); }
  return b;
}

size_t refresh_bytes_per_matrix(const fira_matrix_desc& d) {
  return refresh_data_bytes(d) + TABLE_PER_MATRIX + TABLE_SLACK;
}

#define RF_CUDA(call)                                                          \
  do {                                                                         \
    cudaError_t e_ = (call);                                                   \
    if (e_ != cudaSuccess) {                                                   \
      set_error(std::string(#call) + ": " + cudaGetErrorString(e_));           \
      return FIRA_ERR_CUDA;                                                    \
    }                                                                          \
  } while (0)

// Refreshes the matrices of `which` in chunks that fit the work area.  The work
// area is shared with the step's scratch, whose contents are dead between steps.
// basis_out (may be null): per matrix index an optional device pointer that receives the kept
// basis in fp32 (d x r) before it is rounded to the storage type.
fira_status refresh_impl(fira_ctx* c, const void* const* G_dev, const std::vector<int>& which,
                         uint64_t seed, int iters, float* const* basis_out, const RefreshTarget* target) {
  if (iters < 0) iters = 4;
  RefreshTarget own;
  own.work_base = c->work_base; own.work_bytes = c->work_bytes; own.stream = c->stream;
  const RefreshTarget& tg = target ? *target : own;
  if (!tg.P_out) c->proj_weights_dirty = true;
  cudaStream_t st = tg.stream;
  size_t pos = 0;
  while (pos < which.size()) {
    // ---- carve a chunk: as many matrices as fit (data regions first, then the tables of all)
    std::vector<size_t> offs;
    size_t need = 0, off = 0, q = pos;
    for (; q < which.size(); ++q) {
      size_t data = 0;
      carve_refresh(c->descs[which[q]], nullptr, &data);
      need += refresh_data_bytes(c->descs[which[q]]) + TABLE_PER_MATRIX;
      if (need + TABLE_SLACK > tg.work_bytes) break;
      offs.push_back(off);
      off += data;
    }
    if (q == pos) { set_error("scratch buffer too small for the projection refresh"); return FIRA_ERR_WORKSPACE_TOO_SMALL; }
    const int nm = (int)(q - pos);
    std::vector<RefreshMat> rms;
    size_t data_end = 0;
    for (int a = 0; a < nm; ++a) {
      const int idx = which[pos + a];
      const MatDev& mt = c->mats[idx];
      size_t bytes = 0;
      RefreshMat rm = carve_refresh(c->descs[idx], tg.work_base + offs[a], &bytes);
      rm.G = G_dev[idx]; rm.P = tg.P_out ? tg.P_out[idx] : mt.P;
      rm.out32 = basis_out ? basis_out[idx] : nullptr;
      data_end = std::max(data_end, offs[a] + bytes);
      rm.key = seed * 0x9E3779B97F4A7C15ull + (unsigned long long)idx * 0xD1B54A32D192ED03ull + 1ull;
      rms.push_back(rm);
    }
    // ---- the products' jobs
    std::vector<PartGemm> pjobs[PART_KINDS];
    std::vector<TcGemmJob> jobs[JOB_KINDS];
    for (size_t a = 0; a < rms.size(); ++a) {
      const RefreshMat& m = rms[a];
      if (m.tc) {
        for (int k = 0; k < JOB_KINDS; ++k) jobs[k].push_back(refresh_job(m, k));
      } else {
        for (int k = 0; k < PART_KINDS; ++k) pjobs[k].push_back(part_job(m, k));
      }
    }
    char* tp = tg.work_base + align_up(data_end);
    cudaError_t cerr = cudaSuccess;
    auto put = [&](const void* src, size_t bytes) -> char* {
      char* dst = tp;
      if (bytes == 0) return dst;
      if ((size_t)(tp + align_up(bytes) - tg.work_base) > tg.work_bytes) { cerr = cudaErrorInvalidValue; return dst; }
      cudaError_t e = cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, st);
      if (e != cudaSuccess) cerr = e;
      tp += align_up(bytes);
      return dst;
    };
    const RefreshMat* rm_dev = (const RefreshMat*)put(rms.data(), rms.size() * sizeof(RefreshMat));
    if (cerr != cudaSuccess) { set_error(std::string("refresh tables: ") + cudaGetErrorString(cerr)); return FIRA_ERR_CUDA; }
    // tables of the tensor-core jobs (tensor maps and tile records), after the others
    const int ntc = (int)jobs[0].size(), nparts = nm - ntc;
    char* tab[JOB_KINDS] = {};
    int jtiles[JOB_KINDS] = {};
    if (ntc) {
      for (int k = 0; k < JOB_KINDS; ++k) {
        const size_t bytes = tc_gemm_table_bytes(jobs[k].data(), ntc);
        if ((size_t)(tp + bytes - tg.work_base) > tg.work_bytes) {
          set_error("scratch buffer too small for the projection refresh"); return FIRA_ERR_WORKSPACE_TOO_SMALL;
        }
        tab[k] = tp;
        const fira_status ps = tc_gemm_prepare(c, jobs[k].data(), ntc, tab[k], bytes, &jtiles[k], st);
        if (ps != FIRA_OK) return ps;
        tp += bytes;
      }
    }
    char* ptab[PART_KINDS] = {};
    int ptiles[PART_KINDS] = {};
    if (nparts)
      for (int k = 0; k < PART_KINDS; ++k) {
        const size_t bytes = part_gemm_table_bytes(pjobs[k].data(), nparts);
        if ((size_t)(tp + bytes - tg.work_base) > tg.work_bytes) {
          set_error("scratch buffer too small for the projection refresh"); return FIRA_ERR_WORKSPACE_TOO_SMALL;
        }
        ptab[k] = tp;
        const fira_status ps = part_gemm_prepare(pjobs[k].data(), nparts, ptab[k], bytes, &ptiles[k], st);
        if (ps != FIRA_OK) return ps;
        tp += bytes;
      }
    int rmax = 0, gparts = 1;
    for (const RefreshMat& m : rms) {
      rmax = std::max(rmax, m.r);
      if (!m.tc) gparts = std::max(gparts, m.Gp.parts);
    }
    // element-wise helpers: blockIdx.y is the matrix, enough blocks for the largest of its kind (at most two per SM)
    long long gmax = 0, ymax = 0, zmax = 0;
    for (const RefreshMat& m : rms) {
      gmax = std::max(gmax, (long long)m.d * m.l);
      ymax = std::max(ymax, (long long)m.d * m.r);
      zmax = std::max(zmax, (long long)m.l * m.r);
    }
    auto ew_grid = [&](long long elements, int per_thread) {
      return dim3((unsigned)std::min<long long>(296, (elements + 256 * per_thread - 1) / (256 * per_thread)), nm);
    };
    const long long umax = (long long)rmax * rmax;
    auto run = [&](int tc_kind, int part_kind) -> fira_status {
      if (nparts) {
        const bool with_g = part_kind == PART_AZ || part_kind == PART_ATY;
        const fira_status ps = part_gemm_run(ptab[part_kind], nparts, ptiles[part_kind], with_g ? gparts : 3, 3, c->status_dev, st);
        if (ps != FIRA_OK) return ps;
      }
      return ntc ? tc_gemm_run(c, tab[tc_kind], ntc, jtiles[tc_kind], st) : FIRA_OK;
    };
    // CholeskyQR of an iterate: Gram product, U = L^-T, application.
    auto orth = [&](int tc_gram, int part_gram, float shift, int tc_apply, int part_apply) -> fira_status {
      fira_status s = run(tc_gram, part_gram);
      if (s != FIRA_OK) return s;
      RF_CUDA(factor_and_invert(rm_dev, nm, rmax, shift, c->status_dev, st));
      return run(tc_apply, part_apply);
    };
    // split: the iterate enters the products with its bf16 remainder and the orthonormalisation has split operands; the
    // last round.  The second pass there brings the basis to fp32 orthonormality and is needed only for the
    // basis that is kept: one pass (deviation about cond^2 times the product's precision) keeps an
    // intermediate iterate well conditioned, which is all the next product asks.
    auto round_y = [&](bool split, bool split_follows) -> fira_status {
      fira_status s = run(split ? JOB_AZ_SPLIT : JOB_AZ, PART_AZ);
      if (s == FIRA_OK)
        s = orth(split ? JOB_GRAM_Y_SPLIT : JOB_GRAM_Y, PART_GRAM_Y, 1e-6f,
                 split ? JOB_APPLY_Y_SPLIT : split_follows ? JOB_APPLY_Y_LO : JOB_APPLY_Y, PART_APPLY_Y);
      if (s == FIRA_OK && split) s = orth(JOB_GRAM_Y2_SPLIT, PART_GRAM_Y2, 0.f, JOB_APPLY_Y2_SPLIT, PART_APPLY_Y2);
      return s;
    };
    auto round_z = [&](bool split) -> fira_status {
      const fira_status s = run(split ? JOB_ATY_SPLIT : JOB_ATY, PART_ATY);
      if (s != FIRA_OK) return s;
      return orth(split ? JOB_GRAM_Z_SPLIT : JOB_GRAM_Z, PART_GRAM_Z, 1e-6f, split ? JOB_APPLY_Z_SPLIT : JOB_APPLY_Z, PART_APPLY_Z);
    };
    if (nparts) k_to_parts<<<ew_grid(gmax, 8), 256, 0, st>>>(rm_dev);
    k_clear_inverse<<<ew_grid(umax, 4), 256, 0, st>>>(rm_dev);
    k_gauss<<<ew_grid(zmax, 4), 256, 0, st>>>(rm_dev);
    fira_status prs = round_y(iters == 0, iters == 1);
    for (int it = 0; it < iters && prs == FIRA_OK; ++it) {
      prs = round_z(it + 1 == iters);
      if (prs == FIRA_OK) prs = round_y(it + 1 == iters, it + 2 == iters);
    }
    if (prs != FIRA_OK) return prs;
    k_store_projection<<<ew_grid(ymax, 4), 256, 0, st>>>(rm_dev);
    RF_CUDA(cudaGetLastError());
    // the next chunk reuses the work area, and the host tables above die here
    RF_CUDA(cudaStreamSynchronize(st));
    pos = q;
  }
  return FIRA_OK;
}

}  // namespace fira
