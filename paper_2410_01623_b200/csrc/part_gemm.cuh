// Grouped products of matrices that are stored as bf16 parts, in fp32 precision (see split_gemm.cuh for the
// arithmetic: an fp32 matrix is three bf16 parts, six of the nine part products are taken; a bf16
// matrix is one part).
#pragma once
#include <vector>

#include "common.cuh"

namespace fira {

// A matrix as parts: row-major [parts][rows][pitch], 16-byte aligned, pitch a multiple of 8 elements, or of 64 where the
// products need it along its rows.
struct PartMatrix {
  __nv_bfloat16* base = nullptr;
  long long rows = 0, cols = 0, pitch = 0, part_stride = 0;
  int parts = 0;
};
inline long long part_pitch(long long cols) { return (cols + 63) / 64 * 64; }
inline size_t part_matrix_bytes(long long rows, long long cols, int parts) {
  return align_up((size_t)parts * rows * part_pitch(cols) * 2);
}
inline PartMatrix part_matrix(void* base, long long rows, long long cols, int parts) {
  PartMatrix p;
  p.base = (__nv_bfloat16*)base; p.rows = rows; p.cols = cols; p.pitch = part_pitch(cols);
  p.part_stride = rows * p.pitch; p.parts = parts;
  return p;
}

// C(i, j) = sum_k A(i, k) B(k, j).  a_t: A is stored transposed ([k][i]); b_t: B is ([j][k]).
// The result goes to `c` (fp32, row-major, pitch ldc) or is split into the parts of `out`.
struct PartGemm {
  PartMatrix a, b;
  bool a_t = false, b_t = false;
  float* c = nullptr;
  long long ldc = 0;
  PartMatrix out;
  bool lower = false;       // only the tiles that meet the lower triangle of the result are wanted
  bool upper_b = false;     // B is upper triangular: column j needs k <= j only
};
size_t part_gemm_table_bytes(const PartGemm* jobs, int njobs);
// Builds the tables on the host and uploads them to table_dev (256-byte aligned) on the given stream.
fira_status part_gemm_prepare(const PartGemm* jobs, int njobs, char* table_dev, size_t table_bytes, int* ntiles, cudaStream_t st);
// One grouped launch over the prepared jobs.  a_parts, b_parts: the most parts that an operand of theirs has.
fira_status part_gemm_run(const char* table_dev, int njobs, int ntiles, int a_parts, int b_parts, unsigned* status_dev, cudaStream_t st);

// ---- the three products of the fp32-precision step for long lists: the projection (part_project.cu),
// D = Pi R and D = Pi X (part_back.cu); R, X and Pi are kept as parts.
struct PartStepPlan {
  const char* table = nullptr;      // device; null: the list is short, its products split their operands themselves
  const char* proj_table = nullptr;
  int njobs = 0, ntiles = 0;
  std::vector<int> proj_start;      // 256 x 128 tiles of R, prefix sums over the list
  std::vector<unsigned char> jobs;  // host image of the table's first part: the norm's jobs, then the update's
  std::vector<int> tile_start;      // 256 x 128 tiles of W, prefix sums over the list
  int deep = 0;                     // some rank exceeds split::PROMOTE
  int one_kernel_pairs = 0;         // norm and update in one kernel, on so many CTA pairs (0: two kernels, some matrix has too many tiles)
};
constexpr int PART_STEP_MAX_RANK = 512;    // (k_moments keeps a row of R in registers)
constexpr int PART_SUMS_PER_TILE = 16;   // partial sums of ||S||^2 that a tile leaves
constexpr int PART_SHARE_WORDS = 2;      // or, in their place, marked words of k_part_step
static_assert(PART_SHARE_WORDS * 8 <= PART_SUMS_PER_TILE * 4, "the words fit where the sums would be");
inline int part_rank_pitch(int r) { return (r + 7) / 8 * 8; }
__host__ __device__ inline int part_step_tiles(int m, int n) { return ((m + 255) / 256) * ((n + 127) / 128); }
inline int part_project_tiles(int l, int r) { return ((l + 255) / 256) * ((r + 127) / 128); }
// Whether k_moments forms X (for limiter factor 1): its factors are known row by row.
__host__ __device__ inline bool part_forms_x(const Hyper& hp) { return (hp.mode & HYPER_X_IS_N) || !(hp.mode & (HYPER_MATRIX_SCALING | HYPER_ONLY_SCALING)); }
size_t part_project_table_bytes(int njobs, int ntiles);
fira_status part_project_prepare(const std::vector<MatDev>& mats, const std::vector<int>& list, char* table_dev, PartStepPlan* plan, cudaStream_t st);
fira_status part_project_run(const PartStepPlan& plan, const MatDev* mats_dev, int qa, int qb, unsigned* status_dev, cudaStream_t st);
size_t part_step_table_bytes(int njobs, int ntiles);
// mats: the host copies of the problem table, list: the indices of this engine's matrices in it.
fira_status part_step_prepare(const std::vector<MatDev>& mats, const std::vector<int>& list, char* table_dev, PartStepPlan* plan, cudaStream_t st);
// Called when W / G pointers changed.
fira_status part_step_update_pointers(const std::vector<MatDev>& mats, const std::vector<int>& list, PartStepPlan* plan, cudaStream_t st);
// The norm (update = 0) or the update of the matrices [qa, qb) of the list.
fira_status part_step_run(const PartStepPlan& plan, const MatDev* mats_dev, int qa, int qb, int update, const Hyper& hp,
                          unsigned* status_dev, cudaStream_t st);
// Norm, limiter and update in one kernel (plan.one_kernel_pairs).
fira_status part_step_run_one_kernel(const PartStepPlan& plan, const MatDev* mats_dev, int qa, int qb, const Hyper& hp, unsigned* status_dev, cudaStream_t st);

}  // namespace fira
