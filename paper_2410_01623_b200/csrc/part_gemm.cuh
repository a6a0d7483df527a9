// Grouped products of matrices that are stored as bf16 parts, in fp32 precision (see split_gemm.cuh for the
// arithmetic: an fp32 matrix is three bf16 parts, six of the nine part products are taken; a bf16
// matrix is one part).
#pragma once
#include <vector>

#include "common.cuh"

namespace fira {

// A matrix as parts: row-major [parts][rows][pitch], pitch a multiple of 64 elements, 16-byte aligned.
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

}  // namespace fira
