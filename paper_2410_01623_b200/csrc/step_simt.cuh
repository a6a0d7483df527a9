// Launch interface of the grouped step kernels that work in fp32 precision (any size, type and pitch).
#pragma once
#include "common.cuh"
#include "part_gemm.cuh"

namespace fira {

constexpr int SIMT_TILE = 128;              // tiles of R (l x r) and of W (m x n)
inline int simt_tiles(long long extent) { return (int)((extent + SIMT_TILE - 1) / SIMT_TILE); }

// The factor k_l from the row sums.
__device__ __forceinline__ float row_factor(const MatDev& mt, int l, const Hyper& hp) {
  float nn = 0.f, rn = 0.f;
  for (int q = 0; q < mt.aux_slots; ++q) { nn += mt.aux[(long long)q * mt.l + l]; rn += mt.aux[(long long)(mt.aux_slots + q) * mt.l + l]; }
  return sqrtf(nn) / (sqrtf(rn) + hp.eps);
}

// Whether the projection's epilogue has made the factors k_l itself: the row sums were complete in one tile.
__device__ __forceinline__ bool factors_ready(const MatDev& mt, const Hyper& hp) {
  return mt.Rp || mt.r <= SIMT_TILE;             // (Rp: k_moments has)
}

inline int psi_of(const Hyper& hp) { return hp.mode & HYPER_PSI_RMSPROP ? PSI_RMSPROP : hp.mode & HYPER_PSI_ADAGRAD ? PSI_ADAGRAD : PSI_ADAM; }
// The direction N of one entry (Eq. 4, or the other base optimizer's) from its updated moments.
template <int PSI>
__device__ __forceinline__ float direction(const Hyper& hp, float bias, float r, float m, float v) {
  return (PSI == PSI_ADAM ? bias * m : r) / (sqrtf(v) + hp.eps);
}
// Updates the moments of one entry (Eq. 2-3; M is left alone by RMSProp and Adagrad) and returns N.
template <int PSI>
__device__ __forceinline__ float adam_direction(const Hyper& hp, float bias, float r, float& m, float& v) {
  v = PSI == PSI_ADAGRAD ? v + r * r : hp.beta2 * v + (1.f - hp.beta2) * r * r;
  if (PSI == PSI_ADAM) m = hp.beta1 * m + (1.f - hp.beta1) * r;
  return direction<PSI>(hp, bias, r, m, v);
}

// Device-resident schedule of one list of matrices.  `list` holds indices into
// `mats`; the *_start arrays have nlist + 1 ascending entries (prefix sums).
struct SimtPlan {
  const MatDev* mats = nullptr;
  const int* list = nullptr;
  int nlist = 0;
  bool chained = false;                  // the kernel in front of the step lets its first kernel in early (short lists)
  const int* proj_tile_start = nullptr;  // 128 x 128 tiles of R (l x r)
  int proj_tiles = 0;
  int max_d = 0, max_r = 0;              // largest d and r of the list
  long long max_proj_units = 0;          // long lists: largest projection, in units of eight entries of its parts
  const int* w_tile_start = nullptr;     // 128 x 128 tiles of W (m x n)
  int w_tiles = 0;
  int resident = 0;                      // short lists: norm, limiter and update in one kernel, on so many blocks at most (short_one_kernel; MatDev::shares are there)
  float* norm_out = nullptr;             //   a single matrix's remembered norm and step count go there as well
  long long* t_out = nullptr;
  const int* npart = nullptr;            // partial sums of ||S||^2 per matrix
  const int* row_start = nullptr;        // rows l (long lists)
  const int* npart_tiles = nullptr;      // the same where there is one per 128 x 128 tile of W
  PartStepPlan parts;                    // long lists: the products with the projection
  std::vector<int> h_row_start;
  // long lists: the matrices whose rows TMA cannot address; their G and W are worked on as copies with an aligned pitch
  const int* stage_list = nullptr;
  const int* stage_start = nullptr;      // rows m
  std::vector<int> h_stage_pos, h_stage_start;   // staged matrices among the first q of the list; their rows
  // host copies of the two prefix arrays (needed only to step a sub-range of the list)
  std::vector<int> h_proj_tile_start, h_w_tile_start;
};

// Whether a list of these matrices (the ones of this engine) is long: its products with the projection then run on
// parts (part_gemm.cu), which R, X and the projection are kept as.
bool simt_long_list(const std::vector<fira_matrix_desc>& list);
// Whether a short list's norm, limiter and update are one kernel: w_tiles 128 x 128 tiles of W in nlist matrices, one block each and one
// more per matrix, all resident at once, one to an SM (resident: how many can be; there is room for the words of SHORT_RESIDENT).
constexpr int SHORT_RESIDENT = 148;
inline bool short_one_kernel(int w_tiles, int nlist, int max_r, int resident = SHORT_RESIDENT) { return nlist > 0 && w_tiles + nlist <= resident && max_r <= 128; }
// SMs that kernels of the stream may run on: the device's, or fewer in a context or on a stream that has a part of them.
int stream_sms(cudaStream_t st);
inline int short_resident(cudaStream_t st) { const int sms = stream_sms(st); return sms < SHORT_RESIDENT ? sms : SHORT_RESIDENT; }
// Copies rows of staged matrices (MatDev Gs, Ws): dir 0 G and W in, 1 W out (step_tc.cu).
void launch_stage(const MatDev* mats, const int* list, int nlist, const int* row_start, int first_row, int rows, int dir, cudaStream_t st);
// Enqueues the phases for the matrices [qa, qb) of the list (qb < 0: the whole list); returns
// the number of launches (negative: error, message set).
int launch_simt_step(const SimtPlan& pl, const Hyper& hp, unsigned* status_dev, cudaStream_t st,
                     PhaseTimer* tm, int qa = 0, int qb = -1);
// The names of the phases that a step of the list marks.
std::vector<const char*> simt_phase_names(const SimtPlan& pl, bool only_scaling);

// One block of 256 threads per matrix of the list: sums the matrix's partial sums
// of ||S||^2 (npart_of[i] floats at mt.part) in a fixed order, applies the limiter
// rule (Eq. 12 in Algorithm 1's form), stores lambda and the new ||S_prev||,
// records the range of k and advances t.
__global__ void k_finalize(const MatDev* __restrict__ mats, const int* __restrict__ list, int nlist,
                           const int* __restrict__ npart_of, Hyper hp, unsigned* __restrict__ status);

// Fira-only-scaling, element-wise over tiles of `tile` x `tile` (at most 256) elements of W (one block
// of 256 threads per tile; tile_start holds nlist + 1 ascending tile counts; `first` is added to the
// block index, `tiles` blocks are launched).  update = 0: part[tile] = sum over the tile of (k_l G)^2, the
// norm that the limiter sees; update = 1: W <- W - lr a_res lambda k_l G.
void launch_scaled_gradient(const MatDev* mats, const int* list, int nlist, const int* tile_start, int first,
                            int tiles, int tile, int update, const Hyper& hp, cudaStream_t st);

}  // namespace fira
