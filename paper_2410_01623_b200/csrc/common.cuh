// Shared declarations of the Fira library's translation units: the per-matrix
// device table and small device helpers.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "../../include/fira.h"

namespace fira {

// Scalars kept per matrix in the state buffer.  prev_norm and t are optimizer
// state (the "+1" of the paper's comparison table and the step count); the rest
// are diagnostics of the latest step.
struct MatScalars {
  float prev_norm;    // ||S_prev|| after limiting; < 0 means "not set yet"
  float lambda;       // limiter factor of the latest step
  float norm_scaled;  // ||S|| before the limiter
  float k_min, k_max;
  float bias;         // bias factor sqrt(1-b2^s)/(1-b1^s) of the latest step (bf16 engine; nothing reads it)
  long long t;        // steps taken
};
static_assert(sizeof(MatScalars) == 32, "MatScalars layout");

// The bias factor that k_finalize works out ahead for the step after, while it waits (in double it costs a microsecond), and
// the step it is for: whoever takes it compares that with the step count in the state buffer, whose bytes the caller may
// have changed since, and makes his own if they differ.
struct BiasSlot {
  long long step;
  float next;         // the factor of `step`
  float now;          // long lists of fp32 precision: the factor of the running step
  float prev;         // norm and update in one kernel: the remembered norm before the step, left by a kernel in front of it (the state's is stored anew by a block that others are not ordered before)
};

// One entry of the device-resident problem table.  l = max(m,n) indexes the
// unprojected extent, d = min(m,n) the projected one.
struct MatDev {
  void* W;
  const void* G;
  void* P;            // d x r, row major, dtype
  float* M;           // l x r
  float* V;           // l x r
  MatScalars* sc;
  BiasSlot* bias;     // scratch, outside the area that the refresh uses
  float* Rt;          // scratch: l x r fp32 low-rank gradient (transposed layout)
  float* Xt;          // scratch: l x r fp32 N
  __nv_bfloat16* Rp;  //   "      long lists (PartStepPlan): R and X as three bf16 parts [3][l][rp_pitch]
  __nv_bfloat16* Xp;
  __nv_bfloat16* Pp;  //   "      the projection as parts [3 or 1][d][pp_pitch]
  int rp_pitch, pp_pitch;
  int aux_slots;      // row sums per l in aux
  float* kvec;        // scratch: l factors
  float* part;        // scratch: partial sums of ||S||^2
  unsigned long long* shares;   //   "      short lists that step in one kernel after the projection: marked words, two per tile of W
  float* aux;         // scratch: row sums [aux_slots][l] of ||N_l||^2, then of ||R_l||^2 (engine 0, short lists: one slot per tile of r)
  __nv_bfloat16* Nb;  // scratch of the tensor-core path: l x r bf16 N
  __nv_bfloat16* Rb;  //   "      l x r bf16 R
  __nv_bfloat16* Xb;  //   "      l x r bf16 X
  float* colpart;     //   "      per (r-tile, l) partial sums of N^2 and R^2, then per-l sums of G^2
  void* Gs;           //   "      copies of G and W with 16-byte aligned rows (pitch lds), only when the
  void* Ws;           //          caller's rows are not (odd widths): TMA needs aligned rows
  long long lds;
  long long ld;
  int m, n, r;
  int left;           // 1: m <= n (left projection), 0: right projection
  int bf16;           // storage type of W, G, P
  int engine;         // 0 fp32 precision, any size (step_simt.cu), 1 bf16 (step_tc.cu)
  int l, d;
};

struct Hyper {
  float beta1, beta2, eps, lr, a_low, a_res, gamma;
  unsigned mode;      // HYPER_* bits: ablation variants (Section 5.4)
};
enum HyperMode : unsigned {
  HYPER_MATRIX_SCALING = 1u,   // one factor per matrix (Eq. 9)
  HYPER_NO_SCALING = 2u,       // factor 1
  HYPER_NO_RESIDUAL = 4u,      // no residual term (Eq. 6)
  HYPER_PSI_RMSPROP = 8u,      // base optimizer: RMSProp instead of Adam
  HYPER_PSI_ADAGRAD = 16u,     // base optimizer: Adagrad instead of Adam
  HYPER_X_IS_N = 64u,          // k_moments (with a_low = 1, a_res = 0): X = N, whatever the variant
  HYPER_ONLY_SCALING = 32u,    // Fira-only-scaling: W <- W - lr phi(R) G (no P N term, S = G diag k)
};

// sqrt(1 - b2^s) / (1 - b1^s) (Eq. 4), in double.
__device__ __forceinline__ float bias_factor(float beta1, float beta2, long long s) {
  return (float)(sqrt(1.0 - pow((double)beta2, (double)s)) / (1.0 - pow((double)beta1, (double)s)));
}
// The factor of step s.  (A call: the arithmetic inline cost the projection its registers.)
__device__ __noinline__ inline float bias_factor_call(float beta1, float beta2, long long s) { return bias_factor(beta1, beta2, s); }
__device__ __forceinline__ float step_bias(const BiasSlot& slot, long long s, const Hyper& hp) {
  return slot.step == s ? slot.next : bias_factor_call(hp.beta1, hp.beta2, s);
}

enum DeviceStatusBits : unsigned {
  DEV_STATUS_TIMEOUT = 1u,
  DEV_STATUS_NONFINITE = 2u,
};

// The base optimizers, as template parameters of the projection's epilogues (Adam: Eq. 2-4).
enum { PSI_ADAM = 0, PSI_RMSPROP = 1, PSI_ADAGRAD = 2 };

template <typename T>
__device__ __forceinline__ float to_float(T v);
template <>
__device__ __forceinline__ float to_float<float>(float v) { return v; }
template <>
__device__ __forceinline__ float to_float<__nv_bfloat16>(__nv_bfloat16 v) {
  return __bfloat162float(v);
}
template <typename T>
__device__ __forceinline__ T from_float(float v);
template <>
__device__ __forceinline__ float from_float<float>(float v) { return v; }
template <>
__device__ __forceinline__ __nv_bfloat16 from_float<__nv_bfloat16>(float v) {
  return __float2bfloat16_rn(v);
}

// Index of the matrix whose tile range contains `tile`: the largest i with
// start[i] <= tile (start has count + 1 ascending entries).
__device__ __forceinline__ int find_matrix(const int* __restrict__ start, int count, int tile) {
  int lo = 0, hi = count;
  while (hi - lo > 1) {
    int mid = (lo + hi) >> 1;
    if (start[mid] <= tile) lo = mid; else hi = mid;
  }
  return lo;
}

void set_error(const std::string& msg);

// Launches a kernel in clusters of `cluster` blocks (1: none, or the kernel's own).  chained: every block of the kernel
// calls ptx::grid_wait, and its blocks may start while the kernel in front of it in the stream is still running: between
// two short kernels that saves 3 to 5 us.
// RESIDENT: blocks of the grid wait for one another: it starts when all of it fits on the device (a cooperative launch), whatever
// else runs there.
template <bool RESIDENT, typename... P, typename... A>
inline cudaError_t launch_with(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, bool chained, int cluster, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = dim3((unsigned)threads); cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute at[3];
  unsigned n = 0;
  if (RESIDENT) { at[n].id = cudaLaunchAttributeCooperative; at[n].val.cooperative = 1; ++n; }
  if (chained) { at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization; at[n].val.programmaticStreamSerializationAllowed = 1; ++n; }
  if (cluster > 1) {
    at[n].id = cudaLaunchAttributeClusterDimension;
    at[n].val.clusterDim.x = (unsigned)cluster; at[n].val.clusterDim.y = 1; at[n].val.clusterDim.z = 1;
    ++n;
  }
  cfg.attrs = at; cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}
template <typename... P, typename... A>
inline cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, bool chained, int cluster, A... args) {
  return launch_with<false>(kernel, grid, threads, smem, st, chained, cluster, args...);
}
template <typename... P, typename... A>
inline cudaError_t launch_resident(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, bool chained, int cluster, A... args) {
  return launch_with<true>(kernel, grid, threads, smem, st, chained, cluster, args...);
}

// Optional per-kernel timing of a step: marks are CUDA events recorded between the
// launches.  slot = the step's row of the event ring, next = the next mark.
struct PhaseTimer {
  bool on = false;
  std::vector<cudaEvent_t> events;   // FIRA_TIMING_MAX_STEPS x (FIRA_TIMING_MAX_PHASES + 1)
  std::vector<const char*> names;    // phase names in launch order
  int slot = 0, next = 0;
  long long steps = 0;               // steps recorded since enabling
  void begin_step() { next = 0; slot = (int)(steps % FIRA_TIMING_MAX_STEPS); }
  void mark(cudaStream_t st) {
    if (!on || next > FIRA_TIMING_MAX_PHASES) return;
    cudaEventRecord(events[(size_t)slot * (FIRA_TIMING_MAX_PHASES + 1) + next], st);
    ++next;
  }
};

inline size_t align_up(size_t x, size_t a = 256) { return (x + a - 1) / a * a; }

}  // namespace fira
