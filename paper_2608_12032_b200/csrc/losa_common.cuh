// Shared host/device helpers of liblosa: status word, problem geometry, error macros.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "losa.h"

namespace losa {

// Upper bound on the number of persistent CTAs any kernel here launches; workspace is
// sized for it so that losa_workspace_bytes() needs no GPU.
constexpr int kMaxPersistentCtas = 160;

// Per-device state of the library, created on a device's first call (thread-safe) and kept until
// the process exits: the SM count and the device-visible status word (one int of pinned, mapped
// host memory per device).  Kernels record the first error with a system-scope compare-and-swap;
// the host reads the word after a stream sync.
constexpr int kMaxDevices = 64;
struct DeviceState {
  int ordinal;
  int sm_count;
  int* status_host;
  int* status_dev;  // the same word as the kernels of this device address it
};
// State of the CURRENT device, or nullptr with *rc = LOSA_ERR_UNSUPPORTED (not an sm_100 GPU, or
// a device ordinal beyond kMaxDevices) or LOSA_ERR_CUDA (a runtime call failed).
const DeviceState* device_state(int* rc);
// LOSA_OK if the current device can run the library's kernels (compute capability 10.x); makes no
// allocation.
int check_device();
const char* set_cuda_error(cudaError_t e, const char* what);

// Division by a number that the host knows: the quotient of n < 2^31 is the high word of a product
// (Granlund and Montgomery, "Division by invariant integers using multiplication": mul is 2^(31 + shift) / d rounded
// up, d <= 2^shift < 2 d, so that n mul / 2^(31 + shift) exceeds n / d by less than 1 / d).  A work unit's place takes
// five divisions, one behind the other, that every one of its warps waits for.
struct Divisor {
  uint32_t d, mul, shift;
  Divisor() = default;
  explicit Divisor(uint32_t by) : d(by), mul(0), shift(0) {
    while ((1ull << shift) < d) ++shift;
    mul = (uint32_t)(((1ull << (31 + shift)) + d - 1) / d);
  }
  __device__ __forceinline__ int div(int n) const { return (int)(__umulhi((uint32_t)n << 1, mul) >> shift); }
  __device__ __forceinline__ int divmod(int n, int& rest) const {
    const int q = div(n);
    rest = n - q * (int)d;
    return q;
  }
};

__device__ __forceinline__ void report_error(int* status, int code) {
  atomicCAS_system(status, 0, code);
}

struct Geometry {
  int B, H, N, D, R, C;
  int nQb, nKb;
  int nQt;     // 128-row query tiles per head
  int nPairs;  // pairs of query tiles per head (one CTA work item)
  int64_t sb, sh, sn;
  float scale;
};

int make_geometry(const losa_problem_t* p, Geometry* g);  // LOSA_OK or an error code

#define LOSA_CUDA_TRY(expr)                                        \
  do {                                                             \
    cudaError_t e__ = (expr);                                      \
    if (e__ != cudaSuccess) {                                      \
      ::losa::set_cuda_error(e__, #expr);                          \
      return LOSA_ERR_CUDA;                                        \
    }                                                              \
  } while (0)

// Launches `kern`; `dependent`: it may be scheduled before the kernel ahead of it in the stream has
// finished, and waits for it itself (grid_dependency_wait).
template <typename... P, typename... A>
int launch(void (*kern)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, bool dependent, const A&... args) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = dependent ? 1 : 0;
  LOSA_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, args...));
  return LOSA_OK;
}

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// ---- entry points of the kernel translation units (host launchers) -------------------

size_t select_workspace_bytes(int64_t rows, int nKb);
int select_launches(int64_t rows, int nKb, bool fixed);  // kernels that such a call launches
int launch_select(int rows, int nKb, const float* mass, double tau, int fixed_count,
                  int32_t* offsets, int32_t* kv_idx, int64_t kv_capacity, void* ws, int* status,
                  int dev, cudaStream_t st);  // fixed_count > 0: keep that many blocks per row instead;
                                              // status: device-visible word that receives device-side errors
int launch_row_recall(int rows, int nKb, const float* mass, const int32_t* offsets,
                      const int32_t* kv_idx, double* retained, double* total, cudaStream_t st);
size_t select_noalloc_workspace_limit();
int launch_select_noalloc(int rows, int nKb, const float* mass, double tau, int32_t* offsets,
                          int32_t* kv_idx, int64_t kv_capacity, int32_t* device_status,
                          cudaStream_t st);
int launch_validate_csr(int rows, int nKb, const int32_t* offsets, const int32_t* kv_idx,
                        cudaStream_t st);

enum AttnMode { kDense = 0, kSparse = 1, kMass = 2, kFused = 3 };  // kFused: dense O and mass

size_t attn_workspace_bytes(AttnMode mode, const Geometry& g, int n_prob = 1);
void arm_stalled_launch(uint32_t polls);  // the next attention launch publishes no work (diagnostic)
int attn_work_slots(AttnMode mode, const Geometry& g, const DeviceState& dev);
int attn_launches(AttnMode mode, const Geometry& g, const DeviceState& dev);
int launch_attn(AttnMode mode, const Geometry& g, const void* q, const void* k, const void* v,
                const int32_t* offsets, const int32_t* kv_idx, void* o, int o_dtype, float* mass,
                float* lse, void* ws, cudaStream_t st, int n_prob = 1,
                const losa_layer_t* layers = nullptr);

}  // namespace losa
