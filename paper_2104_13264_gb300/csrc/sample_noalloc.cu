// tnmc_sample_noalloc: the SIMT sampler of tnmc_sample, run with its samples'
// right-vector stacks in a fixed, file-scope device array instead of memory the
// library allocates.
//
// Why: tnmc_sample grows its scratch with cudaMallocAsync / cudaFreeAsync the
// first time it needs more.  Some callers must not have the library allocate:
// code that runs under a fixed device-memory budget owned by another allocator,
// and latency-sensitive loops where an allocation (or the device-wide
// synchronisation a cudaFree implies) is not acceptable.  This entry point
// allocates nothing; the caller still passes every input and output.
//
// The scratch is one static __device__ array of kNoAllocScratchBytes.  Every GPU
// that loads the library holds it until the process exits.  All calls on a device
// share it, and it keeps the previous call's contents: calls that overlap on the
// GPU (two streams, or two threads) race and must be ordered by the caller.  The
// kernel writes every scratch word before it reads it, so nothing has to be
// cleared between calls.
//
// Host code cannot use the array's name as a device address (in host code it is
// a host-side stand-in).  The first call on each device therefore looks the
// address up with cudaGetSymbolAddress while that device is current and caches
// it; make that first call before any stream capture.
#include <mutex>

#include "common.cuh"

namespace {

constexpr size_t kNoAllocScratchBytes = (size_t)64 << 20;   // 64 MiB per device
constexpr int kMaxDevices = 64;

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

std::mutex g_setup_mu;
void* g_scratch_ptr[kMaxDevices] = {};

// Device address of the static scratch on the current device (set-up on first use).
tnmc_status scratch_address(void** out) {
  int dev = 0;
  TNMC_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) {
    tnmc_set_error("device ordinal %d is beyond the %d devices tnmc_sample_noalloc supports", dev, kMaxDevices);
    return TNMC_E_UNSUPPORTED;
  }
  std::lock_guard<std::mutex> lock(g_setup_mu);
  if (!g_scratch_ptr[dev]) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p) {
      tnmc_set_error("cudaGetSymbolAddress of the no-alloc scratch failed on device %d: %s", dev,
                     cudaGetErrorString(e));
      return TNMC_E_CUDA;
    }
    g_scratch_ptr[dev] = p;
  }
  *out = g_scratch_ptr[dev];
  return TNMC_OK;
}

// The lattices accepted are those whose plain stacks for 64 samples in FP64, 128 in FP32, fit the
// scratch.  The launch takes a grid whose stacks fit: at least one CTA does, with at most 64 samples
// (one warp's), whose FP32 stacks are padded to at most 4/3 of the plain ones.
tnmc_status check_fit(const tnmc::DeviceEnv& d, int samples, size_t elem) {
  const size_t need = (size_t)(d.Lx + 1) * d.P * samples * elem;
  if (need > kNoAllocScratchBytes) {
    tnmc_set_error("tnmc_sample_noalloc: %d samples need %zu bytes of scratch for this %d x %d lattice "
                   "(chi padding %d) but the fixed scratch holds %zu bytes; use tnmc_sample",
                   samples, need, d.Ly, d.Lx, d.P, kNoAllocScratchBytes);
    return TNMC_E_INVALID_ARG;
  }
  return TNMC_OK;
}

}  // namespace

extern "C" tnmc_status tnmc_sample_noalloc(const tnmc_env* env, int precision, int64_t B, uint64_t seed,
                                           uint64_t sample_offset, int8_t* spins, double* logq, double* energy,
                                           int32_t* flags, void* stream) {
  tnmc_set_error("%s", "");
  if (!env) {
    tnmc_set_error("env must be non-null");
    return TNMC_E_INVALID_ARG;
  }
  if (B < 0 || (B > 0 && !(spins && logq && energy))) {
    tnmc_set_error("B must be >= 0 and spins, logq, energy non-null");
    return TNMC_E_INVALID_ARG;
  }
  if (precision != TNMC_F64 && precision != TNMC_F32) {
    tnmc_set_error("tnmc_sample_noalloc supports TNMC_F64 and TNMC_F32 only");
    return TNMC_E_UNSUPPORTED;
  }
  if (!(env->precision_mask & (1 << precision))) {
    tnmc_set_error("the env was built without the sampler copy for precision %d", precision);
    return TNMC_E_UNSUPPORTED;
  }
  if (B == 0) return TNMC_OK;
  tnmc_status st = precision == TNMC_F64 ? check_fit(env->d, 64, sizeof(double)) : check_fit(env->d, 128, sizeof(float));
  if (st != TNMC_OK) return st;
  void* scratch = nullptr;
  st = scratch_address(&scratch);
  if (st != TNMC_OK) return st;
  return tnmc_launch_sample_simt(env, precision, B, seed, sample_offset, nullptr, spins, logq, energy, flags, scratch,
                                 kNoAllocScratchBytes, static_cast<cudaStream_t>(stream));
}
