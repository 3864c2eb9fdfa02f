// tnmc_sample_noalloc: the SIMT sampler of tnmc_sample, run with its per-thread
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
#include "sample_f32_kernel.cuh"
#include "sample_f64_kernel.cuh"

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

// The lattices accepted are those whose plain stacks for one tile (64 samples in FP64, 128 in
// FP32) fit the scratch.
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

// FP32: tnmc_sample's kernel with a grid whose stacks fit the scratch (a padded stack of one
// warp's samples may be up to 1.5 times the plain one, so at least 64 samples fit).
template <int SB, int XBM>
tnmc_status launch_noalloc_f32_block(tnmc::SampleArgs<float> a, int nsm, int max_smem, cudaStream_t stream) {
  using namespace tnmc;
  auto kern = sample_f32_kernel<SB, XBM>;
  const size_t per_sample = f32_stack_floats(a.e.P, a.e.Lx) * sizeof(float);
  int NW = f32_warps(a.e.P, a.e.Lx, SB, 4, (size_t)max_smem);
  while (NW > 1 && (size_t)NW * 8 * SB * per_sample > kNoAllocScratchBytes) NW >>= 1;
  if (NW == 0) {
    tnmc_set_error("sampler needs %zu bytes of shared memory per CTA (device allows %d)",
                   f32_smem(a.e.P, a.e.Lx, SB, 1).total, max_smem);
    return TNMC_E_UNSUPPORTED;
  }
  const size_t smem = f32_smem(a.e.P, a.e.Lx, SB, NW).total;
  TNMC_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  int per_sm = 0;
  TNMC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * NW, smem));
  if (per_sm < 1) per_sm = 1;
  const int64_t tile = (int64_t)NW * 8 * SB;
  int64_t grid = (a.B + tile - 1) / tile;
  if (grid > (int64_t)nsm * per_sm) grid = (int64_t)nsm * per_sm;
  const int64_t fit = (int64_t)(kNoAllocScratchBytes / (tile * per_sample));
  if (grid > fit) grid = fit;
  kern<<<(unsigned)grid, 32 * NW, smem, stream>>>(a);
  TNMC_CUDA_TRY(cudaGetLastError());
  return TNMC_OK;
}

// FP64: one warp per CTA, as tnmc_sample launches it, with a grid whose stacks fit.
template <int LS, int SB>
tnmc_status launch_noalloc_f64_tile(tnmc::SampleArgs<double> a, int nsm, cudaStream_t stream) {
  using namespace tnmc;
  constexpr int S = LS * SB;
  auto kern = sample_f64_kernel<LS, SB>;
  const size_t smem = f64_tile_smem(a.e.P, a.e.Lx, S);
  const size_t per_cta = (size_t)(a.e.Lx + 1) * a.e.P * S * sizeof(double);
  if (smem > 48 * 1024) TNMC_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  int per_sm = 0;
  TNMC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32, smem));
  if (per_sm < 1) per_sm = 1;
  int64_t grid = (a.B + S - 1) / S;
  if (grid > (int64_t)nsm * per_sm) grid = (int64_t)nsm * per_sm;
  const int64_t fit = (int64_t)(kNoAllocScratchBytes / per_cta);   // >= 2: 64 samples fit
  if (grid > fit) grid = fit;
  kern<<<(unsigned)grid, 32, smem, stream>>>(a);
  TNMC_CUDA_TRY(cudaGetLastError());
  return TNMC_OK;
}

tnmc_status launch_noalloc(const tnmc_env* env, int precision, int64_t B, uint64_t seed, uint64_t offset,
                           int8_t* spins, double* logq, double* energy, int32_t* flags, cudaStream_t stream) {
  using namespace tnmc;
  const DeviceEnv& d = env->d;
  tnmc_status st = precision == TNMC_F64 ? check_fit(d, 64, sizeof(double)) : check_fit(d, 128, sizeof(float));
  if (st != TNMC_OK) return st;
  void* scratch = nullptr;
  st = scratch_address(&scratch);
  if (st != TNMC_OK) return st;
  int dev = 0, nsm = 0, max_smem = 0;
  TNMC_CUDA_TRY(cudaGetDevice(&dev));
  TNMC_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  TNMC_CUDA_TRY(cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  if (precision == TNMC_F32) {
    const SampleArgs<float> a{d, d.K32, d.R32, d.fe32, B, seed, offset, nullptr, spins, logq, energy, flags,
                              static_cast<float*>(scratch)};
    return by_f32_block(f32_block(B, d.P, nsm), d.P, [&](auto sb, auto xbm) -> tnmc_status {
      return launch_noalloc_f32_block<decltype(sb)::value, decltype(xbm)::value>(a, nsm, max_smem, stream);
    });
  }
  const SampleArgs<double> a{d, d.M64, d.R64, d.fe, B, seed, offset, nullptr, spins, logq, energy, flags,
                             static_cast<double*>(scratch)};
  switch (f64_tile_samples(B, d.P, nsm)) {
    case 32: return launch_noalloc_f64_tile<8, 4>(a, nsm, stream);
    case 16: return launch_noalloc_f64_tile<8, 2>(a, nsm, stream);
    case 8: return launch_noalloc_f64_tile<8, 1>(a, nsm, stream);
    case 4: return launch_noalloc_f64_tile<4, 1>(a, nsm, stream);
    default: return launch_noalloc_f64_tile<2, 1>(a, nsm, stream);
  }
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
  return launch_noalloc(env, precision, B, seed, sample_offset, spins, logq, energy, flags,
                        static_cast<cudaStream_t>(stream));
}
