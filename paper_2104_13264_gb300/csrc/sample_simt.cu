// SIMT sampler / evaluator of q = pi~ (Sec. 2, eqs. bayes, pi-approx, tns-prior;
// App. A) in FP64 or FP32, and the kernel that derives the sampler copies of the
// environment.
//
// For every row r a sample
//   (right sweep) builds R_{Lx} = 1, R_c = sum_s f_c(s) M_c[:, s, :] R_{c+1}
//                 for c = Lx-1 .. 1, each rescaled by a power of two and pushed
//                 to a stack in global scratch;
//   (left sweep)  walks c = 0 .. Lx-1:  U[s] = Lambda_c M_c[:, s, :],
//                 w(s) = f_c(s) <U[s], R_{c+1}>, clamps at 0, normalises,
//                 draws the spin from the 64-bit Philox word (or reads it in
//                 forced mode), accumulates log q, and sets
//                 Lambda_{c+1} = f_c(s) U[s], rescaled by a power of two.
// f_c(s) = exp(beta Jv[r-1][c] s_{r-1,c} s) carries the (exactly contracted)
// product state of the rows above.  On the odd rows of the snake order the two sweeps
// change roles (draws from the right).  The kernels are in sample_f64_kernel.cuh (launched from
// sample_f64.cu) and sample_f32_kernel.cuh.
#include <math.h>

#include "common.cuh"
#include "sample_f32_kernel.cuh"

namespace tnmc {
namespace {

// Sampler copies: L (same layout as M64), R ([b][a][s]), K ([a][b][s]) and the field table.
template <typename T>
__global__ void derive_kernel(DeviceEnv e, T* L, T* R, T* K, size_t ntens) {
  const int P = e.P;
  const size_t per = (size_t)P * 2 * P;
  const size_t total = ntens * per;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
    const size_t t = i / per;
    const int rem = (int)(i % per);
    const int b = rem % P, s = (rem / P) & 1, aa = rem / (2 * P);
    const T v = (T)e.M64[i];
    if (L) L[i] = v;
    R[t * per + ((size_t)b * P + aa) * 2 + s] = v;
    if (K) K[t * per + ((size_t)aa * P + b) * 2 + s] = v;
  }
}

__global__ void fields_kernel(DeviceEnv e, double* fe, float* fe32) {
  const int Lx = e.Lx, Ly = e.Ly;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < Lx * Ly; i += gridDim.x * blockDim.x) {
    const int r = i / Lx, c = i % Lx;
    double d = 1.0, s = 1.0;
    if (r > 0) {
      const double jv = e.Jv[(r - 1) * Lx + c];
      d = exp(-e.beta * jv);
      s = exp(e.beta * jv);
    }
    fe[2 * i] = d;
    fe[2 * i + 1] = s;
    fe32[2 * i] = (float)d;
    fe32[2 * i + 1] = (float)s;
  }
}

// FP32: CTAs of up to 4 warps, 8 SB samples per warp (f32_plan).
template <int SB, int XBM, bool EDGE>
tnmc_status launch_sample_f32(const SimtScratch& scr, SampleArgs<float> a, const F32Plan& p, int nsm,
                              cudaStream_t stream) {
  auto kern = sample_f32_kernel<SB, XBM, EDGE>;
  TNMC_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.smem));
  int per_sm = 0;
  TNMC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * p.NW, p.smem));
  if (per_sm < 1) per_sm = 1;
  const int64_t tile = (int64_t)p.NW * 8 * SB;
  int64_t grid = (a.B + tile - 1) / tile;
  if (grid > (int64_t)nsm * per_sm) grid = (int64_t)nsm * per_sm;
  void* scratch = nullptr;
  const tnmc_status st =
      take_scratch(scr, grid, (size_t)tile * f32_stack_floats(a.e.P, a.e.Lx) * sizeof(float), stream, &scratch);
  if (st != TNMC_OK) return st;
  a.scratch = static_cast<float*>(scratch);
  kern<<<(unsigned)grid, 32 * p.NW, p.smem, stream>>>(a);
  TNMC_CUDA_TRY(cudaGetLastError());
  return TNMC_OK;
}

}  // namespace
}  // namespace tnmc

tnmc_status tnmc_launch_derive(tnmc_env* env, int mask, cudaStream_t stream) {
  using namespace tnmc;
  DeviceEnv& d = env->d;
  const size_t ntens = (size_t)d.Lx * d.Ly;
  fields_kernel<<<256, 256, 0, stream>>>(d, const_cast<double*>(d.fe), const_cast<float*>(d.fe32));
  TNMC_CUDA_TRY(cudaGetLastError());
  derive_kernel<double><<<1024, 256, 0, stream>>>(d, nullptr, const_cast<double*>(d.R64), nullptr, ntens);
  TNMC_CUDA_TRY(cudaGetLastError());
  if (mask & (1 << TNMC_F32)) {
    derive_kernel<float><<<1024, 256, 0, stream>>>(d, const_cast<float*>(d.L32), const_cast<float*>(d.R32),
                                                   const_cast<float*>(d.K32), ntens);
    TNMC_CUDA_TRY(cudaGetLastError());
  }
  return TNMC_OK;
}

namespace tnmc {
namespace {
// FP32 copies [b][a][s] and [a][b][s] from the left layout [a][s][b]
__global__ void rederive_f32_kernel(const float* L, float* R, float* K, int P, size_t ntens) {
  const size_t per = (size_t)P * 2 * P;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < ntens * per; i += (size_t)gridDim.x * blockDim.x) {
    const size_t t = i / per;
    const int rem = (int)(i % per);
    const int b = rem % P, s = (rem / P) & 1, aa = rem / (2 * P);
    const float v = L[i];
    R[t * per + ((size_t)b * P + aa) * 2 + s] = v;
    K[t * per + ((size_t)aa * P + b) * 2 + s] = v;
  }
}
}  // namespace
}  // namespace tnmc

tnmc_status tnmc_launch_rederive_f32(tnmc_env* env, cudaStream_t stream) {
  using namespace tnmc;
  DeviceEnv& d = env->d;
  rederive_f32_kernel<<<1024, 256, 0, stream>>>(d.L32, const_cast<float*>(d.R32), const_cast<float*>(d.K32), d.P,
                                                (size_t)d.Lx * d.Ly);
  TNMC_CUDA_TRY(cudaGetLastError());
  return TNMC_OK;
}

tnmc_status tnmc_launch_sample_simt(const tnmc_env* env, int precision, int64_t B, uint64_t seed, uint64_t offset,
                                    const int8_t* spins_in, int8_t* spins_out, double* logq, double* energy,
                                    int32_t* flags, void* fixed_scratch, size_t fixed_bytes, cudaStream_t stream) {
  using namespace tnmc;
  const DeviceEnv& d = env->d;
  if (B == 0) return TNMC_OK;
  const SimtScratch scr{env, fixed_scratch, fixed_bytes};
  int dev = 0, nsm = 0, max_smem = 0, smem_sm = 0;
  TNMC_CUDA_TRY(cudaGetDevice(&dev));
  TNMC_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  TNMC_CUDA_TRY(cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  TNMC_CUDA_TRY(cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev));
  if (precision == TNMC_F64)
    return tnmc_launch_sample_f64(env, B, seed, offset, spins_in, spins_out, logq, energy, flags, fixed_scratch,
                                  fixed_bytes, nsm, smem_sm, stream);
  const SampleArgs<float> a{d, d.K32, d.R32, d.fe32, B, seed, offset, spins_in, spins_out, logq, energy, flags, nullptr};
  const size_t stack = f32_stack_floats(d.P, d.Lx) * sizeof(float);
  const F32Plan p = f32_plan(
      B, d.P, d.strong, nsm, (size_t)max_smem, (size_t)smem_sm,
      [&](int SB, int NW, bool edge) { return f32_smem(d.P, d.Lx, SB, NW, edge).total; },
      [&](int SB) {      // a CTA's stacks have to fit a fixed scratch
        int NW = 4;
        while (fixed_scratch && NW > 1 && (size_t)NW * 8 * SB * stack > fixed_bytes) NW >>= 1;
        return NW;
      });
  if (p.NW == 0) {
    tnmc_set_error("sampler needs %zu bytes of shared memory per CTA (device allows %d)", p.smem, max_smem);
    return TNMC_E_UNSUPPORTED;
  }
  return by_f32_block(p, d.P, [&](auto sb, auto xbm, auto edge) -> tnmc_status {
    return launch_sample_f32<decltype(sb)::value, decltype(xbm)::value, decltype(edge)::value>(scr, a, p, nsm, stream);
  });
}

tnmc_status tnmc_launch_sample(const tnmc_env* env, int precision, int64_t B, uint64_t seed, uint64_t offset,
                               const int8_t* spins_in, int8_t* spins_out, double* logq, double* energy,
                               int32_t* flags, cudaStream_t stream) {
  if (B == 0) return TNMC_OK;
  if (precision == TNMC_F64 || precision == TNMC_F32)
    return tnmc_launch_sample_simt(env, precision, B, seed, offset, spins_in, spins_out, logq, energy, flags, nullptr,
                                   0, stream);
  if (precision == TNMC_BF16)
    return tnmc_launch_sample_tc(env, B, seed, offset, spins_in, spins_out, logq, energy, flags, stream);
  tnmc_set_error("unknown precision %d", precision);
  return TNMC_E_UNSUPPORTED;
}
