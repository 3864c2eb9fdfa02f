// Launch of the FP64 sampler / evaluator (sample_f64_kernel.cuh) on one lattice.
#include "common.cuh"
#include "sample_f64_kernel.cuh"

namespace tnmc {
namespace {

// FP64: one warp per CTA, S samples per warp (f64_plan).
template <int LS, int SB, bool EDGE>
tnmc_status launch_sample_f64(const SimtScratch& scr, SampleArgs<double> a, size_t smem, int nsm, cudaStream_t stream) {
  constexpr int S = LS * SB;
  auto kern = sample_f64_kernel<LS, SB, EDGE>;
  if (smem > 48 * 1024) TNMC_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  int per_sm = 0;
  TNMC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32, smem));
  if (per_sm < 1) per_sm = 1;
  int64_t grid = (a.B + S - 1) / S;
  if (grid > (int64_t)nsm * per_sm) grid = (int64_t)nsm * per_sm;
  void* scratch = nullptr;
  const tnmc_status st = take_scratch(scr, grid, (size_t)(a.e.Lx + 1) * a.e.P * S * sizeof(double), stream, &scratch);
  if (st != TNMC_OK) return st;
  a.scratch = static_cast<double*>(scratch);
  kern<<<(unsigned)grid, 32, smem, stream>>>(a);
  TNMC_CUDA_TRY(cudaGetLastError());
  return TNMC_OK;
}

}  // namespace
}  // namespace tnmc

tnmc_status tnmc_launch_sample_f64(const tnmc_env* env, int64_t B, uint64_t seed, uint64_t offset,
                                   const int8_t* spins_in, int8_t* spins_out, double* logq, double* energy,
                                   int32_t* flags, void* fixed_scratch, size_t fixed_bytes, int nsm, int smem_sm,
                                   cudaStream_t stream) {
  using namespace tnmc;
  const DeviceEnv& d = env->d;
  const SimtScratch scr{env, fixed_scratch, fixed_bytes};
  const SampleArgs<double> a{d, d.M64, d.R64, d.fe, B, seed, offset, spins_in, spins_out, logq, energy, flags, nullptr};
  const F64Plan p =
      f64_plan(B, d.P, nsm, (size_t)smem_sm, [&](int S, bool edge) { return f64_tile_smem(d.P, d.Lx, S, edge); });
  return by_f64_tile(p, [&](auto ls, auto sb, auto edge) -> tnmc_status {
    return launch_sample_f64<decltype(ls)::value, decltype(sb)::value, decltype(edge)::value>(scr, a, p.smem, nsm, stream);
  });
}
