// Arguments of the sampler kernels (FP64 and FP32), shared by the translation units that
// launch them.
#pragma once

#include "common.cuh"

namespace tnmc {
namespace {

template <typename T>
struct SampleArgs {
  DeviceEnv e;
  const T* L;     // FP64: [Ly][Lx][P][2][P] (M64); FP32: [Ly][Lx][P][P][2], [a][b][s] (K32)
  const T* Rt;    // [Ly][Lx][P][P][2]
  const T* fe;    // [Ly][Lx][2]
  int64_t B;
  uint64_t seed, offset;
  const int8_t* spins_in;   // forced mode when non-null
  int8_t* spins_out;        // may be null in forced mode
  double* logq;
  double* energy;
  int32_t* flags;
  T* scratch;               // per CTA: the right-vector stacks of its samples, [Lx+1][P] each
};

// Scratch of a launch: the caller's fixed bytes, or the env's, grown as needed.
struct SimtScratch {
  const tnmc_env* env;
  void* fixed;
  size_t bytes;
};

// The largest grid of at most `grid` CTAs whose stacks (per_cta bytes each) the scratch holds.
inline tnmc_status take_scratch(const SimtScratch& s, int64_t& grid, size_t per_cta, cudaStream_t stream, void** out) {
  if (s.fixed) {
    const int64_t fit = (int64_t)(s.bytes / per_cta);
    if (grid > fit) grid = fit;
    *out = s.fixed;
    return TNMC_OK;
  }
  tnmc_env* me = const_cast<tnmc_env*>(s.env);
  const tnmc_status st = grow_scratch(me, (size_t)grid * per_cta, stream, "sampler");
  *out = me->scratch.ptr;
  return st;
}

}  // namespace
}  // namespace tnmc
