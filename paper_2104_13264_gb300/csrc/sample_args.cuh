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

}  // namespace
}  // namespace tnmc
