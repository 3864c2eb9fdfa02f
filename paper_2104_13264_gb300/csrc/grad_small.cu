// Backward of sum_b w_b log q(s_b) for small bonds and large batches: the sweeps of grad.cu with
// one thread per sample, 128 per CTA (64 while that leaves an SM without two CTAs).
//
// grad.cu's CTA spreads a site's outputs over 16 lanes, of which a bond of 4 uses a quarter at most;
// its time hardly falls with the bond.  One thread per sample does the work of the bond it has, and
// its vectors are rescaled at once, so that strong vertical bonds need nothing of their own.  What bounds it:
// the loads of the vector stacks and the site's barriers.  Measured, ms, here / grad.cu: 16 x 16,
// chi 2, 100000 samples 2.4 / 11.0, 15000 1.1 / 2.1, 6000 1.1 / 1.1; chi 4, 100000 3.0 / 11.1; chi 8,
// 100000 6.1 / 11.6, 40000 3.8 / 5.2, 15000 3.5 / 2.2.
#include <math.h>

#include "common.cuh"

namespace tnmc {
namespace {

struct GradSmallArgs {
  DeviceEnv e;
  const float* L;       // [Ly][Lx][P][2][P]
  const float* fe;      // [Ly][Lx][2]
  int64_t B;
  const int8_t* spins;
  const float* weights;
  float* grad;          // [Ly][Lx][P][2][P], accumulated
  float* scratch;       // per CTA: grad_small_floats
};

// Per CTA of nt samples: three stacks [Lx + 1][P][nt] (R, Lambda, Lbar) and per site w(-), w(+) and
// the exponents of k, k'.
inline size_t grad_small_floats(int P, int Lx, int nt) { return (size_t)3 * (Lx + 1) * P * nt + (size_t)4 * Lx * nt; }

__device__ inline float scale2f(float x, int e) { return scalbnf(x, e); }

// Shared vectors have a stride of kNT + 1 floats (conflict free).  Six CTAs per SM leave 80 (128 samples)
// and 96 (64) registers; the compiler's own choice is 56 and 32 (15000 samples of 16 x 16, chi 2 1.9
// instead of 1.1 ms), eight CTAs 64 and 96 (40000 samples of 32 x 32, chi 8 22.6 instead of 19.4 ms).
template <int kNT>
__global__ void __launch_bounds__(kNT, 6) logq_grad_small_kernel(GradSmallArgs a) {
  constexpr int kSP = kNT + 1;
  extern __shared__ float sm[];
  const int Lx = a.e.Lx, Ly = a.e.Ly, P = a.e.P;
  const int W = (Lx + 31) >> 5;
  const int t = threadIdx.x;
  float* V0 = sm;                        // [P][SP]  Lambda_c (P1)
  float* V2 = V0 + P * kSP;              // [P][SP]  Rbar_c (P2)
  float* V3 = V2 + P * kSP;              // [P][SP]  scratch vector
  float* Y = V3 + P * kSP;               // [2][P][SP]
  float* Z = Y + 2 * P * kSP;            // [2][P][SP]
  uint32_t* bits_prev = reinterpret_cast<uint32_t*>(Z + 2 * P * kSP);   // [W][NT]
  uint32_t* bits_cur = bits_prev + W * kNT;
  const int n = Lx * Ly;
  const size_t stack = (size_t)(Lx + 1) * P * kNT;
  float* Rs = a.scratch + (size_t)blockIdx.x * (3 * stack + 4 * (size_t)Lx * kNT);
  float* Ls = Rs + stack;
  float* LBs = Ls + stack;
  float* w0s = LBs + stack;              // [Lx][NT] raw w(-)
  float* w1s = w0s + (size_t)Lx * kNT;   // [Lx][NT] raw w(+)
  int* ek = reinterpret_cast<int*>(w1s + (size_t)Lx * kNT);    // exponent of k_c (Lambda_{c+1})
  int* ekp = ek + (size_t)Lx * kNT;                           // exponent of k'_c (R_c)
  for (int64_t b0 = (int64_t)blockIdx.x * kNT; b0 < a.B; b0 += (int64_t)gridDim.x * kNT) {
    const int64_t b = b0 + t;
    const bool active = b < a.B;
    const float wt = active ? a.weights[b] : 0.0f;

    for (int wd = 0; wd < W; ++wd) bits_prev[wd * kNT + t] = 0u;
    for (int r = 0; r < Ly; ++r) {
      const int32_t* bond = a.e.bond + r * (Lx + 1);
      const float* fer = a.fe + (size_t)r * Lx * 2;
      for (int wd = 0; wd < W; ++wd) bits_cur[wd * kNT + t] = 0u;
      if (active) {
        const int8_t* src = a.spins + (size_t)b * n + (size_t)r * Lx;
        for (int c = 0; c < Lx; ++c)
          if (src[c] > 0) bits_cur[(c >> 5) * kNT + t] |= 1u << (c & 31);
      }
      auto fval = [&](int c, int s) -> float {
        if (r == 0) return 1.0f;
        const bool up = (bits_prev[(c >> 5) * kNT + t] >> (c & 31)) & 1u;
        return ((up ? 1 : 0) == s) ? fer[2 * c + 1] : fer[2 * c];
      };
      auto spin = [&](int c) -> int { return (bits_cur[(c >> 5) * kNT + t] >> (c & 31)) & 1u; };
      // ---- 1. right sweep ----
      for (int k = 0; k < P; ++k) Rs[((size_t)Lx * P + k) * kNT + t] = (k == 0) ? 1.0f : 0.0f;
      for (int c = Lx - 1; c >= 1; --c) {
        const int dc = bond[c], dc1 = bond[c + 1];
        const float f0 = fval(c, 0), f1 = fval(c, 1);
        const float* M = a.L + ((size_t)r * Lx + c) * P * 2 * P;
        const float* Rn = Rs + (size_t)(c + 1) * P * kNT;
        float mx = 0.0f;
        for (int aa = 0; aa < dc; ++aa) {
          float s0 = 0.0f, s1 = 0.0f;
          for (int bb = 0; bb < dc1; ++bb) {
            const float rb = Rn[bb * kNT + t];
            s0 = fmaf(__ldg(M + ((size_t)aa * 2) * P + bb), rb, s0);
            s1 = fmaf(__ldg(M + ((size_t)aa * 2 + 1) * P + bb), rb, s1);
          }
          const float v = f0 * s0 + f1 * s1;
          V3[aa * kSP + t] = v;
          mx = fmaxf(mx, fabsf(v));
        }
        const int e = (mx > 0.0f) ? -ilogbf(mx) : 0;
        ekp[(size_t)c * kNT + t] = e;
        float* Rc = Rs + (size_t)c * P * kNT;
        for (int aa = 0; aa < P; ++aa) Rc[aa * kNT + t] = (aa < dc) ? scale2f(V3[aa * kSP + t], e) : 0.0f;
      }
      // ---- 2. left sweep (forced) ----
      for (int k = 0; k < P; ++k) Ls[(size_t)k * kNT + t] = (k == 0) ? 1.0f : 0.0f;
      for (int c = 0; c < Lx; ++c) {
        const int dc = bond[c], dc1 = bond[c + 1];
        const float f0 = fval(c, 0), f1 = fval(c, 1);
        const int s = spin(c);
        const float* M = a.L + ((size_t)r * Lx + c) * P * 2 * P;
        const float* Lc = Ls + (size_t)c * P * kNT;
        const float* Rn = Rs + (size_t)(c + 1) * P * kNT;
        float w0 = 0.0f, w1 = 0.0f, mx = 0.0f;
        for (int bb = 0; bb < dc1; ++bb) {
          float u0 = 0.0f, u1 = 0.0f;
          for (int aa = 0; aa < dc; ++aa) {
            const float la = Lc[aa * kNT + t];
            u0 = fmaf(la, __ldg(M + ((size_t)aa * 2) * P + bb), u0);
            u1 = fmaf(la, __ldg(M + ((size_t)aa * 2 + 1) * P + bb), u1);
          }
          const float rb = Rn[bb * kNT + t];
          w0 = fmaf(u0, rb, w0);
          w1 = fmaf(u1, rb, w1);
          const float us = (s ? u1 : u0) * (s ? f1 : f0);
          V3[bb * kSP + t] = us;
          mx = fmaxf(mx, fabsf(us));
        }
        w0s[(size_t)c * kNT + t] = w0 * f0;
        w1s[(size_t)c * kNT + t] = w1 * f1;
        const int e = (mx > 0.0f) ? -ilogbf(mx) : 0;
        ek[(size_t)c * kNT + t] = e;
        float* Ln = Ls + (size_t)(c + 1) * P * kNT;
        for (int bb = 0; bb < P; ++bb) Ln[bb * kNT + t] = (bb < dc1) ? scale2f(V3[bb * kSP + t], e) : 0.0f;
      }
      // per-site weight adjoints g_c(s); a sample with a non-positive normaliser, or with
      // q = 0, contributes nothing (its log q is not differentiable)
      bool ok = wt != 0.0f;
      for (int c = 0; c < Lx && ok; ++c) {
        const float w0 = fmaxf(w0s[(size_t)c * kNT + t], 0.0f), w1 = fmaxf(w1s[(size_t)c * kNT + t], 0.0f);
        const float ws = spin(c) ? w1 : w0;
        ok = (w0 + w1 > 0.0f) && isfinite(w0 + w1) && ws > 0.0f;
      }
      auto gw = [&](int c, int s_) -> float {
        if (!ok) return 0.0f;
        const float w0r = w0s[(size_t)c * kNT + t], w1r = w1s[(size_t)c * kNT + t];
        const float w0 = fmaxf(w0r, 0.0f), w1 = fmaxf(w1r, 0.0f);
        const int sc = spin(c);
        const float ws = sc ? w1 : w0;
        float g = -1.0f / (w0 + w1);
        if (s_ == sc) g += 1.0f / ws;
        const float raw = s_ ? w1r : w0r;
        return (raw > 0.0f) ? wt * g * fval(c, s_) : 0.0f;
      };
      // ---- 4. Lambda adjoint, right to left: LBs[c] = Lbar_c (c = 1..Lx) ----
      for (int k = 0; k < P; ++k) LBs[((size_t)Lx * P + k) * kNT + t] = 0.0f;
      for (int c = Lx - 1; c >= 1; --c) {
        const int dc = bond[c], dc1 = bond[c + 1];
        const int s = spin(c);
        const float g0 = gw(c, 0), g1 = gw(c, 1);
        const float kf = scale2f(1.0f, ek[(size_t)c * kNT + t]) * fval(c, s);
        const float* M = a.L + ((size_t)r * Lx + c) * P * 2 * P;
        const float* Rn = Rs + (size_t)(c + 1) * P * kNT;
        const float* LBn = LBs + (size_t)(c + 1) * P * kNT;
        float* LBc = LBs + (size_t)c * P * kNT;
        for (int aa = 0; aa < P; ++aa) {
          float acc = 0.0f;
          if (aa < dc) {
            for (int bb = 0; bb < dc1; ++bb) {
              const float m0 = __ldg(M + ((size_t)aa * 2) * P + bb), m1 = __ldg(M + ((size_t)aa * 2 + 1) * P + bb);
              const float rb = Rn[bb * kNT + t];
              acc = fmaf(g0 * m0 + g1 * m1, rb, acc);
              acc = fmaf(kf * (s ? m1 : m0), LBn[bb * kNT + t], acc);
            }
          }
          LBc[aa * kNT + t] = acc;
        }
      }
      // ---- 5. R adjoint left to right, and the site gradients ----
      for (int k = 0; k < P; ++k) V2[k * kSP + t] = 0.0f;   // Rbar_0 (unused: R_0 is never formed)
      for (int c = 0; c < Lx; ++c) {
        const int dc = bond[c], dc1 = bond[c + 1];
        const int s = spin(c);
        const float f0 = fval(c, 0), f1 = fval(c, 1);
        const float g0 = gw(c, 0), g1 = gw(c, 1);
        const float kf = scale2f(1.0f, ek[(size_t)c * kNT + t]) * (s ? f1 : f0);
        const float kp = (c >= 1) ? scale2f(1.0f, ekp[(size_t)c * kNT + t]) : 0.0f;
        const float* M = a.L + ((size_t)r * Lx + c) * P * 2 * P;
        const float* Lc = Ls + (size_t)c * P * kNT;
        const float* Rn = Rs + (size_t)(c + 1) * P * kNT;
        const float* LBn = LBs + (size_t)(c + 1) * P * kNT;
        // operands of G_c: P1 = Lambda_c, P2 = Rbar_c, Y_s, Z_s
        for (int k = 0; k < P; ++k) {
          V0[k * kSP + t] = Lc[k * kNT + t];
          const float rb = Rn[k * kNT + t];
          const float lb = (c + 1 < Lx) ? LBn[k * kNT + t] : 0.0f;
          Y[(0 * P + k) * kSP + t] = g0 * rb + (s == 0 ? kf * lb : 0.0f);
          Y[(1 * P + k) * kSP + t] = g1 * rb + (s == 1 ? kf * lb : 0.0f);
          Z[(0 * P + k) * kSP + t] = kp * f0 * rb;
          Z[(1 * P + k) * kSP + t] = kp * f1 * rb;
        }
        __syncthreads();
        // G_c partial over the CTA's samples: thread -> (a, s, b) entries
        float* G = a.grad + ((size_t)r * Lx + c) * P * 2 * P;
        for (int idx = t; idx < dc * 2 * dc1; idx += kNT) {
          const int bb = idx % dc1, s_ = (idx / dc1) & 1, aa = idx / (2 * dc1);
          const float* y = Y + (size_t)(s_ * P + bb) * kSP;
          const float* z = Z + (size_t)(s_ * P + bb) * kSP;
          const float* p1 = V0 + (size_t)aa * kSP;
          const float* p2 = V2 + (size_t)aa * kSP;
          float acc = 0.0f;
          for (int q = 0; q < kNT; ++q) acc = fmaf(p1[q], y[q], fmaf(p2[q], z[q], acc));
          if (acc != 0.0f) atomicAdd(G + ((size_t)aa * 2 + s_) * P + bb, acc);
        }
        __syncthreads();
        // Rbar_{c+1} = sum_s g(s) Lambda_c M_c[s] + k'_c sum_s f(s) M_c[s]^T Rbar_c
        if (c + 1 < Lx) {
          for (int bb = 0; bb < dc1; ++bb) {
            float acc = 0.0f;
            for (int aa = 0; aa < dc; ++aa) {
              const float m0 = __ldg(M + ((size_t)aa * 2) * P + bb), m1 = __ldg(M + ((size_t)aa * 2 + 1) * P + bb);
              acc = fmaf(Lc[aa * kNT + t], g0 * m0 + g1 * m1, acc);
              acc = fmaf(V2[aa * kSP + t], kp * (f0 * m0 + f1 * m1), acc);
            }
            V3[bb * kSP + t] = acc;
          }
          __syncthreads();
          for (int k = 0; k < P; ++k) V2[k * kSP + t] = (k < dc1) ? V3[k * kSP + t] : 0.0f;
        }
        __syncthreads();
      }
      for (int wd = 0; wd < W; ++wd) bits_prev[wd * kNT + t] = bits_cur[wd * kNT + t];
    }
  }
}

}  // namespace
}  // namespace tnmc

namespace tnmc {
namespace {

inline size_t small_smem(int Lx, int P, int nt) {
  return (size_t)7 * P * (nt + 1) * sizeof(float) + (size_t)2 * ((Lx + 31) / 32) * nt * sizeof(uint32_t);
}

template <int kNT>
tnmc_status launch_small(const tnmc_env* env, GradSmallArgs a, int nsm, cudaStream_t stream) {
  const DeviceEnv& d = env->d;
  auto kern = logq_grad_small_kernel<kNT>;
  const size_t smem = small_smem(d.Lx, d.P, kNT);
  TNMC_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  int per_sm = 0;
  TNMC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kNT, smem));
  int64_t grid = (a.B + kNT - 1) / kNT;
  if (grid > (int64_t)nsm * (per_sm < 1 ? 1 : per_sm)) grid = (int64_t)nsm * (per_sm < 1 ? 1 : per_sm);
  tnmc_env* me = const_cast<tnmc_env*>(env);
  const size_t need = (size_t)grid * grad_small_floats(d.P, d.Lx, kNT) * sizeof(float);
  const tnmc_status gs = grow_scratch(me, need, stream, "gradient");
  if (gs != TNMC_OK) return gs;
  a.scratch = static_cast<float*>(me->scratch.ptr);
  kern<<<(unsigned)grid, kNT, smem, stream>>>(a);
  TNMC_CUDA_TRY(cudaGetLastError());
  return TNMC_OK;
}

}  // namespace
}  // namespace tnmc

size_t tnmc_grad_small_smem(int Lx, int P) { return tnmc::small_smem(Lx, P, 128); }

tnmc_status tnmc_launch_logq_grad_small(const tnmc_env* env, int64_t B, const int8_t* spins, const float* weights,
                                        float* grad, int nsm, cudaStream_t stream) {
  using namespace tnmc;
  const DeviceEnv& d = env->d;
  const GradSmallArgs a{d, d.L32, d.fe32, B, spins, weights, grad, nullptr};
  return (B + 127) / 128 < 2 * (int64_t)nsm ? launch_small<64>(env, a, nsm, stream)
                                            : launch_small<128>(env, a, nsm, stream);
}
