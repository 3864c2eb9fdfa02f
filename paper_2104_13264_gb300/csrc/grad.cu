// Backward of sum_b w_b log q(s_b) with respect to every environment tensor
// M^(r)_c (the FP32 sampler copy), by reverse-mode differentiation of the forced
// evaluation (Sec. 2, eq. pi-approx; App. A): per-site normalised, clamped
// conditionals, power-of-two rescalings treated as constants.
//
// Per row r and sample:
//   1. forward right sweep  R_c = k'_c sum_s f_c(s) M_c[s] R_{c+1}      (stack)
//   2. forward left sweep   Lambda_{c+1} = k_c f_c(s_c) Lambda_c M_c[s_c]   (stack),
//      raw weights w_c(s) = f_c(s) <Lambda_c M_c[s], R_{c+1}>
//   3. g_c(s) = d/dw_c(s) [w log w_c(s_c) - w log(w_+ + w_-)] f_c(s), zero where clamped
//   4. right-to-left adjoint of Lambda (stack):
//        Lbar_c = sum_s M_c[s] Y_s,  Y_s = g_c(s) R_{c+1} + [s = s_c] k_c f_c(s) Lbar_{c+1}
//   5. left-to-right adjoint of R and the gradient of site c:
//        Rbar_{c+1} = sum_s M_c[s]^T V_s,  V_s = g_c(s) Lambda_c + k'_c f_c(s) Rbar_c
//        G_c[a,s,b] += sum_t V_s[a] R_{c+1}[b] + W_s[a] Lbar_{c+1}[b],
//          W_s = [s = s_c] k_c f_c(s) Lambda_c
//
// A CTA of 4 warps owns 32 samples.  Its 128 threads are 8 sample lanes (4 samples each) x 16
// output lanes, so every sweep is a register-blocked product whose operands come from shared
// memory (vectors, and site tensors through a cp.async ring); the site gradient is a
// (2 chi x 32) . (32 x chi) product over the CTA's samples with up to 8 x 8 outputs per thread,
// added to global memory by vector reductions.  One __syncthreads per site and sweep: vectors
// ping-pong between two buffer sets, and a sample's rescaling uses the previous vector's
// largest entry.  The stacks are read back by the threads that wrote them.
//
// What bounds it: shared-memory words (8 per 16 FMAs in the sweeps at chi = 32) and, for
// batches of a few thousand samples, the barrier and load latencies of 2 CTAs per SM.  One
// thread per sample without register blocks took 67 ms for 12 x 48, chi = 32, 8192 samples;
// this form takes 5.3 ms (11.6 TFLOP/s).
#include <math.h>

#include "common.cuh"
#include "sample_f32_kernel.cuh"

namespace tnmc {
namespace {

constexpr int kGT = 32;              // samples per CTA
constexpr int kGThreads = 128;
constexpr int kGStride = kGT + 4;    // floats per vector row (16 B aligned, rows 4 banks apart)

struct GradArgs {
  DeviceEnv e;
  const float* K;       // [Ly][Lx][P][P][2]  [a][b][s]
  const float* Rt;      // [Ly][Lx][P][P][2]  [b][a][s]
  const float* fe;      // [Ly][Lx][2]
  int64_t B;
  const int8_t* spins;
  const float* weights;
  float* grad;          // [Ly][Lx][P][2][P], accumulated
  float* scratch;       // per CTA: grad_cta_floats
};

// Per CTA: three stacks [Lx + 1][P][kGT] (R, Lambda, Lbar) and per site and sample w / g of
// both spins and the exponents of k, k'.
inline __host__ __device__ size_t grad_cta_floats(int P, int Lx) {
  return (size_t)3 * (Lx + 1) * P * kGT + (size_t)4 * Lx * kGT;
}

// Shared memory: the tensor ring, two buffer sets of 6 P vector rows, partial maxima and
// weights, spin masks of the row, sample flags, and if `staged` the row's field factors and
// bond dimensions.
struct GradSmem {
  int nbuf;
  size_t set, mpart, wpart, fer, bond, mask, ok, total;
};
inline __host__ __device__ GradSmem grad_smem(int P, int Lx, bool staged) {
  GradSmem m;
  m.nbuf = P > 32 ? 2 : 3;
  size_t o = ((size_t)m.nbuf * P * 2 * P + 128) * sizeof(float);
  m.set = o;
  o += (size_t)2 * 6 * P * kGStride * sizeof(float);
  m.mpart = o;
  o += (size_t)2 * 4 * kGT * sizeof(float);
  m.wpart = o;
  o += (size_t)2 * 4 * 2 * kGT * sizeof(float);
  m.mask = o;
  o += (size_t)2 * Lx * sizeof(uint32_t);
  m.ok = o;
  o += kGT * sizeof(int);
  m.fer = o;
  if (staged) o += (size_t)2 * Lx * sizeof(float);
  m.bond = o;
  if (staged) o += (size_t)(Lx + 1) * sizeof(int);
  m.total = o;
  return m;
}

// f(IntF<XB>): outputs per thread for dX outputs on 16 output lanes
template <class F>
__device__ __forceinline__ void by_outputs(int dX, F&& f) {
  if (dX <= 16) f(IntF<1>{});
  else if (dX <= 32) f(IntF<2>{});
  else if (dX <= 48) f(IntF<3>{});
  else f(IntF<4>{});
}

__device__ __forceinline__ void load4(const float* p, float (&v)[4]) { load_run<4>(p, v); }

// acc[s][j][b] = sum_k M[k][x0 + j][s] X[k][b]  (x0 = XB ol)
template <int XB>
__device__ __forceinline__ void contract_out(const float* M, int P, int dK, const float* X, int ol, int sl,
                                             float (&acc)[2][XB][4]) {
#pragma unroll
  for (int j = 0; j < XB; ++j)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[0][j][b] = acc[1][j][b] = 0.0f;
  const float* m = M + 2 * XB * ol;
  const float* x = X + 4 * sl;
#pragma unroll 4
  for (int k = 0; k < dK; ++k) {
    float xv[4], mv[2 * XB];
    load4(x + k * kGStride, xv);
    load_run<2 * XB>(m + (size_t)k * 2 * P, mv);
#pragma unroll
    for (int j = 0; j < XB; ++j)
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        acc[0][j][b] = fmaf(mv[2 * j], xv[b], acc[0][j][b]);
        acc[1][j][b] = fmaf(mv[2 * j + 1], xv[b], acc[1][j][b]);
      }
  }
}

// acc[j][b] = sum_k sum_s M[k][x0 + j][s] Y[2 k + s][b]
template <int XB>
__device__ __forceinline__ void contract_in(const float* M, int P, int dK, const float* Y, int ol, int sl,
                                            float (&acc)[XB][4]) {
#pragma unroll
  for (int j = 0; j < XB; ++j)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[j][b] = 0.0f;
  const float* m = M + 2 * XB * ol;
  const float* y = Y + 4 * sl;
#pragma unroll 4
  for (int k = 0; k < dK; ++k) {
    float y0[4], y1[4], mv[2 * XB];
    load4(y + (2 * k) * kGStride, y0);
    load4(y + (2 * k + 1) * kGStride, y1);
    load_run<2 * XB>(m + (size_t)k * 2 * P, mv);
#pragma unroll
    for (int j = 0; j < XB; ++j)
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        acc[j][b] = fmaf(mv[2 * j], y0[b], acc[j][b]);
        acc[j][b] = fmaf(mv[2 * j + 1], y1[b], acc[j][b]);
      }
  }
}

// G[rho][b] += sum_t V[rho][t] R[b][t] + W[rho][t] Lb[b][t], rho = 2 a + s < nr, b < nc.  The four
// warps take 2 x 2 blocks of 8 Q x 4 Q outputs, a thread Q x Q of them.
template <int Q>
__device__ __forceinline__ void site_gradient(const float* V, const float* W, const float* R, const float* Lb, int P,
                                              int nr, int nc, float* G) {
  const bool vec = (reinterpret_cast<uintptr_t>(G) & 15) == 0;      // the caller's buffer may be only 4-byte aligned
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int row0 = (warp & 1) * 8 * Q + (lane & 7), col0 = ((warp >> 1) * 4 + (lane >> 3)) * Q;
  float acc[Q][Q];
  int ro[Q], co[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    ro[i] = min(row0 + 8 * i, 2 * P - 1) * kGStride;
    co[i] = min(col0 + i, P - 1) * kGStride;
#pragma unroll
    for (int j = 0; j < Q; ++j) acc[i][j] = 0.0f;
  }
  auto add = [&](const float* A, const float* C) {
#pragma unroll 1
    for (int t = 0; t < kGT; t += 4) {
      float av[Q][4], cv[Q][4];
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        load4(A + ro[i] + t, av[i]);
        load4(C + co[i] + t, cv[i]);
      }
#pragma unroll
      for (int i = 0; i < Q; ++i)
#pragma unroll
        for (int j = 0; j < Q; ++j)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[i][j] = fmaf(av[i][q], cv[j][q], acc[i][j]);
    }
  };
  add(V, R);
  add(W, Lb);
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int rho = row0 + 8 * i;
    if (rho >= nr) continue;
    float* g = G + (size_t)rho * P + col0;
    if constexpr (Q % 4 == 0) {
#pragma unroll
      for (int j = 0; j < Q; j += 4) {
        if (vec && col0 + j + 3 < nc) {
          atomicAdd(reinterpret_cast<float4*>(g + j), make_float4(acc[i][j], acc[i][j + 1], acc[i][j + 2], acc[i][j + 3]));
        } else {
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (col0 + j + q < nc) atomicAdd(g + j + q, acc[i][j + q]);
        }
      }
    } else if constexpr (Q % 2 == 0) {
#pragma unroll
      for (int j = 0; j < Q; j += 2) {
        if (vec && col0 + j + 1 < nc) {
          atomicAdd(reinterpret_cast<float2*>(g + j), make_float2(acc[i][j], acc[i][j + 1]));
        } else {
#pragma unroll
          for (int q = 0; q < 2; ++q)
            if (col0 + j + q < nc) atomicAdd(g + j + q, acc[i][j + q]);
        }
      }
    } else {
#pragma unroll
      for (int j = 0; j < Q; ++j)
        if (col0 + j < nc) atomicAdd(g + j, acc[i][j]);
    }
  }
}

// The row's field factors and bond dimensions are in shared memory.  EDGE: rows too wide for that
// (P = 64: more than 2630 columns), which read them from global memory, and strong vertical bonds.
template <bool EDGE>
__global__ void __launch_bounds__(kGThreads, 2) logq_grad_kernel(GradArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const unsigned kFull = 0xffffffffu;
  const int Lx = a.e.Lx, Ly = a.e.Ly, P = a.e.P;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int sl = lane & 7, ol = (lane >> 3) + 4 * warp;      // samples 4 sl .. 4 sl + 3, outputs XB ol ..
  const GradSmem lay = grad_smem(P, Lx, !EDGE);
  float* ring = reinterpret_cast<float*>(smem_raw);
  float* set0 = reinterpret_cast<float*>(smem_raw + lay.set);
  const size_t set_sz = (size_t)6 * P * kGStride;
  float* mpart = reinterpret_cast<float*>(smem_raw + lay.mpart);     // [2][4][kGT]
  float* wpart = reinterpret_cast<float*>(smem_raw + lay.wpart);     // [2][4][2][kGT]
  uint32_t* prev = reinterpret_cast<uint32_t*>(smem_raw + lay.mask);
  uint32_t* cur = prev + Lx;
  int* okf = reinterpret_cast<int*>(smem_raw + lay.ok);
  const size_t n = (size_t)Lx * Ly, tstride = (size_t)P * 2 * P, slot = (size_t)P * kGT;
  float* Rs = a.scratch + (size_t)blockIdx.x * grad_cta_floats(P, Lx);
  float* Ls = Rs + (Lx + 1) * slot;
  float* Bs = Ls + (Lx + 1) * slot;
  float* w0s = Bs + (Lx + 1) * slot;             // [Lx][kGT]: raw w(-), then g(-)
  float* w1s = w0s + (size_t)Lx * kGT;
  int* ek = reinterpret_cast<int*>(w1s + (size_t)Lx * kGT);      // exponent of k_c
  int* ekp = ek + (size_t)Lx * kGT;                               // exponent of k'_c

  const int nstep = 4 * Lx - 3, dist = lay.nbuf - 1;
  for (int64_t base = (int64_t)blockIdx.x * kGT; base < a.B; base += (int64_t)gridDim.x * kGT) {
    const int rows = (a.B - base) < kGT ? (int)(a.B - base) : kGT;
    __syncthreads();       // the previous tile is done with shared memory
    for (int c = tid; c < Lx; c += kGThreads) prev[c] = 0u;
    int pr = 0, pi = 0, pbuf = 0;
    auto copy_next = [&]() {
      if (pr < Ly) {
        // steps: right sweep, left sweep, Lambda adjoint, R adjoint (sites 0 .. Lx - 2)
        const int p1 = Lx - 1, p2 = p1 + Lx, p3 = p2 + Lx - 1;
        const int c = pi < p1 ? Lx - 1 - pi : pi < p2 ? pi - p1 : pi < p3 ? Lx - 1 - (pi - p2) : pi - p3;
        const bool right = pi < p1 || (pi >= p2 && pi < p3);
        const float* src = (right ? a.Rt : a.K) + ((size_t)pr * Lx + c) * tstride;
        float* dst = ring + (size_t)pbuf * tstride;
        for (int q = tid; q < P * P / 2; q += kGThreads) cp_async16(dst + 4 * q, src + 4 * q);
        if (++pi == nstep) {
          pi = 0;
          ++pr;
        }
      }
      if (++pbuf == lay.nbuf) pbuf = 0;
      cp_async_commit();
    };
    for (int q = 0; q < dist; ++q) copy_next();
    int buf = 0;
    auto begin_step = [&]() -> const float* {
      if (dist == 2) cp_async_wait<1>();
      else cp_async_wait<0>();
      __syncthreads();
      copy_next();
      const float* M = ring + (size_t)buf * tstride;
      if (++buf == lay.nbuf) buf = 0;
      return M;
    };
    // the rescaling exponent of this thread's samples from the previous vector's maxima
    auto lag = [&](int par, int (&e)[4]) {
      float m[4], q[4];
      load4(mpart + par * 4 * kGT + 4 * sl, m);
#pragma unroll
      for (int w = 1; w < 4; ++w) {
        load4(mpart + (par * 4 + w) * kGT + 4 * sl, q);
#pragma unroll
        for (int b = 0; b < 4; ++b) m[b] = fmaxf(m[b], q[b]);
      }
#pragma unroll
      for (int b = 0; b < 4; ++b) e[b] = exponent_f32(__float_as_int(m[b]));
    };
    auto put_max = [&](int par, float (&m)[4]) {
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        m[b] = fmaxf(m[b], __shfl_xor_sync(kFull, m[b], 8));
        m[b] = fmaxf(m[b], __shfl_xor_sync(kFull, m[b], 16));
      }
      if (lane < 8) store_run<4>(mpart + (par * 4 + warp) * kGT + 4 * sl, m);
    };
    // Strong vertical bonds: a vector just written (rows x of X and of the stack slot St, this
    // thread's samples) is rescaled at once, by the exponent of its own largest entry (e on return).
    // The weights then hold one field factor instead of up to three (f_c, and those of Lambda_c
    // and R_{c+1}), whose product leaves FP32 from beta |Jv| = 29 on.
    auto rescale_now = [&](int par, int dX, float* X, float* St, int (&e)[4]) {
      __syncthreads();
      lag(par, e);
      by_outputs(dX, [&](auto xbc) {
        constexpr int XB = decltype(xbc)::value;
        for (int x = XB * ol; x < XB * ol + XB && x < dX; ++x) {
          float v[4];
          load4(X + x * kGStride + 4 * sl, v);
#pragma unroll
          for (int b = 0; b < 4; ++b) v[b] *= pow2_f32(-e[b]);
          store_run<4>(X + x * kGStride + 4 * sl, v);
          store_run<4>(St + x * kGT + 4 * sl, v);
        }
      });
    };
    // the exponent of the vector a step reads: lag, or 0 where rescale_now has divided it out
    auto lag_of = [&](int par, int (&e)[4]) {
      if (EDGE && a.e.strong) {
#pragma unroll
        for (int b = 0; b < 4; ++b) e[b] = 0;
      } else {
        lag(par, e);
      }
    };
    auto put_one = [&](float* X) {       // the boundary vector: one row of ones
      if (tid < kGT) X[tid] = 1.0f;
      if (tid < 4 * kGT) mpart[tid] = 1.0f;      // parity 0
    };

    for (int r = 0; r < Ly; ++r) {
      __syncthreads();
      const int* bond = a.e.bond + (size_t)r * (Lx + 1);
      const float* fer = a.fe + (size_t)r * Lx * 2;       // 1 on row 0
      if constexpr (!EDGE) {
        int* sbond = reinterpret_cast<int*>(smem_raw + lay.bond);
        float* sfer = reinterpret_cast<float*>(smem_raw + lay.fer);
        for (int c = tid; c <= Lx; c += kGThreads) sbond[c] = bond[c];
        for (int c = tid; c < 2 * Lx; c += kGThreads) sfer[c] = fer[c];
        bond = sbond;
        fer = sfer;
      }
      for (int c = tid; c < Lx; c += kGThreads) {
        const int8_t* src = a.spins + (size_t)base * n + (size_t)r * Lx + c;
        uint32_t m = 0;
#pragma unroll 8
        for (int s = 0; s < rows; ++s) m |= (src[(size_t)s * n] > 0 ? 1u : 0u) << s;
        cur[c] = m;
      }
      if (tid < kGT) {
        okf[tid] = 1;
        Rs[Lx * slot + tid] = 1.0f;      // R_Lx, Lambda_0 = 1 and Lbar_Lx = 0 (one bond)
        Ls[tid] = 1.0f;
        Bs[Lx * slot + tid] = 0.0f;
      }
      put_one(set0);
      // ---- 1. right sweep ----
      int step = 0;
      for (int c = Lx - 1; c >= 1; --c, ++step) {
        const float* M = begin_step();
        const int dK = bond[c + 1], dX = bond[c];
        const uint32_t up = prev[c];
        const float fdiff = fer[2 * c], fsame = fer[2 * c + 1];
        const float* X = set0 + (step & 1) * set_sz;
        float* Xn = set0 + ((step + 1) & 1) * set_sz;
        by_outputs(dX, [&](auto xbc) {
          constexpr int XB = decltype(xbc)::value;
          float acc[2][XB][4], m[4];
          int e[4];
          contract_out<XB>(M, P, dK, X, ol, sl, acc);
          lag_of(step & 1, e);
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            const bool u = (up >> (4 * sl + b)) & 1u;
            const float sc = pow2_f32(-e[b]);
            const float f0 = (u ? fdiff : fsame) * sc, f1 = (u ? fsame : fdiff) * sc;
            m[b] = 0.0f;
#pragma unroll
            for (int j = 0; j < XB; ++j) {
              acc[0][j][b] = fmaf(f0, acc[0][j][b], f1 * acc[1][j][b]);
              if (XB * ol + j < dX) m[b] = fmaxf(m[b], fabsf(acc[0][j][b]));
            }
          }
#pragma unroll
          for (int j = 0; j < XB; ++j) {
            const int x = XB * ol + j;
            if (x < dX) {
              store_run<4>(Xn + x * kGStride + 4 * sl, acc[0][j]);
              store_run<4>(Rs + c * slot + x * kGT + 4 * sl, acc[0][j]);
            }
          }
          if (ol == 0) *reinterpret_cast<int4*>(ekp + c * kGT + 4 * sl) = make_int4(-e[0], -e[1], -e[2], -e[3]);
          put_max((step + 1) & 1, m);
        });
        if (EDGE && a.e.strong) {
          int e[4];
          rescale_now((step + 1) & 1, dX, Xn, Rs + c * slot, e);
          if (ol == 0) *reinterpret_cast<int4*>(ekp + c * kGT + 4 * sl) = make_int4(-e[0], -e[1], -e[2], -e[3]);
        }
      }
      // ---- 2. left sweep (forced) ----
      __syncthreads();
      put_one(set0);
      step = 0;
      auto finish_weights = [&](int c) {      // raw weights of site c from the four warps' sums
        if (tid < 2 * kGT) {
          const int s = tid / kGT, t = tid % kGT;
          const float* wp = wpart + (c & 1) * 8 * kGT + s * kGT + t;
          const float w = (wp[0] + wp[2 * kGT]) + (wp[4 * kGT] + wp[6 * kGT]);
          const bool same = (int)((prev[c] >> t) & 1u) == s;
          (s ? w1s : w0s)[c * kGT + t] = w * (same ? fer[2 * c + 1] : fer[2 * c]);
        }
      };
      for (int c = 0; c < Lx; ++c, ++step) {
        const float* M = begin_step();
        if (c > 0) finish_weights(c - 1);
        const int dK = bond[c], dX = bond[c + 1];
        const uint32_t up = prev[c], sp = cur[c];
        const float fdiff = fer[2 * c], fsame = fer[2 * c + 1];
        const float* X = set0 + (step & 1) * set_sz;
        float* Xn = set0 + ((step + 1) & 1) * set_sz;
        by_outputs(dX, [&](auto xbc) {
          constexpr int XB = decltype(xbc)::value;
          float rv[XB][4];
#pragma unroll
          for (int j = 0; j < XB; ++j) {
            const int x = XB * ol + j;
            if (x < dX) load4(Rs + (c + 1) * slot + x * kGT + 4 * sl, rv[j]);
          }
          float acc[2][XB][4], m[4], w0[4], w1[4];
          int e[4];
          contract_out<XB>(M, P, dK, X, ol, sl, acc);
          lag_of(step & 1, e);
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            const bool u = (up >> (4 * sl + b)) & 1u, s = (sp >> (4 * sl + b)) & 1u;
            const float fs = ((u == s) ? fsame : fdiff) * pow2_f32(-e[b]);
            m[b] = w0[b] = w1[b] = 0.0f;
#pragma unroll
            for (int j = 0; j < XB; ++j) {
              if (XB * ol + j < dX) {
                w0[b] = fmaf(acc[0][j][b], rv[j][b], w0[b]);
                w1[b] = fmaf(acc[1][j][b], rv[j][b], w1[b]);
                acc[0][j][b] = (s ? acc[1][j][b] : acc[0][j][b]) * fs;
                m[b] = fmaxf(m[b], fabsf(acc[0][j][b]));
              }
            }
          }
#pragma unroll
          for (int j = 0; j < XB; ++j) {
            const int x = XB * ol + j;
            if (x < dX) {
              store_run<4>(Xn + x * kGStride + 4 * sl, acc[0][j]);
              store_run<4>(Ls + (c + 1) * slot + x * kGT + 4 * sl, acc[0][j]);
            }
          }
          if (ol == 0) *reinterpret_cast<int4*>(ek + c * kGT + 4 * sl) = make_int4(-e[0], -e[1], -e[2], -e[3]);
          put_max((step + 1) & 1, m);
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            w0[b] += __shfl_xor_sync(kFull, w0[b], 8);
            w1[b] += __shfl_xor_sync(kFull, w1[b], 8);
            w0[b] += __shfl_xor_sync(kFull, w0[b], 16);
            w1[b] += __shfl_xor_sync(kFull, w1[b], 16);
          }
          if (lane < 8) {
            store_run<4>(wpart + (c & 1) * 8 * kGT + 2 * warp * kGT + 4 * sl, w0);
            store_run<4>(wpart + (c & 1) * 8 * kGT + (2 * warp + 1) * kGT + 4 * sl, w1);
          }
        });
        if (EDGE && a.e.strong) {
          int e[4];
          rescale_now((step + 1) & 1, dX, Xn, Ls + (c + 1) * slot, e);
          if (ol == 0) *reinterpret_cast<int4*>(ek + c * kGT + 4 * sl) = make_int4(-e[0], -e[1], -e[2], -e[3]);
        }
      }
      __syncthreads();
      finish_weights(Lx - 1);
      __syncthreads();
      // ---- 3. weight adjoints; a sample with a non-positive normaliser, or with q = 0,
      // contributes nothing (its log q is not differentiable) ----
      for (int q = tid; q < Lx * kGT; q += kGThreads) {
        const int c = q / kGT, t = q % kGT;
        const float w0 = fmaxf(w0s[q], 0.0f), w1 = fmaxf(w1s[q], 0.0f);
        const float ws = ((cur[c] >> t) & 1u) ? w1 : w0;
        if (!(w0 + w1 > 0.0f && isfinite(w0 + w1) && ws > 0.0f)) okf[t] = 0;
      }
      if (tid < kGT) {
        const float wt = tid < rows ? a.weights[base + tid] : 0.0f;
        if (!(wt != 0.0f)) okf[tid] = 0;
      }
      __syncthreads();
      for (int q = tid; q < Lx * kGT; q += kGThreads) {
        const int c = q / kGT, t = q % kGT;
        const float w0r = w0s[q], w1r = w1s[q];
        const float w0 = fmaxf(w0r, 0.0f), w1 = fmaxf(w1r, 0.0f);
        const bool sc = (cur[c] >> t) & 1u, u = (prev[c] >> t) & 1u;
        float g0 = 0.0f, g1 = 0.0f;
        if (okf[t]) {
          const float wt = a.weights[base + t];
          const float inv = -1.0f / (w0 + w1), is = 1.0f / (sc ? w1 : w0);
          if (w0r > 0.0f) g0 = wt * (inv + (sc ? 0.0f : is)) * (u ? fer[2 * c] : fer[2 * c + 1]);
          if (w1r > 0.0f) g1 = wt * (inv + (sc ? is : 0.0f)) * (u ? fer[2 * c + 1] : fer[2 * c]);
        }
        w0s[q] = g0;
        w1s[q] = g1;
      }
      __syncthreads();
      // this thread's samples that contribute (the others' vectors count as zero below)
      bool ok[4];
#pragma unroll
      for (int b = 0; b < 4; ++b) ok[b] = okf[4 * sl + b] != 0;
      // g, k f of the sample's own spin, and the spin, of site c
      struct SiteW {
        float g0[4], g1[4], kf[4];
        uint32_t sp;
      };
      auto site_weights = [&](int c, SiteW& w) {
        load4(w0s + c * kGT + 4 * sl, w.g0);
        load4(w1s + c * kGT + 4 * sl, w.g1);
        const int4 e = *reinterpret_cast<const int4*>(ek + c * kGT + 4 * sl);
        const int ev[4] = {e.x, e.y, e.z, e.w};
        w.sp = cur[c] >> (4 * sl);
        const uint32_t up = prev[c] >> (4 * sl);
#pragma unroll
        for (int b = 0; b < 4; ++b)
          w.kf[b] = ((((up ^ w.sp) >> b) & 1u) ? fer[2 * c] : fer[2 * c + 1]) * pow2_f32(ev[b]);
      };
      // Y rows x of site c from R_{c+1} and Lbar_{c+1}
      auto put_y = [&](float* Y, int x, const float (&rv)[4], const float (&lb)[4], const SiteW& w) {
        float y0[4], y1[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const float rr = ok[b] ? rv[b] : 0.0f, t = w.kf[b] * lb[b];
          const bool s = (w.sp >> b) & 1u;
          y0[b] = fmaf(w.g0[b], rr, s ? 0.0f : t);
          y1[b] = fmaf(w.g1[b], rr, s ? t : 0.0f);
        }
        store_run<4>(Y + (2 * x) * kGStride + 4 * sl, y0);
        store_run<4>(Y + (2 * x + 1) * kGStride + 4 * sl, y1);
      };
      // ---- 4. Lambda adjoint, right to left ----
      if (Lx > 1 && ol == 0) {
        SiteW w;
        site_weights(Lx - 1, w);
        const float one[4] = {1.0f, 1.0f, 1.0f, 1.0f}, zero[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        put_y(set0, 0, one, zero, w);
      }
      step = 0;
      for (int c = Lx - 1; c >= 1; --c, ++step) {
        const float* M = begin_step();
        const int dK = bond[c + 1], dX = bond[c];
        const float* Y = set0 + (step & 1) * set_sz;
        float* Yn = set0 + ((step + 1) & 1) * set_sz;
        SiteW w;
        if (c > 1) site_weights(c - 1, w);
        by_outputs(dX, [&](auto xbc) {
          constexpr int XB = decltype(xbc)::value;
          float rv[XB][4];
#pragma unroll
          for (int j = 0; j < XB; ++j) {
            const int x = XB * ol + j;
            if (x < dX && c > 1) load4(Rs + c * slot + x * kGT + 4 * sl, rv[j]);
          }
          float acc[XB][4];
          contract_in<XB>(M, P, dK, Y, ol, sl, acc);
#pragma unroll
          for (int j = 0; j < XB; ++j) {
            const int x = XB * ol + j;
            if (x < dX) {
              store_run<4>(Bs + c * slot + x * kGT + 4 * sl, acc[j]);
              if (c > 1) put_y(Yn, x, rv[j], acc[j], w);
            }
          }
        });
      }
      __syncthreads();
      // ---- 5. R adjoint left to right, and the site gradients.  Buffer set: V [2 P], W [2 P],
      // R [P], Lbar [P] rows of site c ----
      const int oW = 2 * P * kGStride, oR = 4 * P * kGStride, oL = 5 * P * kGStride;
      // V and W rows x of site c from Lambda_c and k'_c f Rbar_c (rb holds Rbar_c)
      auto put_v = [&](float* S, int x, const float (&lv)[4], const float (&rb)[4], const SiteW& w, int c) {
        const uint32_t up = prev[c] >> (4 * sl);
        const int4 e = c > 0 ? *reinterpret_cast<const int4*>(ekp + c * kGT + 4 * sl) : make_int4(0, 0, 0, 0);
        const int ev[4] = {e.x, e.y, e.z, e.w};
        float v0[4], v1[4], x0[4], x1[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const float l = ok[b] ? lv[b] : 0.0f;
          const float kr = pow2_f32(ev[b]) * rb[b];
          const bool u = (up >> b) & 1u, s = (w.sp >> b) & 1u;
          v0[b] = fmaf(w.g0[b], l, (u ? fer[2 * c] : fer[2 * c + 1]) * kr);
          v1[b] = fmaf(w.g1[b], l, (u ? fer[2 * c + 1] : fer[2 * c]) * kr);
          const float t = w.kf[b] * l;
          x0[b] = s ? 0.0f : t;
          x1[b] = s ? t : 0.0f;
        }
        store_run<4>(S + (2 * x) * kGStride + 4 * sl, v0);
        store_run<4>(S + (2 * x + 1) * kGStride + 4 * sl, v1);
        store_run<4>(S + oW + (2 * x) * kGStride + 4 * sl, x0);
        store_run<4>(S + oW + (2 * x + 1) * kGStride + 4 * sl, x1);
      };
      // R_{c+1} and Lbar_{c+1} rows of site c
      auto put_right = [&](float* S, int c) {
        const int d = bond[c + 1];
        by_outputs(d, [&](auto xbc) {
          constexpr int XB = decltype(xbc)::value;
#pragma unroll
          for (int j = 0; j < XB; ++j) {
            const int x = XB * ol + j;
            if (x < d) {
              float rv[4], lb[4];
              load4(Rs + (c + 1) * slot + x * kGT + 4 * sl, rv);
              load4(Bs + (c + 1) * slot + x * kGT + 4 * sl, lb);
#pragma unroll
              for (int b = 0; b < 4; ++b) {
                rv[b] = ok[b] ? rv[b] : 0.0f;
                lb[b] = ok[b] ? lb[b] : 0.0f;
              }
              store_run<4>(S + oR + x * kGStride + 4 * sl, rv);
              store_run<4>(S + oL + x * kGStride + 4 * sl, lb);
            }
          }
        });
      };
      if (ol == 0) {
        SiteW w;
        site_weights(0, w);
        const float one[4] = {1.0f, 1.0f, 1.0f, 1.0f}, zero[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        put_v(set0, 0, one, zero, w, 0);
      }
      put_right(set0, 0);
      for (int c = 0; c < Lx; ++c) {
        float* S = set0 + (c & 1) * set_sz;
        float* Sn = set0 + ((c + 1) & 1) * set_sz;
        const int dl = bond[c], dr = bond[c + 1];
        if (c + 1 < Lx) {
          const float* M = begin_step();
          SiteW w;
          site_weights(c + 1, w);
          by_outputs(dr, [&](auto xbc) {
            constexpr int XB = decltype(xbc)::value;
            float lv[XB][4];
#pragma unroll
            for (int j = 0; j < XB; ++j) {
              const int x = XB * ol + j;
              if (x < dr) load4(Ls + (c + 1) * slot + x * kGT + 4 * sl, lv[j]);
            }
            float acc[XB][4];
            contract_in<XB>(M, P, dl, S, ol, sl, acc);
#pragma unroll
            for (int j = 0; j < XB; ++j) {
              const int x = XB * ol + j;
              if (x < dr) put_v(Sn, x, lv[j], acc[j], w, c + 1);
            }
          });
          put_right(Sn, c + 1);
        } else {
          __syncthreads();
        }
        float* G = a.grad + ((size_t)r * Lx + c) * tstride;
        const int q = (max(dl, dr) + 7) >> 3;
        if (q <= 1) site_gradient<1>(S, S + oW, S + oR, S + oL, P, 2 * dl, dr, G);
        else if (q == 2) site_gradient<2>(S, S + oW, S + oR, S + oL, P, 2 * dl, dr, G);
        else if (q <= 4) site_gradient<4>(S, S + oW, S + oR, S + oL, P, 2 * dl, dr, G);
        else site_gradient<8>(S, S + oW, S + oR, S + oL, P, 2 * dl, dr, G);
      }
      __syncthreads();
      for (int c = tid; c < Lx; c += kGThreads) prev[c] = cur[c];
    }
    cp_async_wait<0>();
  }
}

}  // namespace
}  // namespace tnmc

tnmc_status tnmc_launch_logq_grad(const tnmc_env* env, int64_t B, const int8_t* spins, const float* weights,
                                  float* grad, cudaStream_t stream) {
  using namespace tnmc;
  const DeviceEnv& d = env->d;
  const size_t gsz = (size_t)d.Lx * d.Ly * d.P * 2 * d.P;
  TNMC_CUDA_TRY(cudaMemsetAsync(grad, 0, gsz * sizeof(float), stream));
  if (B == 0) return TNMC_OK;
  int dev = 0, max_optin = 0, nsm = 0;
  TNMC_CUDA_TRY(cudaGetDevice(&dev));
  TNMC_CUDA_TRY(cudaDeviceGetAttribute(&max_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  TNMC_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  // small bonds, large batches (P = 4: from about 9700 samples, P = 8: from 39000): one thread per
  // sample, measured on both sides in grad_small.cu
  if (d.P <= 8 && B >= (int64_t)(d.P == 4 ? 64 : 256) * nsm && tnmc_grad_small_smem(d.Lx, d.P) <= (size_t)max_optin)
    return tnmc_launch_logq_grad_small(env, B, spins, weights, grad, nsm, stream);
  const bool staged = !d.strong && grad_smem(d.P, d.Lx, true).total <= (size_t)max_optin;
  const size_t smem = grad_smem(d.P, d.Lx, staged).total;
  if (smem > (size_t)max_optin) {
    tnmc_set_error("gradient kernel needs %zu bytes of shared memory (device allows %d)", smem, max_optin);
    return TNMC_E_UNSUPPORTED;
  }
  auto kern = staged ? logq_grad_kernel<false> : logq_grad_kernel<true>;
  TNMC_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  int per_sm = 0;
  TNMC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kGThreads, smem));
  int64_t grid = (B + kGT - 1) / kGT;
  if (grid > (int64_t)nsm * (per_sm < 1 ? 1 : per_sm)) grid = (int64_t)nsm * (per_sm < 1 ? 1 : per_sm);
  tnmc_env* me = const_cast<tnmc_env*>(env);
  {
    const tnmc_status gs = grow_scratch(me, (size_t)grid * grad_cta_floats(d.P, d.Lx) * sizeof(float), stream, "gradient");
    if (gs != TNMC_OK) return gs;
  }
  GradArgs a;
  a.e = d;
  a.K = d.K32;
  a.Rt = d.R32;
  a.fe = d.fe32;
  a.B = B;
  a.spins = spins;
  a.weights = weights;
  a.grad = grad;
  a.scratch = static_cast<float*>(me->scratch.ptr);
  kern<<<(unsigned)grid, kGThreads, smem, stream>>>(a);
  TNMC_CUDA_TRY(cudaGetLastError());
  return TNMC_OK;
}
