// FP32 sampler / evaluator: a CTA of independent warps, each drawing (or evaluating) a tile
// of S = 8 SB samples (see sample_simt.cu for the algorithm).  Shared by the translation units
// that launch it.
//
// What bounds it: per site and sweep a (S x chi) . (chi x 2 chi) product whose operands must
// reach the FFMA pipe.  With one sample per thread every 8 FMAs needed 9 words from the load
// pipe (128 B per cycle and SM), 4.5 times what the FMAs take.  Here the 32 lanes are 8 sample
// lanes x 4 output lanes and a lane keeps a block of SB samples x XB bonds x 2 spins in
// registers: SB + 2 XB words per 2 SB XB FMAs, so SB = 8 with XB >= 4 balances the two pipes.
//   - The site tensors go through a ring of shared-memory buffers filled by cp.async one or two
//     sites ahead, shared by the CTA's warps (one __syncthreads per site).
//   - A lane reads back from the vector stack exactly what it wrote, so the stack is laid out
//     per lane (512 B per warp instruction) and needs no synchronisation.
//   - The spins of a row are one bit mask per column; the energy is an exact 64-bit fixed-point
//     sum from the masks, and log q a product with integer exponents (one log per sample), so
//     that nothing per site runs on the FP64 pipe.
// Measured against one thread per sample (128 per CTA): 32 x 32, chi = 16, 65536 samples 11.3 ->
// 4.8 ms (25 % of the FFMA peak; 1.7 warps per scheduler: latency, a third of it the ordered dot
// product, draws and stores); 24 x 45, chi = 32, 16384 samples 28.8 -> 4.3 ms.
//
// The products and sums that decide a draw are taken in the order of a plain loop over the
// bonds (the dot product <U[s], R> is passed from output lane to output lane), so the results
// do not depend on the tile shape.  Rescalings are powers of two.
#pragma once

#include <math.h>

#include <type_traits>

#include "common.cuh"
#include "sample_args.cuh"
#include "umma.cuh"

namespace tnmc {
namespace {

template <int N>
struct IntF {
  static constexpr int value = N;
};

// Bonds per output lane for dX outputs: the smallest supported XB with 4 XB >= dX.
__host__ __device__ inline int f32_xb(int dX) {
  const int q = (dX + 3) >> 2;
  return q <= 4 ? (q < 1 ? 1 : q) : q <= 6 ? 6 : q <= 8 ? 8 : q <= 12 ? 12 : 16;
}

template <int XBM, class F>
__device__ __forceinline__ void by_xb(int dX, F&& f) {
  const int q = (dX + 3) >> 2;
  if (q <= 1) f(IntF<1>{});
  else if (q == 2) f(IntF<2>{});
  else if (q == 3) f(IntF<3>{});
  else if (q == 4 || XBM <= 4) f(IntF<4>{});
  else if constexpr (XBM > 4) {
    if (q <= 6) f(IntF<6>{});
    else if (q <= 8 || XBM <= 8) f(IntF<8>{});
    else if constexpr (XBM > 8) {
      if (q <= 12) f(IntF<12>{});
      else f(IntF<16>{});
    }
  }
}

__device__ __forceinline__ float pow2_f32(int e) { return __int_as_float((127 + e) << 23); }   // |e| <= 126
// Exponent of a magnitude's bits; 0 for zero, subnormal, infinite and NaN.
__device__ __forceinline__ int exponent_f32(int bits) {
  const int ex = (bits >> 23) & 0xff;
  return (ex == 0 || ex == 255) ? 0 : min(ex - 127, 126);
}

// N consecutive floats from an address aligned to gcd(N, 4) floats
template <int N>
__device__ __forceinline__ void load_run(const float* p, float* o) {
  if constexpr (N % 4 == 0) {
#pragma unroll
    for (int i = 0; i < N; i += 4) {
      const float4 v = *reinterpret_cast<const float4*>(p + i);
      o[i] = v.x; o[i + 1] = v.y; o[i + 2] = v.z; o[i + 3] = v.w;
    }
  } else if constexpr (N % 2 == 0) {
#pragma unroll
    for (int i = 0; i < N; i += 2) {
      const float2 v = *reinterpret_cast<const float2*>(p + i);
      o[i] = v.x; o[i + 1] = v.y;
    }
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) o[i] = p[i];
  }
}

template <int N>
__device__ __forceinline__ void store_run(float* p, const float* v) {
  if constexpr (N % 4 == 0) {
#pragma unroll
    for (int i = 0; i < N; i += 4) *reinterpret_cast<float4*>(p + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
  } else if constexpr (N % 2 == 0) {
#pragma unroll
    for (int i = 0; i < N; i += 2) *reinterpret_cast<float2*>(p + i) = make_float2(v[i], v[i + 1]);
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) p[i] = v[i];
  }
}

// A lane's SB samples of a row of S: runs of VS = min(SB, 4), 8 lanes apart.
template <int SB>
struct F32Lane {
  static constexpr int S = 8 * SB, VS = SB < 4 ? SB : 4, NO = (S + 31) / 32;
  // sample of block entry b: bit bit(sg, b) of mask word word(b)
  __device__ static constexpr int word(int b) { return (b / VS) * (8 * VS) / 32; }
  __device__ static __forceinline__ int bit(int sg, int b) { return (b / VS) * (8 * VS) % 32 + VS * sg + b % VS; }
  __device__ static __forceinline__ void load(const float* row, int sg, float* o) {
#pragma unroll
    for (int q = 0; q < SB / VS; ++q) load_run<VS>(row + q * (8 * VS) + VS * sg, o + q * VS);
  }
  __device__ static __forceinline__ void store(float* row, int sg, const float* v) {
#pragma unroll
    for (int q = 0; q < SB / VS; ++q) store_run<VS>(row + q * (8 * VS) + VS * sg, v + q * VS);
  }
};

// acc[s][j][b] = sum_k M[k][x0 + j][s] X[k][sample b], x0 = XB g, in the order k = 0, 1, ...
// Paired FP32 FMAs halve the issue slots; the pairs run over the spins where the block has fewer
// samples than tensor entries (one duplicated operand per sample instead of one per entry), else
// over the samples.  Against single FMAs (chi 24 / 32): 65536 samples of 12 x 40 3.85 -> 3.67 /
// 5.09 -> 4.87 ms, 16384 samples 1.45 -> 1.37 / 1.81 -> 1.73 ms.
// Outputs past the bond dimension are never used.
template <int SB, int XB>
__device__ __forceinline__ void f32_contract(const float* M, int P, int dK, const float* X, int g, int sg,
                                             float (&acc)[2][XB][SB]) {
  using Ln = F32Lane<SB>;
#pragma unroll
  for (int j = 0; j < XB; ++j)
#pragma unroll
    for (int b = 0; b < SB; ++b) acc[0][j][b] = acc[1][j][b] = 0.0f;
  // the operands of step k + 1 are loaded before the products of step k (the last load reads one
  // row past the end: inside shared memory, never used)
  const float* m = M + 2 * XB * g;
  float xv[2][SB], mv[2][2 * XB];
  Ln::load(X, sg, xv[0]);
  load_run<2 * XB>(m, mv[0]);
  auto products = [&](const float (&xk)[SB], const float (&mk)[2 * XB]) {
#pragma unroll
    for (int j = 0; j < XB; ++j)
      if constexpr (SB < 8 && SB < 2 * XB) {
        const float2 mm = make_float2(mk[2 * j], mk[2 * j + 1]);
#pragma unroll
        for (int b = 0; b < SB; ++b) {
          const float2 r = umma::f2_fma(mm, make_float2(xk[b], xk[b]), make_float2(acc[0][j][b], acc[1][j][b]));
          acc[0][j][b] = r.x; acc[1][j][b] = r.y;
        }
      } else if constexpr (SB > 1) {
        const float2 m0 = make_float2(mk[2 * j], mk[2 * j]), m1 = make_float2(mk[2 * j + 1], mk[2 * j + 1]);
#pragma unroll
        for (int b = 0; b < SB; b += 2) {
          const float2 x2 = make_float2(xk[b], xk[b + 1]);
          const float2 r0 = umma::f2_fma(m0, x2, make_float2(acc[0][j][b], acc[0][j][b + 1]));
          const float2 r1 = umma::f2_fma(m1, x2, make_float2(acc[1][j][b], acc[1][j][b + 1]));
          acc[0][j][b] = r0.x; acc[0][j][b + 1] = r0.y;
          acc[1][j][b] = r1.x; acc[1][j][b + 1] = r1.y;
        }
      } else {
        acc[0][j][0] = fmaf(mk[2 * j], xk[0], acc[0][j][0]);
        acc[1][j][0] = fmaf(mk[2 * j + 1], xk[0], acc[1][j][0]);
      }
  };
  if constexpr (XB > 8) {      // no registers for a second set of operands
    for (int k = 0; k < dK; ++k) {
      if (k > 0) {
        m += 2 * P;
        Ln::load(X + k * Ln::S, sg, xv[0]);
        load_run<2 * XB>(m, mv[0]);
      }
      products(xv[0], mv[0]);
    }
    return;
  }
  int k = 0;
#pragma unroll (SB * XB >= 16 ? 1 : 2)
  for (; k + 2 <= dK; k += 2, m += 4 * P) {
    Ln::load(X + (k + 1) * Ln::S, sg, xv[1]);
    load_run<2 * XB>(m + 2 * P, mv[1]);
    products(xv[0], mv[0]);
    Ln::load(X + (k + 2) * Ln::S, sg, xv[0]);
    load_run<2 * XB>(m + 4 * P, mv[0]);
    products(xv[1], mv[1]);
  }
  if (k < dK) products(xv[0], mv[0]);
}

// Lane coordinates the compiler takes as new at every site.  Otherwise it forms the addresses
// of all block sizes before the site loop and spills them.
__device__ __forceinline__ void refresh(int& a, int& b, int& c) { asm volatile("" : "+r"(a), "+r"(b), "+r"(c)); }

// Shared memory of a CTA of NW warps: the tensor ring (nbuf tiles and slack for the reads of
// unused outputs), the field factors and bond dimensions of two rows (EDGE: neither, they are read
// from global memory), then per warp X [P][S], the per-sample state of the finished rows, w [2][S],
// the scales [S] and two rows of spin masks.
struct F32Smem {
  int nbuf;
  size_t ring, fer, bond, warp0, warp_bytes, total;
};
template <int S, bool EDGE>
using F32Mask = std::conditional_t<!EDGE || (S > 16), uint32_t, std::conditional_t<(S > 8), uint16_t, uint8_t>>;
inline __host__ __device__ F32Smem f32_smem(int P, int Lx, int SB, int NW, bool edge) {
  F32Smem m;
  m.nbuf = P > 32 ? 2 : 3;
  const int S = 8 * SB, NO = (S + 31) / 32;
  m.ring = 0;
  size_t o = ((size_t)m.nbuf * P * 2 * P + 128) * sizeof(float);
  m.fer = o;
  if (!edge) o += (size_t)4 * Lx * sizeof(float);
  m.bond = o;
  if (!edge) o += (size_t)2 * (Lx + 1) * sizeof(int);
  o = (o + 15) & ~(size_t)15;
  m.warp0 = o;
  m.warp_bytes = (((size_t)P * S + 3 * S) * sizeof(float) + (size_t)3 * 32 * NO * 8 +
                  (size_t)2 * Lx * NO * (edge && S <= 16 ? S / 8 : 4) + 15) & ~(size_t)15;
  m.total = o + NW * m.warp_bytes;
  return m;
}
// Floats of one sample's vector stack: Lx + 1 slots of 4 XB(P) bonds.
inline __host__ __device__ size_t f32_stack_floats(int P, int Lx) { return (size_t)(Lx + 1) * 4 * f32_xb(P); }

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Samples base0 .. of one instance by the whole CTA (NW = blockDim.x / 32 warps, S each).
// `stack`: the CTA's vector stacks, NW S f32_stack_floats(P, Lx) floats.
// EDGE: rows so wide that their field factors and bond dimensions in shared memory would cost the
// SM warps, and strong vertical bonds.
template <int SB, int XBM, bool EDGE>
__device__ void sample_f32_tile(const SampleArgs<float>& a, int64_t base0, unsigned char* smem, float* stack) {
  using Ln = F32Lane<SB>;
  constexpr int S = Ln::S, NO = Ln::NO, LP = S >= 32 ? 1 : 32 / S;
  const unsigned kFull = 0xffffffffu;
  const int Lx = a.e.Lx, Ly = a.e.Ly, P = a.e.P;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, NW = blockDim.x >> 5;
  const int lane_id = lane, lane_sg = lane & 7, lane_g = lane >> 3;
  const F32Smem lay = f32_smem(P, Lx, SB, NW, EDGE);
  float* ring = reinterpret_cast<float*>(smem);
  float* fer2 = reinterpret_cast<float*>(smem + lay.fer);
  int* bond2 = reinterpret_cast<int*>(smem + lay.bond);
  float* X = reinterpret_cast<float*>(smem + lay.warp0 + warp * lay.warp_bytes);
  double* st_q = reinterpret_cast<double*>(X + (size_t)P * S);       // q of the finished rows = st_q 2^st_qexp
  int64_t* st_qexp = reinterpret_cast<int64_t*>(st_q + 32 * NO);
  int64_t* st_e = st_qexp + 32 * NO;                                   // fixed-point energy
  float* wbuf = reinterpret_cast<float*>(st_e + 32 * NO);              // [2][S]
  float* mbuf = wbuf + 2 * S;              // [S]
  using Mask = F32Mask<S, EDGE>;
  Mask* prev = reinterpret_cast<Mask*>(mbuf + S);   // [Lx][NO]
  Mask* cur = prev + (size_t)Lx * NO;
  const size_t n = (size_t)Lx * Ly, tstride = (size_t)P * 2 * P;
  const size_t slot = (size_t)4 * f32_xb(P) * S;            // floats of one stack slot of a warp
  float* stk = stack + (size_t)warp * (Lx + 1) * slot;
  const int64_t base = base0 + (int64_t)warp * S;
  const bool alive = base < a.B;
  const int rows = alive ? ((a.B - base) < S ? (int)(a.B - base) : S) : 0;
  const int nstep = 2 * Lx - 1, dist = lay.nbuf - 1;

  // scalar state of the samples lane % S + 32 o this lane owns; what changes once a row is in
  // shared memory
  int own[NO];
  float prod[NO];
  int pexp[NO], flag[NO];
  uint64_t odd_word[NO];
  int64_t pair_id = -1;
#pragma unroll
  for (int o = 0; o < NO; ++o) {
    own[o] = lane % S + 32 * o;
    prod[o] = 1.0f;
    pexp[o] = flag[o] = 0;
    odd_word[o] = 0;
    st_q[32 * o + lane] = 1.0;
    st_qexp[32 * o + lane] = st_e[32 * o + lane] = 0;
  }
  for (int c = lane; c < Lx * NO; c += 32) prev[c] = 0u;

  // the producer's position: step pi of row pr is the next tensor to copy
  int pr = 0, pi = 0, pbuf = 0;
  auto copy_next = [&]() {
    if (pr < Ly) {
      const bool sn = a.e.order == 1 && (pr & 1);
      const bool first = pi < Lx - 1;
      const int j = first ? pi : pi - (Lx - 1);
      const int c = (first != sn) ? Lx - 1 - j : j;       // raster: first sweep right to left
      const float* src = ((first != sn) ? a.Rt : a.L) + ((size_t)pr * Lx + c) * tstride;
      float* dst = ring + (size_t)pbuf * tstride;
      for (int q = threadIdx.x; q < P * P / 2; q += blockDim.x) cp_async16(dst + 4 * q, src + 4 * q);
      if (++pi == nstep) {
        pi = 0;
        ++pr;
      }
    }
    if (++pbuf == lay.nbuf) pbuf = 0;
    cp_async_commit();
  };
  __syncthreads();      // the ring is free (the CTA's previous tile is done)
  for (int q = 0; q < dist; ++q) copy_next();
  int buf = 0;
  // start of a step: its tensor is visible to the CTA and the buffer of the previous step is free
  auto begin_step = [&]() -> const float* {
    if (dist == 2) cp_async_wait<1>();
    else cp_async_wait<0>();
    __syncthreads();
    copy_next();
    const float* M = ring + (size_t)buf * tstride;
    if (++buf == lay.nbuf) buf = 0;
    return M;
  };

  for (int r = 0; r < Ly; ++r) {
    const float* fer = a.fe + (size_t)r * Lx * 2;      // 1 on row 0
    const int* bond = a.e.bond + (size_t)r * (Lx + 1);
    if constexpr (!EDGE) {
      float* sfer = fer2 + (size_t)(r & 1) * 2 * Lx;
      int* sbond = bond2 + (size_t)(r & 1) * (Lx + 1);
      for (int c = threadIdx.x; c <= Lx; c += blockDim.x) sbond[c] = a.e.bond[r * (Lx + 1) + c];
      for (int c = threadIdx.x; c < 2 * Lx; c += blockDim.x) sfer[c] = r == 0 ? 1.0f : a.fe[(size_t)r * Lx * 2 + c];
      fer = sfer;
      bond = sbond;
    }
    const bool snake = a.e.order == 1 && (r & 1);
    if (a.spins_in && alive) {
      for (int c = lane; c < Lx; c += 32) {
        const int8_t* src = a.spins_in + (size_t)base * n + (size_t)r * Lx + c;
#pragma unroll
        for (int o = 0; o < NO; ++o) {
          const int ns = min(rows - 32 * o, 32);
          uint32_t m = 0;
#pragma unroll 8
          for (int s = 0; s < ns; ++s) m |= (src[(size_t)(32 * o + s) * n] > 0 ? 1u : 0u) << s;
          cur[c * NO + o] = m;
        }
      }
    }
    for (int s = lane; s < S; s += 32) X[s] = 1.0f;      // boundary bonds have dimension 1
    // ---- first sweep (no draws): right to left, or left to right on a snake row ----
    int elag[SB];     // exponent of the last vector's largest entry, divided out one step later
#pragma unroll
    for (int b = 0; b < SB; ++b) elag[b] = 0;
    for (int j = 0; j + 1 < Lx; ++j) {
      const float* M = begin_step();
      if (!alive) continue;
      const int c = snake ? j : Lx - 1 - j;
      const int dl = bond[c], dr = bond[c + 1];
      const int dK = snake ? dl : dr, dX = snake ? dr : dl;
      float* out = stk + (size_t)(snake ? c + 1 : c) * slot;
      uint32_t up[NO];
#pragma unroll
      for (int o = 0; o < NO; ++o) up[o] = prev[c * NO + o];
      const float fdiff = fer[2 * c], fsame = fer[2 * c + 1];
      by_xb<XBM>(dX, [&](auto xbc) {
        constexpr int XB = decltype(xbc)::value;
        int g = lane_g, sg = lane_sg, lane = lane_id;
        refresh(g, sg, lane);
        float acc[2][XB][SB];
        f32_contract<SB, XB>(M, P, dK, X, g, sg, acc);
        __syncwarp();
        float mb[SB];
#pragma unroll
        for (int b = 0; b < SB; ++b) {
          const bool u = (up[Ln::word(b)] >> Ln::bit(sg, b)) & 1u;
          const float sc = pow2_f32(-elag[b]);
          const float fm = (u ? fdiff : fsame) * sc, fp = (u ? fsame : fdiff) * sc;
          mb[b] = 0.0f;
#pragma unroll
          for (int x = 0; x < XB; ++x) {
            const float v = fmaf(fm, acc[0][x][b], fp * acc[1][x][b]);
            acc[0][x][b] = v;
            if (XB * g + x < dX) mb[b] = fmaxf(mb[b], fabsf(v));
          }
        }
#pragma unroll
        for (int x = 0; x < XB; ++x) {
          if (XB * g + x < dX) Ln::store(X + (XB * g + x) * S, sg, acc[0][x]);
#pragma unroll
          for (int q = 0; q < SB; q += Ln::VS)
            store_run<Ln::VS>(out + ((x * SB + q) / Ln::VS * 32 + lane) * Ln::VS, &acc[0][x][q]);
        }
#pragma unroll
        for (int b = 0; b < SB; ++b) {
          mb[b] = fmaxf(mb[b], __shfl_xor_sync(kFull, mb[b], 8));
          mb[b] = fmaxf(mb[b], __shfl_xor_sync(kFull, mb[b], 16));
          elag[b] = exponent_f32(__float_as_int(mb[b]));
        }
      });
      if (EDGE && a.e.strong) {      // f 2^-elag, or f times the vector, may leave FP32: rescale it now
        const int XB = f32_xb(dX);
#pragma unroll 1
        for (int x = 0; x < XB; ++x) {
          float v[SB];
#pragma unroll
          for (int q = 0; q < SB; q += Ln::VS) {
            float* o = out + ((x * SB + q) / Ln::VS * 32 + lane_id) * Ln::VS;
            load_run<Ln::VS>(o, &v[q]);
#pragma unroll
            for (int b = q; b < q + Ln::VS; ++b) v[b] *= pow2_f32(-elag[b]);
            store_run<Ln::VS>(o, &v[q]);
          }
          if (XB * lane_g + x < dX) Ln::store(X + (XB * lane_g + x) * S, lane_sg, v);
        }
#pragma unroll
        for (int b = 0; b < SB; ++b) elag[b] = 0;
      }
      __syncwarp();
    }
    // ---- second sweep: the draws ----
    for (int j = 0; j < Lx; ++j) {
      const float* M = begin_step();
      if (!alive) continue;
      if (j == 0) {
        for (int s = lane; s < S; s += 32) X[s] = 1.0f;
        __syncwarp();
      }
      const int c = snake ? Lx - 1 - j : j;
      const int dl = bond[c], dr = bond[c + 1];
      const int dK = snake ? dr : dl, dX = snake ? dl : dr;
      const bool edge = j + 1 == Lx;                      // the other vector is the boundary's 1
      const float* in = stk + (size_t)(snake ? c : c + 1) * slot;
      uint32_t up[NO];
#pragma unroll
      for (int o = 0; o < NO; ++o) up[o] = prev[c * NO + o];
      const float fdiff = fer[2 * c], fsame = fer[2 * c + 1];
      const int64_t site = (int64_t)r * Lx + c;
      uint64_t word[NO];
      if (!a.spins_in) {
        const bool have = (site & 1) && (site >> 1) == pair_id;
        pair_id = site >> 1;
#pragma unroll
        for (int o = 0; o < NO; ++o) {
          word[o] = odd_word[o];
          if (!have) {
            const uint64_t sample = a.offset + (uint64_t)(base + own[o]);
            const U4 w = philox4x32_10(U4{(uint32_t)(site >> 1), (uint32_t)sample, (uint32_t)(sample >> 32), 0u},
                                       (uint32_t)a.seed, (uint32_t)(a.seed >> 32));
            odd_word[o] = (uint64_t)w.z | ((uint64_t)w.w << 32);
            word[o] = (site & 1) ? odd_word[o] : ((uint64_t)w.x | ((uint64_t)w.y << 32));
          }
        }
      }
      by_xb<XBM>(dX, [&](auto xbc) {
        constexpr int XB = decltype(xbc)::value;
        int g = lane_g, sg = lane_sg, lane = lane_id;
        refresh(g, sg, lane);
        // the other vector: loaded under the contraction, or, where the accumulators leave no
        // registers, brought to L1 now and loaded after it
        constexpr bool early = SB * XB <= 32;
        float rv[XB][SB];
        auto load_rv = [&]() {
#pragma unroll
          for (int x = 0; x < XB; ++x) {
#pragma unroll
            for (int q = 0; q < SB; q += Ln::VS) {
              if (!edge) load_run<Ln::VS>(in + ((x * SB + q) / Ln::VS * 32 + lane) * Ln::VS, &rv[x][q]);
            }
          }
        };
        if (early) {
          load_rv();
        } else if (!edge) {
          for (int q = lane; q < XB * SB; q += 32)      // one 128-byte line per block entry
            asm volatile("prefetch.global.L1 [%0];" ::"l"(in + (size_t)q * 32));
        }
        float acc[2][XB][SB];
        f32_contract<SB, XB>(M, P, dK, X, g, sg, acc);
        if (!early) load_rv();
        if (edge || dX != 4 * XB) {      // unused outputs, and what the stack holds for them, must add nothing
#pragma unroll
          for (int x = 0; x < XB; ++x) {
            const bool in_range = XB * g + x < dX;
#pragma unroll
            for (int b = 0; b < SB; ++b) {
              rv[x][b] = in_range ? (edge ? 1.0f : rv[x][b]) : 0.0f;
              acc[0][x][b] = in_range ? acc[0][x][b] : 0.0f;
              acc[1][x][b] = in_range ? acc[1][x][b] : 0.0f;
            }
          }
        }
        // w(s) = sum_x U[s][x] R[x] in the order of x: output lane t adds its XB terms to what
        // lane t - 1 passed on (the other lanes' sums are not used)
        float w0[SB], w1[SB];
#pragma unroll
        for (int b = 0; b < SB; ++b) w0[b] = w1[b] = 0.0f;
        const int stages = (dX + XB - 1) / XB;
        for (int t = 0; t < stages; ++t) {
#pragma unroll
          for (int b = 0; b < SB; ++b) {
            if (t > 0) {
              w0[b] = __shfl_up_sync(kFull, w0[b], 8);
              w1[b] = __shfl_up_sync(kFull, w1[b], 8);
            }
#pragma unroll
            for (int x = 0; x < XB; ++x) {
              w0[b] = fmaf(acc[0][x][b], rv[x][b], w0[b]);
              w1[b] = fmaf(acc[1][x][b], rv[x][b], w1[b]);
            }
          }
        }
        if (g == stages - 1) {
          Ln::store(wbuf, sg, w0);
          Ln::store(wbuf + S, sg, w1);
        }
        __syncwarp();
        uint32_t mask[NO];
        bool noscale = false;
        float fso[NO];
#pragma unroll
        for (int o = 0; o < NO; ++o) {
          const bool u = (up[o] >> (own[o] & 31)) & 1u;
          const float fm = u ? fdiff : fsame, fp = u ? fsame : fdiff;
          const float v0 = fmaxf(wbuf[own[o]] * fm, 0.0f), v1 = fmaxf(wbuf[S + own[o]] * fp, 0.0f);
          const float tot = v0 + v1;
          const bool bad = !(tot > 0.0f) || !isfinite(tot);
          const float pplus = bad ? 0.5f : v1 / tot;
          const float pminus = bad ? 0.5f : v0 / tot;
          const bool plus = a.spins_in ? (cur[c * NO + o] >> (own[o] & 31)) & 1u : draw_plus_bits(pplus, word[o]);
          prod[o] *= plus ? pplus : pminus;
          if (prod[o] < 0x1.0p-60f && prod[o] > 0.0f) {
            prod[o] *= 0x1.0p60f;
            pexp[o] -= 60;
          }
          flag[o] |= bad ? TNMC_FLAG_NUMERIC : 0;
          mask[o] = __ballot_sync(kFull, plus);       // bit s: lane s owns sample s + 32 o
          // next vector: f(s) U[s] times 2^-ilogb(w(s)), so that <next, R> lands in [1, 2)
          const float ws = plus ? v1 : v0;
          const int we = (__float_as_int(ws) >> 23) & 0xff;
          fso[o] = plus ? fp : fm;
          noscale |= we == 0 || we == 255;
          if (S >= 32 || lane < S) mbuf[own[o]] = fso[o] * pow2_f32(-exponent_f32(__float_as_int(ws)));
        }
        if (!a.spins_in && lane == 0) {
#pragma unroll
          for (int o = 0; o < NO; ++o) cur[c * NO + o] = mask[o];
        }
        if (__any_sync(kFull, noscale)) {
          // a drawn weight that is zero or not finite gives no scale: those samples take it from
          // max |f(s) U[s]|
          const float* fsv = wbuf;      // the drawn weights move to registers first
          float wso[NO];
#pragma unroll
          for (int o = 0; o < NO; ++o) {
            const bool plus = (mask[o] >> (own[o] & 31)) & 1u;
            const bool u = (up[o] >> (own[o] & 31)) & 1u;
            wso[o] = plus ? fmaxf(wbuf[S + own[o]] * (u ? fsame : fdiff), 0.0f) : fmaxf(wbuf[own[o]] * (u ? fdiff : fsame), 0.0f);
          }
          __syncwarp();
#pragma unroll
          for (int o = 0; o < NO; ++o)
            if (S >= 32 || lane < S) wbuf[own[o]] = fso[o];
          __syncwarp();
          float fv[SB];
          Ln::load(fsv, sg, fv);
          float mv[SB];
#pragma unroll
          for (int b = 0; b < SB; ++b) {
            const bool plus = (mask[Ln::word(b)] >> Ln::bit(sg, b)) & 1u;
            int mx = 0;
#pragma unroll
            for (int x = 0; x < XB; ++x)
              mx = max(mx, __float_as_int((plus ? acc[1][x][b] : acc[0][x][b]) * fv[b]) & 0x7fffffff);
            mx = max(mx, __shfl_xor_sync(kFull, mx, 8));
            mx = max(mx, __shfl_xor_sync(kFull, mx, 16));
            mv[b] = fv[b] * pow2_f32(-exponent_f32(mx));
          }
          if (g == 0) Ln::store(wbuf + S, sg, mv);
          __syncwarp();
#pragma unroll
          for (int o = 0; o < NO; ++o) {
            const int we = (__float_as_int(wso[o]) >> 23) & 0xff;
            if ((we == 0 || we == 255) && (S >= 32 || lane < S)) mbuf[own[o]] = wbuf[S + own[o]];
          }
        }
        __syncwarp();
        float mu[SB];
        Ln::load(mbuf, sg, mu);
#pragma unroll
        for (int x = 0; x < XB; ++x) {
          float v[SB];
#pragma unroll
          for (int b = 0; b < SB; ++b) {
            const bool plus = (mask[Ln::word(b)] >> Ln::bit(sg, b)) & 1u;
            v[b] = (plus ? acc[1][x][b] : acc[0][x][b]) * mu[b];
          }
          if (XB * g + x < dX) Ln::store(X + (XB * g + x) * S, sg, v);
        }
      });
      __syncwarp();
    }
    if (!alive) continue;
    // ---- row end: log q, energy terms, spins, and this row becomes the previous one ----
#pragma unroll
    for (int o = 0; o < NO; ++o) {
      double q = st_q[32 * o + lane] * (double)prod[o];
      int64_t qe = st_qexp[32 * o + lane] + pexp[o], ea = st_e[32 * o + lane];
      const int hi = __double2hiint(q);
      if ((hi >> 20) != 0) {       // zero stays zero (a row's product is never subnormal in FP64)
        qe += (hi >> 20) - 1023;
        q = __hiloint2double((hi & 0xfffff) | (1023 << 20), __double2loint(q));
      }
      st_q[32 * o + lane] = q;
      st_qexp[32 * o + lane] = qe;
      prod[o] = 1.0f;
      pexp[o] = 0;
      const int bit = own[o] & 31;
      for (int c = lane / S; c < Lx; c += LP) {
        int64_t loc = a.e.qh[(size_t)r * Lx + c];
        if (c > 0) {
          const int64_t jj = a.e.qJh[(size_t)r * (Lx - 1) + c - 1];
          loc += ((cur[(c - 1) * NO + o] >> bit) & 1u) ? jj : -jj;
        }
        if (r > 0) {
          const int64_t jj = a.e.qJv[(size_t)(r - 1) * Lx + c];
          loc += ((prev[c * NO + o] >> bit) & 1u) ? jj : -jj;
        }
        ea -= ((cur[c * NO + o] >> bit) & 1u) ? loc : -loc;
      }
      st_e[32 * o + lane] = ea;
    }
    __syncwarp();
    for (int c = lane; c < Lx; c += 32) {
#pragma unroll
      for (int o = 0; o < NO; ++o) {
        const uint32_t m = cur[c * NO + o];
        if (a.spins_out && !a.spins_in) {
          int8_t* dst = a.spins_out + (size_t)(base + 32 * o) * n + (size_t)r * Lx + c;
          const int ns = min(rows - 32 * o, 32);
          for (int s = 0; s < ns; ++s) dst[(size_t)s * n] = ((m >> s) & 1u) ? 1 : -1;
        }
        prev[c * NO + o] = m;
      }
    }
    __syncwarp();
  }
  cp_async_wait<0>();
  if (!alive) return;
#pragma unroll
  for (int o = 0; o < NO; ++o) {
    int64_t ea = st_e[32 * o + lane];
#pragma unroll
    for (int k = S; k < 32; k <<= 1) ea += __shfl_xor_sync(kFull, ea, k);
    if (lane < S && own[o] < rows) {
      // a flagged sample keeps the log of the probability it was drawn with (log 1/2 at a site
      // whose normaliser failed): q stays the exact law of the sampler
      a.logq[base + own[o]] = log(st_q[32 * o + lane]) + (double)st_qexp[32 * o + lane] * 0.69314718055994530942;
      a.energy[base + own[o]] = scalbn((double)ea, a.e.qexp);
      if (a.flags) a.flags[base + own[o]] = flag[o];
      if (flag[o]) set_status(a.e.status, TNMC_E_NUMERIC);
    }
  }
}

// Resident CTAs of 4 warps per SM, which bounds the registers: 64 accumulators and two sets of
// operands need 255, 32 fit 168 (fewer registers spill and cost more than the warps give: the
// 8-sample block at 168 registers took 7.99 instead of 4.95 ms).
__host__ __device__ constexpr int f32_min_ctas(int SB, int XBM) { return SB * XBM >= 32 ? 2 : 3; }

template <int SB, int XBM, bool EDGE>
__global__ void __launch_bounds__(128, f32_min_ctas(SB, XBM)) sample_f32_kernel(SampleArgs<float> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int64_t step = (int64_t)(blockDim.x >> 5) * (8 * SB);
  float* stack = a.scratch + (size_t)blockIdx.x * step * f32_stack_floats(a.e.P, a.e.Lx);
  for (int64_t base = blockIdx.x * step; base < a.B; base += gridDim.x * step)
    sample_f32_tile<SB, XBM, EDGE>(a, base, smem_raw, stack);
}

// Samples per lane for `total` samples on `nsm` SMs at pad P.  Large blocks need fewer
// shared-memory words per FMA and share the scalar work, but a warp waits on its own latencies:
// the largest block that leaves 3 warps per SM (4 for the 8-sample block).  Measured, ms per
// launch at SB = 8 / 4 / 2 / 1: 32 x 32, chi = 16: 65536 samples 4.95 / 6.12 / 7.87 / 11.8, 32768
// 3.65 / 3.12 / 5.00 / 6.67, 8192 3.63 / 2.46 / 2.13 / 2.19; 24 x 45, chi = 32: 65536 - / 13.3 /
// 15.0 / 22.5, 8192 - / 4.53 / 3.50 / 4.04.  Above P = 16 (P = 32) an 8-sample (4-sample) block
// would spill its accumulators.
inline int f32_block(int64_t total, int P, int nsm) {
  if (P <= 16 && (total + 63) / 64 >= 4 * (int64_t)nsm) return 8;
  int SB = P > 32 ? 2 : 4;
  while (SB > 1 && (total + 8 * SB - 1) / (8 * SB) < 3 * (int64_t)nsm) SB >>= 1;
  return SB;
}
// Bonds per output lane that the kernel of block SB is compiled for.
__host__ __device__ constexpr int f32_xbm(int SB, int P) { return SB == 8 ? 4 : SB == 4 ? (P <= 16 ? 4 : 8) : P <= 32 ? 8 : 16; }

// The launch of `total` samples: samples per lane, warps per CTA (0: not even one fits), the kernel's
// form and its shared memory.  need(SB, NW, edge): bytes of a CTA; want(SB): most warps per CTA.
//
// f32_block's choice in the plain form, unless shared memory keeps fewer CTAs on an SM than the
// registers allow (from about 1000 columns on): then, over both forms and all smaller blocks, the
// least waves x time of a wave, where a wave of 8 / 4 / 2 / 1 samples per lane takes 1.45 / 1.15 / 1.05 /
// 1 and the EDGE form 1.05 times as long.  Measured, ms, f32_block's choice in the plain form / the
// rule's: 32768 samples of 5 x 4096, chi 16 185 / 100, 4 x 2048, chi 8 33.6 / 18.9, 2 x 4096, chi 2
// 61 / 32, 6 x 4096, chi 32 319 / 165.
struct F32Plan {
  int SB, NW;
  bool edge;
  size_t smem;
};
template <class Need, class Want>
F32Plan f32_plan(int64_t total, int P, bool strong, int nsm, size_t max_smem, size_t smem_sm, Need&& need, Want&& want) {
  auto form = [&](int SB, bool edge) {
    F32Plan p{SB, 0, edge, 0};
    for (p.NW = want(SB); p.NW > 0; p.NW >>= 1) {
      p.smem = need(SB, p.NW, edge);
      if (p.smem <= max_smem) break;
    }
    return p;
  };
  auto fit = [&](const F32Plan& p) { return smem_sm / (p.smem + 1024); };      // CTAs per SM by shared memory
  const int block = f32_block(total, P, nsm);
  F32Plan best = form(strong && block == 8 ? 4 : block, strong);
  if (best.NW > 0 && fit(best) >= (size_t)f32_min_ctas(best.SB, f32_xbm(best.SB, P))) return best;
  double least = 1e300;
  for (int SB = block; SB > 0; SB >>= 1)
    for (int edge = strong; edge < (SB < 8 ? 2 : 1); ++edge) {
      const F32Plan p = form(SB, edge);
      if (p.NW == 0) continue;
      size_t ctas = fit(p);
      const size_t regs = f32_min_ctas(SB, f32_xbm(SB, P));
      ctas = ctas < 1 ? 1 : ctas > regs ? regs : ctas;
      const int64_t wave = (int64_t)ctas * nsm * p.NW * 8 * SB;
      const double t = (double)((total + wave - 1) / wave) * (SB == 8 ? 1.45 : SB == 4 ? 1.15 : SB == 2 ? 1.05 : 1.0) *
                       (edge ? 1.05 : 1.0);
      if (t < least) {
        least = t;
        best = p;
      }
    }
  return best;
}

// Shared memory of a CTA that takes tiles of several lattices (P(i), Lx(i), i < n).  Each tile lays it
// out for its own lattice, and the size does not grow with P alone (the ring holds three
// tensors up to P = 32 and two above), so the reservation is the largest over the lattices.
template <class FP, class FL>
size_t f32_smem_largest(int n, FP&& P, FL&& Lx, int SB, int NW, bool edge) {
  size_t m = 0;
  for (int i = 0; i < n; ++i) {
    const size_t t = f32_smem(P(i), Lx(i), SB, NW, edge).total;
    if (t > m) m = t;
  }
  return m;
}

// f(IntF<SB>, IntF<XBM>, bool constant EDGE) for a plan's kernel (EDGE: at most 4 samples per lane)
template <class F>
tnmc_status by_f32_block(const F32Plan& p, int P, F&& f) {
  auto form = [&](auto sb, auto xbm) -> tnmc_status {
    constexpr int kSB = decltype(sb)::value;
    if constexpr (kSB < 8)
      if (p.edge) return f(sb, xbm, std::true_type{});
    return f(sb, xbm, std::false_type{});
  };
  switch (p.SB) {
    case 8: return form(IntF<8>{}, IntF<4>{});
    case 4: return P <= 16 ? form(IntF<4>{}, IntF<4>{}) : form(IntF<4>{}, IntF<8>{});
    case 2: return P <= 32 ? form(IntF<2>{}, IntF<8>{}) : form(IntF<2>{}, IntF<16>{});
    default: return P <= 32 ? form(IntF<1>{}, IntF<8>{}) : form(IntF<1>{}, IntF<16>{});
  }
}

}  // namespace
}  // namespace tnmc
