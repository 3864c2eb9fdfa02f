// FP64 sampler / evaluator: one warp draws (or evaluates) a tile of S samples (see
// sample_simt.cu for the algorithm).  Shared by the translation units that launch it.
//
// What bounds it: the FP64 pipe.  A GB300 SM retires one warp-wide FP64 instruction per 19
// cycles, whether all 32 lanes are active or one, a single warp can issue one only every 64
// cycles, and FP64 comparisons, maxima and divisions expand into several of them.  So the
// kernel counts warp instructions:
//   - The 32 lanes are LS sample lanes x LO output lanes, each with SB samples: every lane
//     of a contraction instruction carries a useful product even when a batch has few samples,
//     and tiles of down to 2 samples give an SM the warps that fill its FP64 pipe.
//   - Scalar work (normalisation, draw) runs on one lane per sample; log q is a running
//     product with an integer exponent (one log per sample), the division is two Newton steps
//     on rcp.approx and a residual step, clamps, maxima, draws and power-of-two scales are
//     integer operations, and the energy is an exact 64-bit fixed-point sum.
// Measured against one thread per sample (64 per CTA): 23 x 29, chi = 13, 5000 samples 26.2 ->
// 6.0 ms (76 % of the FP64 pipe); 64 lattices 32 x 32, chi = 16 with 32 samples each 47.9 -> 6.1 ms.
//
// A lane owns outputs x = g + LO i.  The dot product <U[s], R> goes through shared memory and is
// summed over x = 0, 1, ... by one lane per (sample, spin): it is where the weights cancel, so
// its order is that of a plain loop, and a sample's results depend on no tile shape.
#pragma once

#include <math.h>

#include <type_traits>

#include "common.cuh"
#include "sample_args.cuh"

namespace tnmc {
namespace {

template <int N>
struct IntC {
  static constexpr int value = N;
};

// f(IntC<NX>) for the smallest supported NX >= nx (nx <= MAX)
template <int MAX, class F>
__device__ __forceinline__ void by_count(int nx, F&& f) {
  if (nx <= 1) f(IntC<1>{});
  else if (nx <= 2 || MAX <= 2) f(IntC<2>{});
  else if (nx <= 3) f(IntC<3>{});
  else if (nx <= 4 || MAX <= 4) f(IntC<4>{});
  else if constexpr (MAX > 4) {
    if (nx <= 6) f(IntC<6>{});
    else if (nx <= 8 || MAX <= 8) f(IntC<8>{});
    else if constexpr (MAX > 8) {
      if (nx <= 12) f(IntC<12>{});
      else f(IntC<16>{});
    }
  }
}

// 2^e, |e| <= 1022
__device__ __forceinline__ double pow2_f64(int e) { return __hiloint2double((1023 + e) << 20, 0); }

// Exponent of a double's magnitude from its high word; 0 for zero, subnormal, infinite and NaN.
__device__ __forceinline__ int exponent_f64(int hi) {
  const int ex = (hi >> 20) & 0x7ff;
  return (ex == 0 || ex == 2047) ? 0 : min(ex - 1023, 1022);
}

// x 2^-e for x >= 0, on the integer pipe while x and the result are normal
__device__ __forceinline__ double scale_down_f64(double x, int e) {
  const int hi = __double2hiint(x), ex = (hi >> 20) - e;
  if ((hi >> 20) >= 1 && ex >= 1 && ex <= 2046) return __hiloint2double(hi - (e << 20), __double2loint(x));
  return x * pow2_f64(-e);
}

// max(w, 0) with NaN -> 0, on the integer pipe
__device__ __forceinline__ double clamp0_f64(double w) {
  const long long b = __double_as_longlong(w);
  return (b < 0 || b > 0x7ff0000000000000ll) ? 0.0 : w;
}

// 1 / t for normal t away from the ends of the range: the hardware's approximation (relative
// error 2^-20 or better) and two Newton-Raphson steps r += r (1 - t r), which square it twice.
__device__ __forceinline__ double reciprocal_f64(double t) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(t));
  r = fma(r, fma(-t, r, 1.0), r);
  return fma(r, fma(-t, r, 1.0), r);
}

// w / t from r = reciprocal_f64(t): the product and one residual step (Markstein's correction), which
// rounds to the nearest double; the product alone is off by up to two units in the last place.
__device__ __forceinline__ double quotient_f64(double w, double t, double r) {
  const double q = w * r;
  return fma(fma(-q, t, w), r, q);
}

// +1 iff x < floor(p 2^64) (draw_plus), from the bits of p
__device__ __forceinline__ bool draw_plus_bits(double p, uint64_t x) {
  const long long b = __double_as_longlong(p);
  if (b >= 0x3ff0000000000000ll) return true;        // p >= 1
  if (b <= 0) return false;                            // p <= 0
  const int sh = (int)(b >> 52) - 1011;                // p 2^64 = mantissa 2^sh, sh <= 11
  const uint64_t m = (uint64_t)(b & 0xfffffffffffffll) | (1ull << 52);   // subnormal p: floor is 0 either way
  const uint64_t t = sh >= 0 ? m << sh : (sh > -64 ? m >> -sh : 0ull);
  return x < t;
}

// acc[s][i][b] = sum_k M[k](x_i, s) X[k][sample b], x_i = g + LO i.  RT: M is [k][x][s] (the
// transposed copy), else [k][s][x].  Loads past the padded row are clamped to its last entry
// (those outputs are never used).
template <int LS, int SB, int NX, bool RT>
__device__ __forceinline__ void f64_contract(const double* __restrict__ M, int P, int dK, const double* X, int g,
                                             int sg, double (&acc)[2][NX][SB]) {
  constexpr int LO = 32 / LS, S = LS * SB;
  int xo[NX];
#pragma unroll
  for (int i = 0; i < NX; ++i) {
    xo[i] = min(g + LO * i, P - 1);
#pragma unroll
    for (int b = 0; b < SB; ++b) acc[0][i][b] = acc[1][i][b] = 0.0;
  }
#pragma unroll (NX * SB > 4 ? 2 : 4)
  for (int k = 0; k < dK; ++k) {
    double xv[SB];
#pragma unroll
    for (int b = 0; b < SB; ++b) xv[b] = X[k * S + sg + LS * b];
#pragma unroll
    for (int i = 0; i < NX; ++i) {
      double m0, m1;
      if (RT) {
        const double2 v = __ldg(reinterpret_cast<const double2*>(M + ((size_t)k * P + xo[i]) * 2));
        m0 = v.x;
        m1 = v.y;
      } else {
        m0 = __ldg(M + (size_t)(2 * k) * P + xo[i]);
        m1 = __ldg(M + (size_t)(2 * k + 1) * P + xo[i]);
      }
#pragma unroll
      for (int b = 0; b < SB; ++b) {
        acc[0][i][b] = fma(m0, xv[b], acc[0][i][b]);
        acc[1][i][b] = fma(m1, xv[b], acc[1][i][b]);
      }
    }
  }
}

// Shared memory of one warp tile: X [P][S] and U [2][P][S] doubles, the row's field factors [Lx][2], two rows
// of spin masks [Lx] and the row's bond dimensions [Lx + 1].  EDGE: the factors and dimensions stay in
// global memory, and a mask has only the bits of S samples.
template <int S, bool EDGE>
using F64Mask = std::conditional_t<!EDGE || (S > 16), uint32_t, std::conditional_t<(S > 8), uint16_t, uint8_t>>;
inline __host__ __device__ size_t f64_tile_smem(int P, int Lx, int S, bool edge) {
  const size_t work = 3 * (size_t)P * S * sizeof(double);
  if (edge) return work + (size_t)2 * Lx * (S > 16 ? 4 : S > 8 ? 2 : 1);
  return work + 2 * (size_t)Lx * sizeof(double) + ((size_t)3 * Lx + 1) * sizeof(uint32_t);
}

// The first dK rows of a site tensor into L1 (the warp's next contraction; its first loads
// would otherwise wait for L2 or DRAM with nothing else in flight).  Beyond P = 32 a
// contraction is long enough to cover them.
__device__ __forceinline__ void f64_prefetch(const double* M, int P, int dK, int lane) {
  if (P > 32) return;
  const int lines = (dK * P + 7) >> 3;       // 128-byte lines: 2 P doubles per row
  for (int l = lane; l < lines; l += 32)
    asm volatile("prefetch.global.L1 [%0];" ::"l"(reinterpret_cast<const char*>(M) + (size_t)l * 128));
}

// Samples base .. base+S-1 of the call (S = LS * SB <= 32, by one warp).  Bit s of a spin mask
// is sample base + s; lane s < S keeps the scalar state of sample s.  `stack`: [Lx+1][P][S].
// EDGE: wide rows (f64_tile_smem).
template <int LS, int SB, bool EDGE>
__device__ void sample_f64_tile(const SampleArgs<double>& a, int64_t base, unsigned char* smem, double* stack) {
  using Mask = F64Mask<LS * SB, EDGE>;
  constexpr int LO = 32 / LS, S = LS * SB, MAXNX = 64 / LO / SB, LP = 32 / S;
  const unsigned kFull = 0xffffffffu;
  const int Lx = a.e.Lx, Ly = a.e.Ly, P = a.e.P;
  const int lane = threadIdx.x & 31, sg = lane % LS, g = lane / LS;
  const int so = lane % S;                      // the sample whose scalars this lane computes
  double* X = reinterpret_cast<double*>(smem);
  double* U = X + (size_t)P * S;
  double* sfer = U + 2 * (size_t)P * S;
  Mask* prev = reinterpret_cast<Mask*>(sfer + (EDGE ? 0 : 2 * (size_t)Lx));
  Mask* cur = prev + Lx;
  int* sbond = reinterpret_cast<int*>(cur + Lx);
  const size_t n = (size_t)Lx * Ly, slot = (size_t)P * S;
  const uint64_t sample = a.offset + (uint64_t)(base + so);
  const int rows = (a.B - base) < S ? (int)(a.B - base) : S;
  double prod = 1.0;        // q of the drawn spins = prod 2^pexp, prod in [1, 2) or 0
  int pexp = 0, flag = 0;
  int64_t eacc = 0;         // fixed-point energy of sample lane % S over columns lane / S + LP j
  for (int c = lane; c < Lx; c += 32) prev[c] = 0u;
  __syncwarp();

  for (int r = 0; r < Ly; ++r) {
    const double* fer = a.fe + (size_t)r * Lx * 2;      // 1 on row 0
    const int* bond = a.e.bond + (size_t)r * (Lx + 1);
    if constexpr (!EDGE) {
      for (int c = lane; c <= Lx; c += 32) sbond[c] = a.e.bond[r * (Lx + 1) + c];
      for (int c = lane; c < 2 * Lx; c += 32) sfer[c] = r == 0 ? 1.0 : a.fe[(size_t)r * Lx * 2 + c];
      fer = sfer;
      bond = sbond;
    }
    const size_t tstride = (size_t)P * 2 * P;
    const double* Lrow = a.L + (size_t)r * Lx * tstride;
    const double* Rrow = a.Rt + (size_t)r * Lx * tstride;
    const bool snake = a.e.order == 1 && (r & 1);
    if (a.spins_in) {
      for (int c = lane; c < Lx; c += 32) {
        const int8_t* src = a.spins_in + (size_t)base * n + (size_t)r * Lx + c;
        uint32_t m = 0;
#pragma unroll 4
        for (int s = 0; s < rows; ++s) m |= (src[s * n] > 0 ? 1u : 0u) << s;
        cur[c] = m;
      }
    }
    // ---- first sweep (no draws): right to left, or left to right on a snake row ----
    {
      double* end = stack + (snake ? 0 : (size_t)Lx * slot);
      if (lane < S) X[lane] = end[lane] = 1.0;      // boundary bonds have dimension 1
    }
    __syncwarp();
    int elag[SB];     // exponent of the last vector's largest entry, divided out one step later
#pragma unroll
    for (int b = 0; b < SB; ++b) elag[b] = 0;
    for (int j = 0; j + 1 < Lx; ++j) {
      const int c = snake ? j : Lx - 1 - j;
      const int dl = bond[c], dr = bond[c + 1];
      const int dK = snake ? dl : dr, dX = snake ? dr : dl;
      const double* M = (snake ? Lrow : Rrow) + c * tstride;
      {
        const int cn = snake ? c + 1 : c - 1;      // the next tensor of this sweep, or the first of the next one
        if (j + 2 < Lx) f64_prefetch((snake ? Lrow : Rrow) + cn * tstride, P, bond[snake ? cn : cn + 1], lane);
        else f64_prefetch((snake ? Rrow : Lrow) + cn * tstride, P, 1, lane);
      }
      double* out = stack + (size_t)(snake ? c + 1 : c) * slot;
      const uint32_t up = prev[c];
      const double fdiff = fer[2 * c], fsame = fer[2 * c + 1];
      auto step = [&](auto nxc, auto rt) {
        constexpr int NX = decltype(nxc)::value;
        double acc[2][NX][SB];
        f64_contract<LS, SB, NX, decltype(rt)::value != 0>(M, P, dK, X, g, sg, acc);
        __syncwarp();
#pragma unroll
        for (int b = 0; b < SB; ++b) {
          const bool u = (up >> (sg + LS * b)) & 1u;
          const double fm = scale_down_f64(u ? fdiff : fsame, elag[b]), fp = scale_down_f64(u ? fsame : fdiff, elag[b]);
          int mh = 0;
#pragma unroll
          for (int i = 0; i < NX; ++i) {
            const int x = g + LO * i;
            const double v = fma(fm, acc[0][i][b], fp * acc[1][i][b]);
            if (x < dX) {
              X[x * S + sg + LS * b] = v;
              out[x * S + sg + LS * b] = v;
              mh = max(mh, __double2hiint(v) & 0x7fffffff);
            }
          }
#pragma unroll
          for (int o = LS; o < 32; o <<= 1) mh = max(mh, __shfl_xor_sync(kFull, mh, o));
          elag[b] = exponent_f64(mh);
        }
        __syncwarp();
      };
      const int nx = (dX + LO - 1) / LO;
      if (snake) by_count<MAXNX>(nx, [&](auto k) { step(k, IntC<0>{}); });
      else by_count<MAXNX>(nx, [&](auto k) { step(k, IntC<1>{}); });
    }
    // ---- second sweep: the draws ----
    if (lane < S) X[lane] = 1.0;
    __syncwarp();
    for (int j = 0; j < Lx; ++j) {
      const int c = snake ? Lx - 1 - j : j;
      const int dl = bond[c], dr = bond[c + 1];
      const int dK = snake ? dr : dl, dX = snake ? dl : dr;
      const double* M = (snake ? Rrow : Lrow) + c * tstride;
      if (j + 1 < Lx) {
        const int cn = snake ? c - 1 : c + 1;
        f64_prefetch((snake ? Rrow : Lrow) + cn * tstride, P, bond[snake ? cn + 1 : cn], lane);
      }
      const double* in = stack + (size_t)(snake ? c : c + 1) * slot;
      const bool u = (prev[c] >> so) & 1u;
      const double fdiff = fer[2 * c], fsame = fer[2 * c + 1];
      const double fm = u ? fdiff : fsame, fp = u ? fsame : fdiff;
      const uint64_t word = a.spins_in ? 0ull : draw_word(a.seed, (int64_t)r * Lx + c, sample);
      auto step = [&](auto nxc, auto rt) {
        constexpr int NX = decltype(nxc)::value;
        double acc[2][NX][SB];
        f64_contract<LS, SB, NX, decltype(rt)::value != 0>(M, P, dK, X, g, sg, acc);
#pragma unroll
        for (int i = 0; i < NX; ++i)
#pragma unroll
          for (int b = 0; b < SB; ++b) {
            const int x = g + LO * i;
            if (x < dX) {
              U[x * S + sg + LS * b] = acc[0][i][b];
              U[(P + x) * S + sg + LS * b] = acc[1][i][b];
            }
          }
        __syncwarp();
        double w0 = 0.0, w1 = 0.0;
        if constexpr (S == 32) {
#pragma unroll 4
          for (int x = 0; x < dX; ++x) {
            const double rx = in[x * S + lane];
            w0 = fma(U[x * S + lane], rx, w0);
            w1 = fma(U[(P + x) * S + lane], rx, w1);
          }
          w0 = clamp0_f64(w0 * fm);
          w1 = clamp0_f64(w1 * fp);
        } else {       // lane = sample + S spin
          const bool hi = (lane / S) & 1;
          const double* us = U + (hi ? (size_t)P * S : 0);
          double w = 0.0;
#pragma unroll 4
          for (int x = 0; x < dX; ++x) w = fma(us[x * S + so], in[x * S + so], w);
          w = clamp0_f64(w * (hi ? fp : fm));
          const double other = __shfl_xor_sync(kFull, w, S);
          w0 = hi ? other : w;
          w1 = hi ? w : other;
        }
        const double tot = w0 + w1;
        const int te = (__double2hiint(tot) >> 20) & 0x7ff;
        const bool bad = te == 2047 || __double_as_longlong(tot) == 0;
        // p(+) for the draw, p(s) for log q.  The draw compares with 64 uniform bits, which a unit in
        // p's last place moves with probability 2^-53: the product will do, off the residual step's
        // latency
        const bool mid = te > 64 && te < 1980;
        double ri = 0.0, pplus, pd;
        if (mid) {
          ri = reciprocal_f64(tot);
          pplus = w1 * ri;
        } else {
          pplus = w1 / tot;
        }
        if (__double_as_longlong(w0) == 0) pplus = 1.0;     // one weight zero: exact
        if (bad) pplus = 0.5;
        const bool plus = a.spins_in ? (cur[c] >> so) & 1u : draw_plus_bits(pplus, word);
        const double wd = plus ? w1 : w0;
        if (mid) pd = quotient_f64(wd, tot, ri);
        else pd = bad ? 0.5 : wd / tot;
        prod *= pd;
        {
          int hi = __double2hiint(prod);
          if ((hi >> 20) == 0 && prod != 0.0) {      // subnormal: exact shift into the normal range
            prod *= 0x1.0p54;
            pexp -= 54;
            hi = __double2hiint(prod);
          }
          if ((hi >> 20) != 0) {                     // zero stays zero
            pexp += (hi >> 20) - 1023;
            prod = __hiloint2double((hi & 0xfffff) | (1023 << 20), __double2loint(prod));
          }
        }
        flag |= bad ? TNMC_FLAG_NUMERIC : 0;
        // next vector: f(s) U[s] times 2^-ilogb(w(s)), so that <next, R> lands in [1, 2)
        const double ws = plus ? w1 : w0, fs = plus ? fp : fm;
        double mult = fs * pow2_f64(-exponent_f64(__double2hiint(ws)));
        const uint32_t mask = __ballot_sync(kFull, plus);     // bit s: lane s owns sample s
        const int we = __double2hiint(ws) >> 20;
        if (__any_sync(kFull, we == 0 || we == 2047)) {
          // a drawn weight that is zero or not finite gives no scale: those samples take it from
          // max |f(s) U[s]|
          int mb[SB];
#pragma unroll
          for (int b = 0; b < SB; ++b) {
            const bool pb = (mask >> (sg + LS * b)) & 1u;
            const double fb = SB == 1 ? fs : __shfl_sync(kFull, fs, sg + LS * b);
            mb[b] = 0;
#pragma unroll
            for (int i = 0; i < NX; ++i)
              if (g + LO * i < dX) mb[b] = max(mb[b], __double2hiint((pb ? acc[1][i][b] : acc[0][i][b]) * fb) & 0x7fffffff);
#pragma unroll
            for (int o = LS; o < 32; o <<= 1) mb[b] = max(mb[b], __shfl_xor_sync(kFull, mb[b], o));
          }
          int mo = mb[0];
#pragma unroll
          for (int b = 1; b < SB; ++b) mo = so / LS == b ? mb[b] : mo;
          if (we == 0 || we == 2047) mult = fs * pow2_f64(-exponent_f64(mo));
        }
        if (!a.spins_in && lane == 0) cur[c] = mask;
#pragma unroll
        for (int b = 0; b < SB; ++b) {
          const double mu = SB == 1 ? mult : __shfl_sync(kFull, mult, sg + LS * b);
          const bool pb = (mask >> (sg + LS * b)) & 1u;
#pragma unroll
          for (int i = 0; i < NX; ++i) {
            const int x = g + LO * i;
            if (x < dX) X[x * S + sg + LS * b] = (pb ? acc[1][i][b] : acc[0][i][b]) * mu;
          }
        }
        __syncwarp();
      };
      const int nx = (dX + LO - 1) / LO;
      if (snake) by_count<MAXNX>(nx, [&](auto k) { step(k, IntC<1>{}); });
      else by_count<MAXNX>(nx, [&](auto k) { step(k, IntC<0>{}); });
    }
    // ---- row end: energy terms, spins, and this row becomes the previous one ----
    {
      const int s = lane % S;
      for (int c = lane / S; c < Lx; c += LP) {
        int64_t q = a.e.qh[(size_t)r * Lx + c];
        if (c > 0) {
          const int64_t j = a.e.qJh[(size_t)r * (Lx - 1) + c - 1];
          q += ((cur[c - 1] >> s) & 1u) ? j : -j;
        }
        if (r > 0) {
          const int64_t j = a.e.qJv[(size_t)(r - 1) * Lx + c];
          q += ((prev[c] >> s) & 1u) ? j : -j;
        }
        eacc -= ((cur[c] >> s) & 1u) ? q : -q;
      }
    }
    __syncwarp();
    for (int c = lane; c < Lx; c += 32) {
      const uint32_t m = cur[c];
      if (a.spins_out && !a.spins_in) {
        int8_t* dst = a.spins_out + (size_t)base * n + (size_t)r * Lx + c;
        for (int s = 0; s < rows; ++s) dst[s * n] = ((m >> s) & 1u) ? 1 : -1;
      }
      prev[c] = m;
    }
    __syncwarp();
  }
#pragma unroll
  for (int o = S; o < 32; o <<= 1) eacc += __shfl_xor_sync(kFull, eacc, o);
  if (lane < rows) {
    // a flagged sample keeps the log of the probability it was drawn with (log 1/2 at a site
    // whose normaliser failed): q stays the exact law of the sampler
    a.logq[base + lane] = log(prod) + (double)pexp * 0.69314718055994530942;
    a.energy[base + lane] = scalbn((double)eacc, a.e.qexp);
    if (a.flags) a.flags[base + lane] = flag;
    if (flag) set_status(a.e.status, TNMC_E_NUMERIC);
  }
  __syncwarp();
}

// At least 12 warps per SM resident (168 registers): the FP64 pipe needs 4 with an instruction
// ready, the others cover shared-memory, shuffle and load latencies.
constexpr int kF64MinWarps = 12;

// One warp per CTA: tiles are handed out in single warps, so that a few thousand samples
// spread evenly over the SMs.  Scratch: one stack [Lx+1][P][S] per CTA.
template <int LS, int SB, bool EDGE>
__global__ void __launch_bounds__(32, kF64MinWarps) sample_f64_kernel(SampleArgs<double> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int S = LS * SB;
  double* stack = a.scratch + (size_t)blockIdx.x * (a.e.Lx + 1) * a.e.P * S;
  for (int64_t base = (int64_t)blockIdx.x * S; base < a.B; base += (int64_t)gridDim.x * S)
    sample_f64_tile<LS, SB, EDGE>(a, base, smem_raw, stack);
}

// The tile shape (samples per warp) for `total` samples on `nsm` SMs at pad P.  Larger tiles
// share the scalar work, but an SM needs several warps to fill its FP64 pipe: the largest tile
// that still leaves kF64WarpsPerSM warps per SM, and at most 64 / P samples per lane (the
// accumulators' registers).  Measured, ms per launch at S = 2 / 4 / 8 / 16 / 32: 16 x 20, chi = 13
// (P = 16): 2048 samples 1.47 / 1.64 / 2.40 / 3.84 / 6.75, 10000 6.02 / 4.54 / 4.19 / 4.63 / 6.76,
// 80000 46.7 / 31.9 / 26.8 / 26.6 / 27.1; 8 x 8, chi = 8: 10000 0.80 / 0.48 / 0.31 / 0.30 / 0.44.
constexpr int kF64WarpsPerSM = 6;
inline int f64_tile_samples(int64_t total, int P, int nsm) {
  int S = 32;
  while (S > 2 && (S / 8 * P > 64 || (total + S - 1) / S < (int64_t)kF64WarpsPerSM * nsm)) S >>= 1;
  return S;
}

// The launch of `total` samples: samples per warp, the kernel's form and its shared memory.
// need(S, edge): bytes of a CTA of one warp.
//
// The EDGE form where the plain one would leave an SM fewer than its 12 warps (from about 500 columns
// on: it costs up to 4 % itself), and there at most 16 samples where more would leave fewer than 7.
// Measured, ms, plain form / the rule's: 8192 samples of 5 x 4096, chi 16 1190 / 212, of 4 x 2048, chi 8
// 114 / 43; 32768 of 4 x 4096, chi 8 1130 / 282 (32 samples per warp: 350).
struct F64Plan {
  int S;
  bool edge;
  size_t smem;
};
template <class Need>
F64Plan f64_plan(int64_t total, int P, int nsm, size_t smem_sm, Need&& need) {
  F64Plan p{f64_tile_samples(total, P, nsm), false, 0};
  auto warps = [&](int S, bool edge) { return (int)(smem_sm / (need(S, edge) + 1024)); };
  p.edge = warps(p.S, false) < kF64MinWarps;
  if (p.edge && p.S == 32 && warps(32, true) < 7) p.S = 16;
  p.smem = need(p.S, p.edge);
  return p;
}

// f(IntC<LS>, IntC<SB>, bool constant EDGE) for a plan's kernel
template <class F>
tnmc_status by_f64_tile(const F64Plan& p, F&& f) {
  auto form = [&](auto ls, auto sb) -> tnmc_status {
    return p.edge ? f(ls, sb, std::true_type{}) : f(ls, sb, std::false_type{});
  };
  switch (p.S) {
    case 32: return form(IntC<8>{}, IntC<4>{});
    case 16: return form(IntC<8>{}, IntC<2>{});
    case 8: return form(IntC<8>{}, IntC<1>{});
    case 4: return form(IntC<4>{}, IntC<1>{});
    default: return form(IntC<2>{}, IntC<1>{});
  }
}

}  // namespace
}  // namespace tnmc
