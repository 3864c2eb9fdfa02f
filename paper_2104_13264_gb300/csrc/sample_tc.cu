// BF16 tensor-core sampler / evaluator of q = pi~ (Sec. 2, eqs. bayes, pi-approx;
// App. A) for sm_103a: tcgen05.mma with the accumulator in TMEM, environment tiles
// streamed into shared memory by bulk async copies, FP32 accumulation.
//
// A CTA owns a tile of 128 samples (UMMA M = 128): sample t is TMEM lane t.  Per
// site one UMMA 128 x 128 x 64 forms, for all samples at once,
//   right sweep  D[t][(u, a)] = sum_b R_{c+1}[t][b] Mt^(u)_c[a][b]   -> R_c = D(u_t, -)
//   left sweep   D[t][(s, b)] = sum_a Lambda_c[t][a] M_c[a][s][b]     -> U[s] = D(s, -)
// where Mt^(u) = sum_s f_u(s) M[:, s, :] is the site tensor with the field factor of the
// spin above (u) already applied (both u at once; the epilogue keeps the sample's own),
// with the vectors (A operand, 128 x 64) in TMEM and the environment tile (B operand,
// 128 x 64) loaded from a pre-swizzled copy of the environment.  Both operands are BF16
// hi + lo pairs; the three products hi*hi + lo*hi + hi*lo keep about 16 significant bits
// (the lo*lo term is below that).
//
// 320 threads.  Warps 0-7 are the epilogue: thread (t, h) = (tid % 128, tid / 128) handles
// sample t for the components k in [32h, 32h + 32) -- warps w and w + 4 read the same TMEM
// lanes (lane quadrant w % 4) at different columns, 16 columns per load -- and writes the next
// A operand straight back to TMEM.  Warp 8 issues the UMMAs; warp 9 refills the ring of
// environment tiles and makes the sites' Philox words one left step ahead.  The two epilogue
// halves exchange their partial maxima (every other right step; every one with strong
// vertical bonds) or partial dot products (left steps) through shared memory and take identical decisions from identical sums.
// Every rescaling is by a power of two, which leaves the arithmetic of q unchanged: right
// vectors by their max, left vectors by the drawn weight w(s).
//
// The left sweep needs R_{c+1} in the reverse of the order the right sweep makes it: every
// thread writes its half of R_c to a per-CTA stack in global memory (Lx x 32 KB per tile and
// row, 512 B per warp store) and reads the same values back into its own shared-memory slots
// with cp.async while the step's UMMA runs.  Steps per row: (Lx - 1) right + Lx left.
//
// What bounds it: the serial chain of a step (UMMA about 1000 cycles of which 768 are tensor
// work, then TMEM reads, the split into hi + lo, the barrier) with 2 CTAs per SM to overlap it,
// and past that the stack's HBM traffic.  Measured on the 8 x 96, chi = 64 strip with 65536
// samples, 8.3 ms before:
//   A operand in TMEM, R through registers (spills), one thread issuing everything: 12.6 ms -- a
//     tile refill costs its thread several hundred cycles, paid between UMMA and epilogue;
//   UMMA, refill and Philox on warps of their own, spins as column masks: 8.4 ms;
//   R through shared-memory slots (no spills), two operations per FP32 instruction, the draw's
//     log-probability factor deferred into the next UMMA: 6.6 ms;
//   both TMEM halves read at once instead of 16 columns at a time, or scalar FP32: 4-5 % slower.
#include <math.h>
#include <stdlib.h>

#include "common.cuh"
#include "umma.cuh"

namespace tnmc {
namespace {

constexpr int kTile = 128;          // samples per CTA (UMMA M)
constexpr int kThreads = 320;       // two epilogue threads per sample (8 warps), an UMMA warp, a producer warp
constexpr int kK = 64;              // padded bond dimension (UMMA K per site)
constexpr int kN = 128;             // 2 x 64 outputs (UMMA N)
constexpr uint32_t kTileBytes = kN * kK * 2;   // 16 KiB: one BF16 operand tile
constexpr uint32_t kStageBytes = 2 * kTileBytes;   // hi + lo tiles of one (r, c)
constexpr int kMaxCols = 3968;      // widest row
constexpr int kStages = 2;          // environment tiles in flight
constexpr uint32_t kRBytes = kTile * kK * 4;   // 32 KiB: R_{c+1} of the tile, FP32
constexpr uint32_t kTmemCols = 256; // 128 accumulator columns, 32 + 32 of the A operand (hi, lo)
constexpr uint32_t kColHi = 128, kColLo = 160;
constexpr uint32_t kPollLimit = 1u << 16;    // polls of a bounded wait ...
constexpr uint32_t kPollHintNs = 1u << 16;   // ... each parked up to ~65 us: at most ~4 s

struct TcArgs {
  DeviceEnv e;
  const __nv_bfloat16* TR;   // [Ly*Lx] right-sweep tiles (n = s*64 + a, k = b), SW128
  const __nv_bfloat16* TL;   // [Ly*Lx] left-sweep tiles  (n = s*64 + b, k = a), SW128
  const float* fe;           // [Ly][Lx][2]
  int64_t B;
  uint64_t seed, offset;
  const int8_t* spins_in;
  int8_t* spins_out;
  double* logq;
  double* energy;
  int32_t* flags;
  float4* stack;             // per CTA: [Lx][2 halves][8 chunks][128 samples] float4
  uint32_t poll_limit;       // polls of each wait inside the sampling loop (kPollLimit;
                             // 0 makes every such wait give up at once)
};

__device__ inline float pow2f(int e) { return __int_as_float((e + 127) << 23); }   // 2^e, |e| < 127
__device__ inline int ilogb_f(float x) { return ((__float_as_int(x) >> 23) & 0xff) - 127; }   // x normal, > 0

// Split 16 FP32 values (components k0 .. k0+15 of this thread's sample) into BF16 hi + lo and
// write them to the A operand in TMEM (a_hi, a_lo: the columns of component k0).
__device__ inline void store_split16(uint32_t a_hi, uint32_t a_lo, const float2* v) {
  uint32_t wh[8], wl[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const __nv_bfloat162 h2 = __floats2bfloat162_rn(v[q].x, v[q].y);
    wh[q] = *reinterpret_cast<const uint32_t*>(&h2);
    const float2 hf = make_float2(__uint_as_float(wh[q] << 16), __uint_as_float(wh[q] & 0xffff0000u));
    const float2 lo = umma::f2_fma(hf, make_float2(-1.0f, -1.0f), v[q]);      // v - hi, exact
    const __nv_bfloat162 l2 = __floats2bfloat162_rn(lo.x, lo.y);
    wl[q] = *reinterpret_cast<const uint32_t*>(&l2);
  }
  umma::tmem_st8(a_hi, wh);
  umma::tmem_st8(a_lo, wl);
}

// e_0 restricted to this thread's half, as the A operand
__device__ inline void store_unit(uint32_t a_hi, uint32_t a_lo, int h) {
#pragma unroll
  for (int ch = 0; ch < 2; ++ch) {
    float2 v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = make_float2((h == 0 && ch == 0 && q == 0) ? 1.0f : 0.0f, 0.0f);
    store_split16(a_hi + 8 * ch, a_lo + 8 * ch, v);
  }
}

__device__ inline void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(umma::smem_u32(dst)), "l"(src) : "memory");
}
__device__ inline void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ inline void pair_sync(int warp) {
  asm volatile("bar.sync %0, 64;" ::"r"(1 + (warp & 3)) : "memory");
}

// The row's field factors and the masks of its own spins are in shared memory.  EDGE: wide rows,
// where the factors are read from the environment and the masks kept behind the stacks in global
// scratch, and strong vertical bonds.
template <bool EDGE>
__global__ void __launch_bounds__(kThreads, 2) sample_tc_kernel(TcArgs a) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  unsigned char* sB = base;                                                   // [kStages] environment tiles (hi, lo)
  float4* sR = reinterpret_cast<float4*>(sB + kStages * kStageBytes);        // [8][256]: each thread's R_{c+1}
  uint64_t* bars = reinterpret_cast<uint64_t*>(sB + kStages * kStageBytes + kRBytes);   // [0 .. kStages-1] tiles, [kStages] UMMA
  uint32_t* misc = reinterpret_cast<uint32_t*>(bars + kStages + 1);          // [0] tmem base, [1] abort, [2] tile ok
  // the producer's copy counter lives in shared memory, where the teardown reads it: environment tiles
  // whose copy was issued
  int64_t* cnt = reinterpret_cast<int64_t*>(misc + 4);
  float* xw = reinterpret_cast<float*>(misc + 6);   // left steps: [2 halves][2][128] partial w(-), w(+)
  float* xmb = xw + 4 * kTile;                      // right steps: [step parity][2 halves][128] partial max
  const int Lx = a.e.Lx, Ly = a.e.Ly;
  uint32_t* xs = reinterpret_cast<uint32_t*>(xw + 8 * kTile);   // [2 pairs][2 sites][2][128]: 64-bit uniforms
  uint32_t* prev = xs + 8 * kTile;                              // [Lx][4]: spins of the row above, one bit a sample
  uint32_t* cur = !EDGE ? prev + 4 * Lx
                        : reinterpret_cast<uint32_t*>(a.stack + (size_t)gridDim.x * Lx * (2 * 8 * kTile)) +
                               (size_t)blockIdx.x * 4 * Lx;

  const int tid = threadIdx.x, warp = tid >> 5;
  const bool ctrl = warp >= 8;                          // the UMMA warp (8) and the producer warp (9)
  const bool lead = tid == 256, prod_lead = tid == 288;      // their elected threads
  const int t = tid & (kTile - 1), h = (tid >> 7) & 1;
  const int64_t ntiles = (a.B + kTile - 1) / kTile;
  const int S = 2 * Lx - 1;
  const int64_t my_tiles = (ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x;
  const int64_t total_steps = my_tiles * (int64_t)Ly * S;
  const int n = Lx * Ly;
  float4* stk_cta = a.stack + (size_t)blockIdx.x * Lx * (2 * 8 * kTile);
  float4* stk = stk_cta + (size_t)h * (8 * kTile) + t;
  const uint32_t idesc = umma::idesc_bf16_f32(kTile, kN);
  const int ksteps = (a.e.P + 15) >> 4;

  if (warp == 0) umma::tmem_alloc(umma::smem_u32(&misc[0]), kTmemCols);
  if (tid == 0) {
    for (int s = 0; s <= kStages; ++s) umma::mbar_init(umma::smem_u32(&bars[s]), 1);
    umma::fence_mbar_init();
    misc[1] = 0;
    misc[2] = 1;
    cnt[0] = 0;
  }
  umma::fence_before_sync();
  __syncthreads();
  umma::fence_after_sync();
  const uint32_t tmem = misc[0];
  const uint32_t tquad = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
  const uint32_t tlane = tquad + 32 * h, a_hi = tquad + kColHi + 16 * h, a_lo = tquad + kColLo + 16 * h;

  // producer position (row, step within the row) of the next tile to load
  int prod_r = 0, prod_i = 0;
  auto next_tile = [&]() -> const __nv_bfloat16* {
    const bool left = prod_i >= Lx - 1;
    const int c = left ? prod_i - (Lx - 1) : Lx - 1 - prod_i;
    const __nv_bfloat16* T = (left ? a.TL : a.TR) + ((size_t)prod_r * Lx + c) * (2 * kN * kK);
    if (++prod_i == S) {
      prod_i = 0;
      if (++prod_r == Ly) prod_r = 0;
    }
    return T;
  };

  if (prod_lead) {
    for (int s = 0; s < kStages && s < total_steps; ++s) {
      umma::mbar_expect_tx(umma::smem_u32(&bars[s]), kStageBytes);
      umma::bulk_g2s(umma::smem_u32(sB + s * kStageBytes), next_tile(), kStageBytes, umma::smem_u32(&bars[s]));
      cnt[0] = s + 1;
    }
  }
  int stage = 0;                     // ring stage of the current step ...
  uint32_t stage_par = 0;            // ... and the parity of its copy

  int64_t g = 0;
  bool abort = false;
  for (int64_t tile = blockIdx.x; tile < ntiles && !abort; tile += gridDim.x) {
    const int64_t b = tile * kTile + t;
    const bool active = b < a.B;
    double lq = 0.0;
    int64_t eacc = 0;            // fixed-point energy over the columns c = h mod 2
    int flag = 0;
    for (int q = tid; q < 4 * Lx; q += kThreads) prev[q] = 0u;
    // producer warp: the uniforms of a site pair, in the buffer of the pair's parity (each is read
    // at most two left steps later, when the other buffer is being written)
    int64_t pair_id = -1;
    auto make_uniforms = [&](int64_t site) {
      if ((site >> 1) == pair_id) return;
      pair_id = site >> 1;
      uint32_t* dst = xs + (pair_id & 1) * (4 * kTile) + (tid & 31);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint64_t id = a.offset + (uint64_t)(tile * kTile + 32 * q + (tid & 31));
        const U4 o = philox4x32_10(U4{(uint32_t)pair_id, (uint32_t)id, (uint32_t)(id >> 32), 0u}, (uint32_t)a.seed,
                                   (uint32_t)(a.seed >> 32));
        dst[32 * q] = o.x;
        dst[kTile + 32 * q] = o.y;
        dst[2 * kTile + 32 * q] = o.z;
        dst[3 * kTile + 32 * q] = o.w;
      }
    };
    for (int r = 0; r < Ly && !abort; ++r) {
      const float* fe_row = a.fe + (size_t)r * Lx * 2;     // [Lx][2]: field factors of the row; 1 on row 0
      if constexpr (!EDGE) {
        float* sfe = reinterpret_cast<float*>(cur + 4 * Lx);
        for (int q = tid; q < 2 * Lx; q += kThreads) sfe[q] = fe_row[q];
        fe_row = sfe;
      }
      if (a.spins_in && warp < 4) {
        const int64_t b0 = tile * kTile + 32 * warp;
        const int ns = (a.B - b0) < 32 ? (int)(a.B - b0) : 32;
        for (int c = tid & 31; c < Lx; c += 32) {
          const int8_t* src = a.spins_in + (size_t)b0 * n + (size_t)r * Lx + c;
          uint32_t m = 0;
#pragma unroll 8
          for (int q = 0; q < ns; ++q) m |= (src[(size_t)q * n] > 0 ? 1u : 0u) << q;
          cur[4 * c + warp] = m;
        }
      }
      if (warp == 9 && !a.spins_in) make_uniforms((int64_t)r * Lx);
      // row start: A = R_{Lx} = e_0 (Lx > 1) or Lambda_0 = e_0 (Lx = 1), whose max is 1
      if (!ctrl) {
        store_unit(a_hi, a_lo, h);
        umma::tmem_wait_st();
      }
      float prod = 1.0f;
      int pexp = 0;
      float pend_w = 0.0f, pend_tot = -1.0f;      // w(s) and w(-) + w(+) of the last drawn site
      umma::fence_before_sync();
      __syncthreads();
      for (int i = 0; i < S; ++i, ++g) {
        const bool left = i >= Lx - 1;
        const int c = left ? i - (Lx - 1) : Lx - 1 - i;
        umma::fence_after_sync();
        if (ctrl) {
          if (lead) {
            // ---- UMMA warp ----
            const bool tile_ok =
                umma::mbar_wait_parked(umma::smem_u32(&bars[stage]), stage_par, a.poll_limit, kPollHintNs);
            misc[2] = tile_ok;
            if (!tile_ok) {
              set_status(a.e.status, TNMC_E_TIMEOUT);
              misc[1] = 1;
            } else {
              const uint64_t bh = umma::sw128_desc(umma::smem_u32(sB + stage * kStageBytes));
              const uint64_t bl = umma::sw128_desc(umma::smem_u32(sB + stage * kStageBytes + kTileBytes));
              // K beyond the bond dimension is zero in both operands: those products add nothing
#pragma unroll
              for (int k = 0; k < kK / 16; ++k)
                if (k < ksteps) umma::mma_bf16_ta(tmem, tmem + kColHi + 8 * k, bh + 2 * k, idesc, k > 0);
#pragma unroll
              for (int k = 0; k < kK / 16; ++k)
                if (k < ksteps) umma::mma_bf16_ta(tmem, tmem + kColLo + 8 * k, bh + 2 * k, idesc, 1);
#pragma unroll
              for (int k = 0; k < kK / 16; ++k)
                if (k < ksteps) umma::mma_bf16_ta(tmem, tmem + kColHi + 8 * k, bl + 2 * k, idesc, 1);
            }
            umma::mma_commit(umma::smem_u32(&bars[kStages]));
          } else if (warp == 9) {
            // ---- producer warp: the previous step's stage (every epilogue thread has waited for that
            // step's UMMA before the step's barrier) takes the tile kStages steps on; then the
            // uniforms of the next left step's site ----
            if (prod_lead && g > 0 && cnt[0] < total_steps) {
              const int ps = stage == 0 ? kStages - 1 : stage - 1;
              umma::mbar_expect_tx(umma::smem_u32(&bars[ps]), kStageBytes);
              umma::bulk_g2s(umma::smem_u32(sB + ps * kStageBytes), next_tile(), kStageBytes, umma::smem_u32(&bars[ps]));
              ++cnt[0];
            }
            __syncwarp();
            if (left && c + 1 < Lx && !a.spins_in) make_uniforms((int64_t)r * Lx + c + 1);
          }
          if (++stage == kStages) {
            stage = 0;
            stage_par ^= 1u;
          }
          __syncthreads();
          if (misc[1]) {
            abort = true;
            break;
          }
          continue;
        }
        // left steps: R_{c+1} of this thread's half (this thread wrote it) into this thread's slots of
        // the R buffer while the UMMA runs; registers are the scarce resource
        if (left) {
          if (c + 1 < Lx) {
            const float4* src = stk + (size_t)(c + 1) * (2 * 8 * kTile);
#pragma unroll
            for (int j = 0; j < 8; ++j) cp_async16(sR + j * 256 + tid, src + j * kTile);
          } else {
#pragma unroll
            for (int j = 0; j < 8; ++j)
              sR[j * 256 + tid] = make_float4((h == 0 && j == 0) ? 1.0f : 0.0f, 0.0f, 0.0f, 0.0f);
          }
        }
        // work that does not need the accumulator, overlapped with the UMMA
        const bool up = (prev[4 * c + (warp & 3)] >> (tid & 31)) & 1u;
        const float fsame = fe_row[2 * c + 1], fdiff = fe_row[2 * c];
        const float fm = up ? fdiff : fsame;   // s = -1
        const float fp = up ? fsame : fdiff;   // s = +1
        if (left && c + 2 < Lx) {
          // R_{c+2} into L2 one step ahead: each lane fetches one of its warp's 32 lines
          const int lane = tid & 31;
          const float4* pf = stk - t + 32 * (warp & 3) + (size_t)(c + 2) * (2 * 8 * kTile) +
                             (size_t)(lane >> 2) * kTile + 8 * (lane & 3);
          asm volatile("prefetch.global.L2 [%0];" ::"l"(pf));
        }
        // the previous left step's factor of log q, off that step's critical path
        if (h == 0 && pend_tot >= 0.0f) {
          const bool bad = !(pend_tot > 0.0f) || !isfinite(pend_tot);
          prod *= bad ? 0.5f : pend_w / pend_tot;
          if (prod < 0x1.0p-60f && prod > 0.0f) {
            prod *= 0x1.0p60f;
            pexp -= 60;
          }
          flag |= bad ? TNMC_FLAG_NUMERIC : 0;
          pend_tot = -1.0f;
        }
        const bool mma_ok =
            umma::mbar_wait_parked(umma::smem_u32(&bars[kStages]), (uint32_t)(g & 1), a.poll_limit, kPollHintNs);
        if (!mma_ok) {
          set_status(a.e.status, TNMC_E_TIMEOUT);
          misc[1] = 1;
        }
        umma::fence_after_sync();
        if (!left) {
          // ---- right-sweep epilogue: R_c = Mt^(u)_c R_{c+1} for this sample's u (the spin
          // above): the UMMA formed both u halves, the epilogue selects one ----
          // every other step rescales by the power of two of the previous A operand's largest entry
          // (the odd steps record both halves' partial maxima, exchanged through the step barrier):
          // the operand stays within two steps' growth of [1, 2) and the accumulator within three,
          // which fit FP32 up to beta |Jv| = 29.  With stronger bonds (EDGE) every step records and
          // rescales: the accumulator holds two steps' growth, up to 44.
          const bool every = EDGE && a.e.strong;
          const bool record = every || (i & 1), scale = every || !(i & 1);
          const int rd = every ? ((i + 1) & 1) * (2 * kTile) : 0;      // the previous step's maxima
          float2 sc = make_float2(1.0f, 1.0f);
          if (scale && i > 0) {
            const float mprev = fmaxf(xmb[rd + t], xmb[rd + kTile + t]);
            if (mprev > 0x1.0p-126f && mprev < INFINITY) sc.x = sc.y = pow2f(-ilogb_f(mprev));
          }
          float m4[4] = {0.0f, 0.0f, 0.0f, 0.0f};   // four independent chains (max is exact)
          float4* dst = stk + (size_t)c * (2 * 8 * kTile);
#pragma unroll
          for (int ch = 0; ch < 2; ++ch) {
            uint32_t d[16], e[16];
            umma::tmem_ld16_issue(tlane + 16 * ch, d);
            umma::tmem_ld16_issue(tlane + 64 + 16 * ch, e);
            umma::tmem_wait_ld();
            umma::tmem_hold16(d);
            umma::tmem_hold16(e);
            float2 v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q)
              v[q] = make_float2(__uint_as_float(up ? e[2 * q] : d[2 * q]), __uint_as_float(up ? e[2 * q + 1] : d[2 * q + 1]));
            if (EDGE && every) {
#pragma unroll
              for (int q = 0; q < 8; ++q) v[q] = umma::f2_mul(v[q], sc);
            }
            if (record) {
#pragma unroll
              for (int q = 0; q < 8; ++q) m4[q & 3] = fmaxf(m4[q & 3], fmaxf(fabsf(v[q].x), fabsf(v[q].y)));
            } else {
#pragma unroll
              for (int q = 0; q < 8; ++q) v[q] = umma::f2_mul(v[q], sc);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
              __stcg(dst + (4 * ch + j) * kTile, make_float4(v[2 * j].x, v[2 * j].y, v[2 * j + 1].x, v[2 * j + 1].y));
            if (c > 1) store_split16(a_hi + 8 * ch, a_lo + 8 * ch, v);
          }
          if (c == 1) store_unit(a_hi, a_lo, h);           // the left sweep starts from Lambda_0 = e_0
          umma::tmem_wait_st();
          if (record)
            xmb[(every ? (i & 1) * (2 * kTile) : 0) + h * kTile + t] = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
        } else {
          // ---- left-sweep epilogue: w(s) = f(s) <U[s], R_{c+1}>, draw, Lambda_{c+1} ----
          cp_async_wait_all();
          // pass 1: partial dot products over this half, 16 components at a time
          float2 a0[2] = {make_float2(0.0f, 0.0f), make_float2(0.0f, 0.0f)};      // chains of components mod 4
          float2 a1[2] = {make_float2(0.0f, 0.0f), make_float2(0.0f, 0.0f)};
#pragma unroll
          for (int ch = 0; ch < 2; ++ch) {
            uint32_t p0[16], p1[16];
            umma::tmem_ld16_issue(tlane + 16 * ch, p0);
            umma::tmem_ld16_issue(tlane + 64 + 16 * ch, p1);
            umma::tmem_wait_ld();
            umma::tmem_hold16(p0);
            umma::tmem_hold16(p1);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float4 q4 = sR[(4 * ch + j) * 256 + tid];
#pragma unroll
              for (int z = 0; z < 2; ++z) {
                const float2 rr = z ? make_float2(q4.z, q4.w) : make_float2(q4.x, q4.y);
                const int k = 4 * j + 2 * z;
                a0[z] = umma::f2_fma(make_float2(__uint_as_float(p0[k]), __uint_as_float(p0[k + 1])), rr, a0[z]);
                a1[z] = umma::f2_fma(make_float2(__uint_as_float(p1[k]), __uint_as_float(p1[k + 1])), rr, a1[z]);
              }
            }
          }
          xw[(2 * h) * kTile + t] = (a0[0].x + a0[0].y) + (a0[1].x + a0[1].y);
          xw[(2 * h + 1) * kTile + t] = (a1[0].x + a1[0].y) + (a1[1].x + a1[1].y);
          uint32_t p0[16], p1[16];
          umma::tmem_ld16_issue(tlane, p0);
          umma::tmem_ld16_issue(tlane + 64, p1);
          pair_sync(warp);
          float w0 = xw[t] + xw[2 * kTile + t];            // half 0 + half 1, same order in both
          float w1 = xw[kTile + t] + xw[3 * kTile + t];
          w0 = fmaxf(w0 * fm, 0.0f);
          w1 = fmaxf(w1 * fp, 0.0f);
          const float tot = w0 + w1;
          const bool bad = !(tot > 0.0f) || !isfinite(tot);
          const float pplus = bad ? 0.5f : w1 / tot;
          bool plus;
          if (a.spins_in) {
            plus = (cur[4 * c + (warp & 3)] >> (tid & 31)) & 1u;
          } else {
            const int64_t site = (int64_t)r * Lx + c;
            const uint32_t* xu = xs + ((site >> 1) & 1) * (4 * kTile) + (site & 1) * (2 * kTile) + t;
            plus = draw_plus_bits(pplus, (uint64_t)xu[0] | ((uint64_t)xu[kTile] << 32));
            const uint32_t m = __ballot_sync(0xffffffffu, plus);
            if (h == 0 && (tid & 31) == 0) cur[4 * c + warp] = m;
          }
          pend_tot = tot;
          pend_w = plus ? w1 : w0;
          // Lambda_{c+1} = f(s) U[s] times a power of two: any such factor leaves q's
          // arithmetic unchanged, so it is taken from w(s) = f(s) <U[s], R_{c+1}> (already
          // summed) rather than from max |U[s]|: <Lambda_{c+1}, R_{c+1}> lands in [1, 2)
          const float ws = pend_w;
          const float mult = (plus ? fp : fm) * ((ws > 0x1.0p-126f && ws < INFINITY) ? pow2f(-ilogb_f(ws)) : 1.0f);
#pragma unroll
          for (int ch = 0; ch < 2; ++ch) {
            umma::tmem_wait_ld();
            umma::tmem_hold16(p0);
            umma::tmem_hold16(p1);
            float2 v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q)
              v[q] = umma::f2_mul(make_float2(__uint_as_float(plus ? p1[2 * q] : p0[2 * q]),
                                              __uint_as_float(plus ? p1[2 * q + 1] : p0[2 * q + 1])),
                                  make_float2(mult, mult));
            if (ch == 0) {
              umma::tmem_ld16_issue(tlane + 16, p0);
              umma::tmem_ld16_issue(tlane + 80, p1);
            }
            store_split16(a_hi + 8 * ch, a_lo + 8 * ch, v);
          }
          umma::tmem_wait_st();
        }
        // the A operand in TMEM becomes visible to the next UMMA
        umma::fence_before_sync();
        __syncthreads();

        if (misc[1]) {
          abort = true;
          break;
        }
      }
      // end of row: log q, energy, spins; this row becomes the previous row
      if (!ctrl && !abort) {
        if (h == 0) {
          const bool bad = !(pend_tot > 0.0f) || !isfinite(pend_tot);
          prod *= bad ? 0.5f : pend_w / pend_tot;
          flag |= bad ? TNMC_FLAG_NUMERIC : 0;
        }
        if (h == 0) lq += log((double)prod) + (double)pexp * 0.69314718055994530942;
        const int wd = warp & 3, bit = tid & 31;
#pragma unroll 4
        for (int c = h; c < Lx; c += 2) {
          int64_t q = a.e.qh[(size_t)r * Lx + c];
          if (c > 0) {
            const int64_t j = a.e.qJh[(size_t)r * (Lx - 1) + c - 1];
            q += ((cur[4 * (c - 1) + wd] >> bit) & 1u) ? j : -j;
          }
          if (r > 0) {
            const int64_t j = a.e.qJv[(size_t)(r - 1) * Lx + c];
            q += ((prev[4 * c + wd] >> bit) & 1u) ? j : -j;
          }
          eacc -= ((cur[4 * c + wd] >> bit) & 1u) ? q : -q;
        }
        if (a.spins_out && !a.spins_in) {
          // warp (h, wd) writes samples 32 wd + 16 h .. + 15, 32 columns at a time
          for (int c = bit; c < Lx; c += 32) {
            const uint32_t m = cur[4 * c + wd] >> (16 * h);
            const int64_t b0 = tile * kTile + 32 * wd + 16 * h;
            int8_t* dst = a.spins_out + (size_t)b0 * n + (size_t)r * Lx + c;
            const int ns = (a.B - b0) < 16 ? (int)(a.B - b0) : 16;
            for (int q = 0; q < ns; ++q) dst[(size_t)q * n] = ((m >> q) & 1u) ? 1 : -1;
          }
        }
      }
      __syncthreads();
      for (int q = tid; q < 4 * Lx; q += kThreads) prev[q] = cur[q];
      __syncthreads();
    }
    // the halves' energies meet in the exchange buffer (int64 [128])
    int64_t* ex = reinterpret_cast<int64_t*>(xw);
    if (!ctrl && h == 1) ex[t] = eacc;
    __syncthreads();
    if (tid < kTile && active && !abort) {
      a.logq[b] = lq;   // flagged samples too: the log of the probability they were drawn with
      a.energy[b] = scalbn((double)(eacc + ex[t]), a.e.qexp);
      if (a.flags) a.flags[b] = flag;
      if (flag) set_status(a.e.status, TNMC_E_NUMERIC);
    }
    __syncthreads();
  }
  // teardown (after the last step, or after a wait gave up): let the copies still in
  // flight land and the last committed UMMA finish (bounded waits with the full limit),
  // then free TMEM.  The UMMA warp observes the tile barriers in order, and the producer warp refills a
  // stage only in the step after its UMMA was waited for: at most one phase of each is outstanding.
  if (lead) {
    // steps the UMMA warp committed (g counts finished steps; an aborted step committed too), and
    // tiles it saw land
    const int64_t committed = g + (abort ? 1 : 0);
    const int64_t tiles_seen = g + ((abort && misc[2]) ? 1 : 0);
    for (int64_t q = tiles_seen; q < cnt[0]; ++q)
      (void)umma::mbar_wait_parked(umma::smem_u32(&bars[q % kStages]), (uint32_t)((q / kStages) & 1), kPollLimit,
                                   kPollHintNs);
    if (committed > 0)
      (void)umma::mbar_wait_parked(umma::smem_u32(&bars[kStages]), (uint32_t)((committed - 1) & 1), kPollLimit,
                                   kPollHintNs);
  }
  umma::fence_before_sync();
  __syncthreads();
  umma::fence_after_sync();
  if (warp == 0) umma::tmem_dealloc(tmem, kTmemCols);
}

// Pre-swizzled BF16 operand tiles of every (r, c).  Left sweep: M itself (n = s*64 + b,
// k = a).  Right sweep: the field-combined tensor of each value u of the spin above,
//   Mt^(u)[a][b] = sum_s f_u(s) M[a][s][b],  f_u(s) = exp(beta Jv[r-1][c] u s)  (1 on row 0),
// formed in FP64 (n = u*64 + a, k = b), so that R_c = Mt^(u) R_{c+1} is one half of the
// UMMA output.  Both are zero outside the bond dimensions and stored as BF16 hi + lo.
__global__ void derive_tc_kernel(DeviceEnv e, __nv_bfloat16* TR, __nv_bfloat16* TL, size_t ntens) {
  const int P = e.P;
  const size_t per = (size_t)kN * kK;
  const size_t total = ntens * per;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
    const size_t tt = i / per;
    const int rem = (int)(i % per);
    const int nn = rem / kK, k = rem % kK;
    const int s = nn >> 6, x = nn & 63;
    const double* M = e.M64 + tt * (size_t)P * 2 * P;
    const double fmin = e.fe[2 * tt], fplus = e.fe[2 * tt + 1];   // exp(-beta Jv), exp(+beta Jv); 1 on row 0
    // right tile: u = s (0: spin above -1), a = x, b = k ; left tile: s, b = x, a = k
    double vr = 0.0;
    if (x < P && k < P) {
      const double m0 = M[((size_t)x * 2 + 0) * P + k], m1 = M[((size_t)x * 2 + 1) * P + k];
      vr = s ? (fmin * m0 + fplus * m1) : (fplus * m0 + fmin * m1);
    }
    const double vl = (x < P && k < P) ? M[((size_t)k * 2 + s) * P + x] : 0.0;
    // hi = bf16(v), lo = bf16(v - hi): the pair carries about 16 significant bits
    const size_t off = tt * 2 * per + umma::sw128_offset(nn, k) / 2;
    const __nv_bfloat16 rh = __double2bfloat16(vr), lh = __double2bfloat16(vl);
    TR[off] = rh;
    TR[off + per] = __double2bfloat16(vr - (double)__bfloat162float(rh));
    TL[off] = lh;
    TL[off + per] = __double2bfloat16(vl - (double)__bfloat162float(lh));
  }
}

}  // namespace
}  // namespace tnmc

size_t tnmc_tc_tile_bytes() { return tnmc::kStageBytes; }

tnmc_status tnmc_launch_derive_tc(tnmc_env* env, cudaStream_t stream) {
  using namespace tnmc;
  DeviceEnv& d = env->d;
  const size_t ntens = (size_t)d.Lx * d.Ly;
  derive_tc_kernel<<<2048, 256, 0, stream>>>(d, const_cast<__nv_bfloat16*>(d.R16), const_cast<__nv_bfloat16*>(d.L16),
                                             ntens);
  TNMC_CUDA_TRY(cudaGetLastError());
  return TNMC_OK;
}

tnmc_status tnmc_launch_sample_tc(const tnmc_env* env, int64_t B, uint64_t seed, uint64_t offset,
                                  const int8_t* spins_in, int8_t* spins_out, double* logq, double* energy,
                                  int32_t* flags, cudaStream_t stream) {
  using namespace tnmc;
  const DeviceEnv& d = env->d;
  if (d.P > kK) {
    tnmc_set_error("the tensor-core sampler supports chi <= 64");
    return TNMC_E_UNSUPPORTED;
  }
  int dev = 0, nsm = 0, max_optin = 0, smem_sm = 0;
  TNMC_CUDA_TRY(cudaGetDevice(&dev));
  TNMC_CUDA_TRY(cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev));
  TNMC_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  TNMC_CUDA_TRY(cudaDeviceGetAttribute(&max_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  if (d.Lx > kMaxCols) {
    tnmc_set_error("the tensor-core sampler supports rows of at most %d sites", kMaxCols);
    return TNMC_E_UNSUPPORTED;
  }
  size_t smem = 1024 + kStages * kStageBytes + kRBytes + (kStages + 1) * 8 + 24 +
                (size_t)16 * kTile * sizeof(float) + (size_t)4 * d.Lx * sizeof(uint32_t);
  // Staged unless that does not fit (more than 3122 columns) or costs the SM its second CTA (204 to
  // 509 columns).  Measured, chi 16, 6 rows, 65536 samples, staged / not: 96 columns 4.59 / 4.68 ms,
  // 256 columns 18.2 (one CTA) / 12.5 (two), 600 columns 42.9 / 44.5.
  const size_t row_bytes = (size_t)6 * d.Lx * sizeof(uint32_t);
  const bool staged = !d.strong && smem + row_bytes <= (size_t)max_optin &&
                      (2 * (smem + row_bytes + 1024) <= (size_t)smem_sm || 2 * (smem + 1024) > (size_t)smem_sm);
  if (staged) smem += row_bytes;
  if (smem > (size_t)max_optin) {
    tnmc_set_error("tensor-core sampler needs %zu bytes of shared memory (device allows %d)", smem, max_optin);
    return TNMC_E_UNSUPPORTED;
  }
  auto kern = staged ? sample_tc_kernel<false> : sample_tc_kernel<true>;
  TNMC_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  TNMC_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                     (int)cudaSharedmemCarveoutMaxShared));
  int per_sm = 0;
  TNMC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kThreads, smem));
  {
    // cross-check the occupancy query against the shared-memory budget of an SM
    int regs_sm = 0;
    TNMC_CUDA_TRY(cudaDeviceGetAttribute(&regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, dev));
    cudaFuncAttributes fa;
    TNMC_CUDA_TRY(cudaFuncGetAttributes(&fa, kern));
    const int by_smem = smem_sm / (int)(smem + 1024);
    const int by_regs = regs_sm / (((fa.numRegs + 7) & ~7) * kThreads);
    const int est = by_smem < by_regs ? by_smem : by_regs;
    if (est > per_sm) per_sm = est;
  }
  if (per_sm < 1) per_sm = 1;
  if (per_sm > 2) per_sm = 2;   // TMEM: 2 x 256 columns per SM
  const int64_t ntiles = (B + kTile - 1) / kTile;
  int64_t grid = (int64_t)nsm * per_sm;
  if (grid > ntiles) grid = ntiles;
  const size_t need = (size_t)grid * d.Lx * (kTile * kK * sizeof(float) + (staged ? 0 : 4 * sizeof(uint32_t)));
  tnmc_env* me = const_cast<tnmc_env*>(env);
  {
    const tnmc_status gs = grow_scratch(me, need, stream, "sampler");
    if (gs != TNMC_OK) return gs;
  }
  TcArgs a;
  a.e = d;
  a.TR = d.R16;
  a.TL = d.L16;
  a.fe = d.fe32;
  a.B = B;
  a.seed = seed;
  a.offset = offset;
  a.spins_in = spins_in;
  a.spins_out = spins_out;
  a.logq = logq;
  a.energy = energy;
  a.flags = flags;
  a.stack = static_cast<float4*>(me->scratch.ptr);
  a.poll_limit = kPollLimit;
  {
    // test hook: TNMC_DEBUG_POLL_LIMIT=<n> caps the polls of the in-loop waits (0: they
    // give up at once), so that the timeout path can be exercised without a stuck copy
    const char* pl = getenv("TNMC_DEBUG_POLL_LIMIT");
    if (pl && *pl) a.poll_limit = (uint32_t)strtoul(pl, nullptr, 10);
  }
  kern<<<(unsigned)grid, kThreads, smem, stream>>>(a);
  TNMC_CUDA_TRY(cudaGetLastError());
  return TNMC_OK;
}
