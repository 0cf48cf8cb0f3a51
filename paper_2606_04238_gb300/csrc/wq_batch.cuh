// wq_batch.cuh -- batched-decode dequant-GEMM (sm_103a): the gated MLP's
// matrix products for a few to 64 tokens.
//
// At these token counts the weights are still read once for little work each
// (Sec. 5's decode regime), so the packed codes go from HBM to the tensor
// cores without being expanded: a code isolated by one AND reads as the
// binary16 subnormal code * 4^c * 2^-24 (c its bit-position class, cancelled
// by the activation's scale), mma.sync m16n8k16 multiplies it exactly with
// binary16 activations and sums in fp32, and per quantization group
//   tot += s sx * (sum code x' - z * sum x')
// is the affine dequantization s (q - z).  The tcgen05 path has to write every
// dequantized weight to shared memory first, whatever the token count; here a
// fragment of 256 weights costs 4 ANDs and is used for all tokens.
//
// Work split: row blocks of 128 rows x 128-feature blocks are the units;
// gridDim.x CTAs (one an SM; OCC = 2 for some routed launches) take equal contiguous ranges of them (row block
// major), so every SM has the same work for any shape.  A unit is computed by
// RG warps of two row tiles each (gate/up: tile w of gate and tile w of up;
// down: two neighbouring tiles), so each activation fragment is used twice;
// WK such sets take the CTA's units in turn and their sums are added through
// shared memory.  A row block whose range spans CTAs is finished by the CTA
// whose part arrives last: it adds the fp32 parts in feature order
// (deterministic, no spin-waits).
//
// The codes are private to a warp: it keeps D units in flight in its own
// shared-memory ring with cp.async, issued before the wait on the previous
// launch.  That hides little between gate/up and down, whose CTAs do not fit on
// an SM together (registers and shared memory): a CTA starts once the SM's last
// one has left.  Beside an input launch, which leaves SMs free, the codes are
// under way before it ends.  The activation records are shared by a set's warps, which take
// turns at issuing their bulk copies LEAD rounds ahead, onto mbarriers
// (bounded waits).
//
// Measured (GB300, us a layer of an MLP stack at W2 g128, the swapped-operand
// tcgen05 launch or the GEMV chain before -> this): d 4096 / inter 14336 at 16,
// 24, 64 tokens 102.2 -> 39.1, 104.1 -> 47.6, 110.4 -> 88.8; d 2560 / inter 9728
// at 16, 32, 64 47.2 -> 25.8, 61.9 -> 35.0, 74.5 -> 51.8.  At 24 tokens of the d 4096
// shape a gate/up launch takes ~24 us, 15 of them in the main loop, which keeps
// the mma.sync pipe (8 cycles an instruction) ~62 % busy; the rest is the
// launch's start (~2 us), the exchange of split parts (~2 us) and the finish.
#pragma once

#include <algorithm>

#include "wq_batch.h"
#include "wq_ptx.cuh"

namespace wq {

// Device status word of this translation unit's kernels: 0 or WQ_ERR_TIMEOUT (-6).
static __device__ int g_batch_status = 0;

namespace {

constexpr int kBatchRows = 128;            // rows of a row block
constexpr int kHsStride = kBatchRows + 8;  // halves a token of the staged h
constexpr int kYsStride = kBatchRows + 4;  // floats a token of the staged y

template <int BITS, int NPROJ, int GROUP, int NT, int OCC = 1>
struct BatchCfg {
  static constexpr int BPK = BITS * 256;  // code bytes per (row tile, block)
  static constexpr int GPB = 128 / GROUP;
  // Few tokens leave a warp few independent MMAs (2 NT) between dependent
  // phases: 16 warps of at most 128 registers; the accumulators of more
  // tokens need 8 warps of up to 255.
  static constexpr int NWARP = NT <= 3 && OCC == 1 ? 16 : 8;
  static constexpr int MAXSMEM = OCC == 2 ? 115712 : 232448;
  static constexpr int RG = NPROJ == 2 ? 8 : 4;
  static constexpr int WK = NWARP / RG;
  // A group's scales and zero points applied two tokens an instruction: the
  // loop is short of issue slots (67 % used beside the MMAs).  us a layer, one
  // -> two tokens an instruction: d 4096 at 32 tokens 60.5 -> 57.4, with groups
  // of 32 at 64 tokens 111 -> 105; only 4-bit gate/up in groups of 128 at 56
  // tokens and more loses (d 2560 W4 at 64 tokens 51.1 with one token in gate/up
  // and two in down, 51.6 with one in both, 51.9 with two).
  static constexpr bool PAIRED = !(BITS == 4 && GPB == 1 && NT == 8 && NPROJ == 2);
  // mma.sync truncates its sums: a down launch of up to 16 tokens adds a group of
  // 128 from two chains of 4, as the GEMV kernels that small matrices take do (d
  // 5120 x 17408 at 4 tokens of mean 0.5: error 1.6e-6 of the result with one
  // chain of 8, 5.8e-7 with two, 7.5e-7 on the GEMV kernels; above 16 tokens the
  // tcgen05 launch that was faster before had 1.05e-5, one chain has 1.65e-6).
  static constexpr bool SPLIT = NPROJ == 1 && GROUP == 128 && NT <= 2;
  static constexpr int REC = NT * (2048 + 32 + 32 * GPB);
  static constexpr int SLOT = 2 * (BPK + GPB * 64);  // two tiles of a unit
  static constexpr int TF = BITS == 4 || OCC == 2 ? 0 : 8 * NT * (int)kTfragBytes;  // LoRA-A products (rank 64; routed: from L2)
  static constexpr int STG_SUM = (WK - 1) * RG * 2 * NT * 512;
  static constexpr int STG_OUT = NPROJ == 2 ? NT * 8 * kHsStride * 2 : NT * 8 * kYsStride * 4;
  static constexpr int STG = std::max(STG_SUM, STG_OUT);
  static constexpr int LIMIT = MAXSMEM - 256 - NT * 32 - TF - STG;
  static constexpr int RXR = LIMIT - 4 * WK * REC >= 5 * NWARP * SLOT ? 4 : 3;  // rounds of WK records in the ring
  static constexpr int RX = RXR * WK, LEAD = RXR - 2;
  static constexpr int D = std::min(64 / NWARP, (LIMIT - RX * REC) / (NWARP * SLOT));
  static_assert(D >= 2, "batched-decode rings do not fit");
  static constexpr int OFF_CODES = RX * REC;
  static constexpr int OFF_TF = OFF_CODES + NWARP * D * SLOT;
  static constexpr int OFF_RS = OFF_TF + TF;
  static constexpr int OFF_STG = OFF_RS + NT * 32;
  static constexpr int OFF_BAR = OFF_STG + STG;
  static constexpr int SMEM = OFF_BAR + (2 * RX + 1) * 8 + 16;
  static_assert(SMEM <= MAXSMEM, "batched-decode shared memory");
  static constexpr int SLOT_F4 = RG * 2 * NT * 32;  // float4s of a part
};

__device__ __forceinline__ float batch_exp2i(int k) { return __int_as_float((k + 127) << 23); }

// Exponent that puts a block's largest |x| (bit pattern mxb) in [2^14, 2^15).
__device__ __forceinline__ int batch_block_exponent(uint32_t mxb) {
  const int be = (int)(mxb >> 23);
  return mxb == 0u || be >= 255 ? 0 : max(-100, min(100, 141 - be));
}

// One token's 128-feature block into its panel record: lane L holds features
// 4L .. 4L + 3 (f).  wide: 4-bit classes (16^-c), else 2-bit (4^-c).
__device__ __forceinline__ void batch_panel_token(uint8_t *rec, int nt_total, int group, bool wide, int m, int lane,
                                                  const float (&f)[4]) {
  const uint32_t v = __float_as_uint(fmaxf(fmaxf(fabsf(f[0]), fabsf(f[1])), fmaxf(fabsf(f[2]), fabsf(f[3]))));
  const int e = batch_block_exponent(__reduce_max_sync(0xffffffffu, v));
  const int st = lane >> 2, hi = (lane >> 1) & 1;
  const float mul = batch_exp2i(e - (wide ? 4 * hi : 4 * (st & 1) + 2 * hi));
  // features 4L, 4L+1 are pair p = 2 (L % 4) of step st, the next two pair
  // p + 1; pair p sits in word p / 4 of lane 4 (m % 8) + p % 4
  const int p = 2 * (lane & 3);
  uint32_t *w = reinterpret_cast<uint32_t *>(rec + (size_t)((m >> 3) * 4 + (st >> 1)) * 512);
  const int at = (4 * (m & 7) + (p & 3)) * 4 + 2 * (st & 1) + (p >> 2);
  const __half2 h0 = __floats2half2_rn(f[0] * mul, f[1] * mul), h1 = __floats2half2_rn(f[2] * mul, f[3] * mul);
  w[at] = *reinterpret_cast<const uint32_t *>(&h0);
  w[at + 4] = *reinterpret_cast<const uint32_t *>(&h1);
  float *sx = reinterpret_cast<float *>(rec + (size_t)nt_total * 2048);
  float gs = (f[0] + f[1]) + (f[2] + f[3]);
  const int lpg = group >> 2;  // lanes of a group
  for (int o = 1; o < lpg; o <<= 1) gs += __shfl_xor_sync(0xffffffffu, gs, o);
  if (lane % lpg == 0) sx[(1 + lane / lpg) * nt_total * 8 + m] = gs * batch_exp2i(e - 24);
  if (lane == 0) sx[m] = batch_exp2i(24 - e);
}

__device__ __forceinline__ float batch_half(uint32_t bits16) {
  return __half2float(__ushort_as_half(static_cast<unsigned short>(bits16 & 0xffffu)));
}

template <int N>
__device__ __forceinline__ void cp_async_wait_group() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

template <int BITS, int NPROJ, int GROUP, int NT, bool ROUTED, int OCC>
__global__ void __launch_bounds__(BatchCfg<BITS, NPROJ, GROUP, NT, OCC>::NWARP * 32, OCC)
    batch_kernel(const __grid_constant__ BatchArgs a) {
  using C = BatchCfg<BITS, NPROJ, GROUP, NT, OCC>;
  constexpr int BPK = C::BPK, GPB = C::GPB, WK = C::WK, RG = C::RG, D = C::D, RX = C::RX, GS = GROUP / 16;
  constexpr int NTHREADS = C::NWARP * 32;
  extern __shared__ __align__(128) uint8_t smem[];
  uint64_t *full = reinterpret_cast<uint64_t *>(smem + C::OFF_BAR), *empty = full + RX, *aux = empty + RX;
  volatile int *abort_s = reinterpret_cast<volatile int *>(aux + 1), *last_s = abort_s + 1;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int U = (a.K + 127) / 128, RB = (a.N + kBatchRows - 1) / kBatchRows;
  // Routed: row block `tile` is block tile % RB of segment tile / RB's expert.
  // The route was written two launches back (the launch in between lets this
  // one start only after its own wait), so it may be read before the wait.
  const int T = ROUTED ? __ldcg(&a.route->n_segs) * RB : RB;
  auto seg_of = [&](int tile) { return __ldcg(&a.route->seg[tile / RB]); };
  // the CTAs that take units, 2 each at least (routed: the grid is sized for the most segments)
  const long long W = (long long)T * U, P = min((long long)gridDim.x, max(1LL, W / 2));
  const bool takes = blockIdx.x < P;
  const long long g0 = takes ? W * blockIdx.x / P : 0;
  const int n = takes ? (int)(W * (blockIdx.x + 1) / P - g0) : 0;  // units of this CTA
  const int tile0 = (int)(g0 / U), kb0 = (int)(g0 - (long long)tile0 * U);
  if (tid == 0) {
    for (int s = 0; s < RX; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], RG);
    }
    mbar_init(aux, 1);
    *abort_s = 0;
    fence_barrier_init();
  }
  __syncthreads();
  // bounded wait; after a timeout every later wait gives up at once
  auto wait = [&](uint64_t *bar, uint32_t parity) -> bool {
    if (mbar_try_wait(bar, parity)) return true;
    if (*abort_s) return false;
    if (mbar_wait(bar, parity)) return true;
    *abort_s = 1;
    atomicExch(&g_batch_status, -6);
    return false;
  };

  const int rg = warp % RG, wk = warp / RG, g = lane >> 2, t = lane & 3;
  const int RT = (a.N + 15) / 16;
  // ---- codes and scales/zeros of this warp's units, pi = wk, wk + WK, .. of
  // row block ptile, block pkb, into its ring.  A lane copies the same 16-byte
  // chunks of every unit: the pointers move on by WK blocks, and are set again
  // at a row block's first unit. ----
  constexpr int CPT = BPK / 16, MPT = 4 * GPB, NQ = 2 * CPT / 32;  // chunks of a tile's codes, scales/zeros; a lane's
  uint8_t *ring = smem + C::OFF_CODES + warp * (D * C::SLOT);
  const uint8_t *csrc[NQ], *msrc;
  bool cin[NQ], min_;
  int pi = wk, pslot = 0, ptile = tile0, pkb = kb0 + wk;
  auto aim = [&]() {
    while (pkb >= U) pkb -= U, ++ptile;
    const int rb8 = (ROUTED ? ptile % RB : ptile) * 8;
    const size_t rte = ROUTED && pi < n ? (size_t)seg_of(ptile).x * RT : 0;  // the expert's first row tile
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const int c = lane + 32 * q, tl = c / CPT, off = c - tl * CPT;
      const int rt = rb8 + (NPROJ == 2 ? rg : 2 * rg + tl);
      cin[q] = rt < RT;
      csrc[q] = reinterpret_cast<const uint8_t *>(NPROJ == 2 && tl ? a.codes[1] : a.codes[0]) +
                (cin[q] ? ((rte + rt) * U + pkb) * BPK + off * 16 : 0);
    }
    const int tl = lane / MPT, off = lane - tl * MPT;
    const int rt = rb8 + (NPROJ == 2 ? rg : 2 * rg + tl);
    min_ = lane < 2 * MPT && rt < RT;
    msrc = reinterpret_cast<const uint8_t *>(NPROJ == 2 && tl ? a.meta[1] : a.meta[0]) +
           (min_ ? ((rte + rt) * U + pkb) * (GPB * 64) + off * 16 : 0);
  };
  aim();
  auto issue = [&]() {
    if (pi < n) {
      uint8_t *dst = ring + pslot * C::SLOT + lane * 16;
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        cp_async16_zfill(dst + q * 512, csrc[q], cin[q] ? 16u : 0u);
        if (cin[q]) csrc[q] += WK * BPK;
      }
      if (lane < 2 * MPT) {
        cp_async16_zfill(dst + 2 * BPK, msrc, min_ ? 16u : 0u);
        if (min_) msrc += WK * GPB * 64;
      }
    }
    cp_async_commit();
    pi += WK;
    if (++pslot == D) pslot = 0;
    pkb += WK;
    if (pkb >= U && pi < n) aim();
  };
  // ---- the set's activation records: the j-th of the set goes to stage
  // j % RXR; warp j % RG of the set issues its copy LEAD rounds ahead, once
  // the stage's previous record is read (by units of two rounds before) ----
  constexpr int RXR = C::RXR, LEAD = C::LEAD;
  uint64_t *sfull = full + wk * RXR, *sempty = empty + wk * RXR;
  uint8_t *xring = smem + wk * RXR * C::REC;
  const int nset = (n - wk + WK - 1) / WK;  // units of this set (n >= wk or 0)
  // (The bookkeeping is the producing warp's alone, every RG rounds: done by
  // every warp each round it took 3 % of a d 4096 layer at 24 tokens.)
  int issued = -1;                          // the last record this warp copied
  int rj = rg, rleft = rg - LEAD;           // the next record it copies, and the rounds until then
  auto produce = [&]() {
    if (rj < nset && elect_one()) {
      const int at = kb0 + wk + rj * WK, rtile = tile0 + at / U, rkb = at % U;
      const uint8_t *panel = a.panel + (ROUTED ? (size_t)(rtile / RB) * U * C::REC : 0);
      const int rst = rj % RXR;
      if (rj < RXR || wait(&sempty[rst], (rj / RXR - 1) & 1)) {
        mbar_arrive_expect_tx(&sfull[rst], (uint32_t)C::REC);
        bulk_g2s(xring + rst * C::REC, panel + (size_t)rkb * C::REC, (uint32_t)C::REC, &sfull[rst]);
        issued = rj;
      }
    }
    rj += RG;
    rleft += RG;
  };
#pragma unroll 1
  for (int j = 0; j < D; ++j) issue();
  pdl_wait();
  pdl_launch_dependents();
  if (rg < LEAD) produce();
  if (NPROJ == 2 && !ROUTED && warp == LEAD && elect_one()) {
    const uint32_t tfb = BITS != 4 && a.tfrag != nullptr ? 2u * ((a.r + 15) / 16) * NT * kTfragBytes : 0u;
    const uint32_t rsb = a.rs != nullptr ? NT * 32u : 0u;
    mbar_arrive_expect_tx(aux, tfb + rsb);
    if (tfb) bulk_g2s(smem + C::OFF_TF, a.tfrag, tfb, aux);
    if (rsb) bulk_g2s(smem + C::OFF_RS, a.rs, rsb, aux);
  }
  __syncwarp();

  float tot[2][NT][4];
  int i = wk, cslot = 0, st = 0, ph = 0;  // this warp's next unit, its code slot, record stage and phase
  for (int i0 = 0, tile = tile0, ub = kb0; i0 < n;) {
    const int len = min(U - ub, n - i0);
    if (NPROJ == 2 && a.tfrag != nullptr && wk == 0 && lane < a.r / 4) {
      // this part's LoRA-B rows towards L2
      const size_t row0 = (ROUTED ? tile % RB : tile) * kBatchRows + rg * 16;
      const size_t off = ((ROUTED ? (size_t)seg_of(tile).x * a.N : 0) + row0) * a.r * 2 + lane * 128;
      if (row0 * a.r * 2 + lane * 128 < (size_t)a.N * a.r * 2) {
        asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const uint8_t *>(a.lora_b[0]) + off));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const uint8_t *>(a.lora_b[1]) + off));
      }
    }
#pragma unroll
    for (int tl = 0; tl < 2; ++tl)
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int q = 0; q < 4; ++q) tot[tl][nt][q] = 0.f;
    for (; i < i0 + len; i += WK) {
      if (--rleft < 0) {
        produce();
        __syncwarp();
      }
      cp_async_wait_group<D - 1>();
      __syncwarp();
      if (wait(&sfull[st], ph)) {
        const uint8_t *X = xring + st * C::REC + lane * 16;
        const float *sxp = reinterpret_cast<const float *>(xring + st * C::REC + NT * 2048) + 2 * t;
        const uint8_t *cw = ring + cslot * C::SLOT;
        constexpr int NW = BITS == 2 ? 4 : BITS == 3 ? 6 : 8;
        uint32_t wd[2][NW];
#pragma unroll
        for (int tl = 0; tl < 2; ++tl) {
          const uint4 w0 = lds128(cw + tl * BPK + lane * 16);
          wd[tl][0] = w0.x; wd[tl][1] = w0.y; wd[tl][2] = w0.z; wd[tl][3] = w0.w;
          if (BITS == 3) {
            const uint2 w1 = lds64(cw + tl * BPK + 512 + lane * 8);
            wd[tl][4] = w1.x; wd[tl][5] = w1.y;
          }
          if (BITS == 4) {
            const uint4 w1 = lds128(cw + tl * BPK + 512 + lane * 16);
            wd[tl][NW - 4] = w1.x; wd[tl][NW - 3] = w1.y; wd[tl][NW - 2] = w1.z; wd[tl][NW - 1] = w1.w;
          }
        }
        float acc[2][NT][4], acc2[2][NT][4];  // acc2: C::SPLIT's second half of the block
#pragma unroll
        for (int kp = 0; kp < 4; ++kp) {
          uint4 b[NT];
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) b[nt] = lds128(X + (nt * 4 + kp) * 512);
#pragma unroll
          for (int hf = 0; hf < 2; ++hf) {
            const int ks = 2 * kp + hf;
            uint32_t af[2][4];
#pragma unroll
            for (int tl = 0; tl < 2; ++tl) {
              if (BITS == 4) {
                const uint32_t x = wd[tl][ks & (NW - 1)], x8 = x >> 8;
                af[tl][0] = x & 0x000F000Fu;
                af[tl][1] = x8 & 0x000F000Fu;
                af[tl][2] = x & 0x00F000F0u;
                af[tl][3] = x8 & 0x00F000F0u;
              } else {
                const uint32_t x = wd[tl][kp], x8 = x >> 8;
                const int s4 = hf * 4;
                af[tl][0] = x & (0x00030003u << s4);
                af[tl][1] = x8 & (0x00030003u << s4);
                af[tl][2] = x & (0x000C000Cu << s4);
                af[tl][3] = x8 & (0x000C000Cu << s4);
                if (BITS == 3) {  // the high bit of each code from the second plane
                  const uint32_t hw = wd[tl][(NW - 2) + (kp >> 1)];
                  const uint32_t h0 = (kp & 1) ? hw >> 6 : hw << 2, h1 = (kp & 1) ? hw >> 7 : hw << 1;
                  af[tl][0] |= h0 & (0x00040004u << s4);
                  af[tl][1] |= h1 & (0x00040004u << s4);
                  af[tl][2] |= h0 & (0x00100010u << s4);
                  af[tl][3] |= h1 & (0x00100010u << s4);
                }
              }
            }
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
              for (int tl = 0; tl < 2; ++tl) {
                const uint32_t b0 = hf ? b[nt].z : b[nt].x, b1 = hf ? b[nt].w : b[nt].y;
                float(&c)[4] = C::SPLIT && ks >= 4 ? acc2[tl][nt] : acc[tl][nt];
                if (ks % (C::SPLIT ? 4 : GS) == 0)
                  mma_f16_16816_zc(c, af[tl], b0, b1);
                else
                  mma_f16_16816(c, af[tl], b0, b1);
              }
            if ((ks + 1) % GS == 0) {
              // the group's share, tot += s sx (sum q x' - z sum x'): the difference
              // first, rounded once (sx is a power of two).  Added to tot one by one the
              // two terms round at their own size, which for activations of one sign is
              // many times the difference's.
              const int gl = ks / GS;
              float sl[2], sh[2], zl[2], zh[2];
#pragma unroll
              for (int tl = 0; tl < 2; ++tl) {
                const uint2 sz = lds64(cw + 2 * BPK + (tl * GPB + gl) * 64 + g * 8);
                sl[tl] = batch_half(sz.x);
                sh[tl] = batch_half(sz.x >> 16);
                zl[tl] = -batch_half(sz.y);
                zh[tl] = -batch_half(sz.y >> 16);
              }
#pragma unroll
              for (int nt = 0; nt < NT; ++nt) {
                const float2 sx = *reinterpret_cast<const float2 *>(sxp + nt * 8);
                const float2 xs = *reinterpret_cast<const float2 *>(sxp + (1 + gl) * NT * 8 + nt * 8);
#pragma unroll
                for (int tl = 0; tl < 2; ++tl) {
                  float *c = tot[tl][nt];
                  float *q = acc[tl][nt];
                  if (C::SPLIT)
#pragma unroll
                    for (int e = 0; e < 4; ++e) q[e] += acc2[tl][nt][e];
                  if (C::PAIRED) {  // the same operations and roundings
                    const uint64_t sx2 = pack_f32x2(sx.x, sx.y), xs2 = pack_f32x2(xs.x, xs.y);
                    const uint64_t dl = fma_f32x2(pack_f32x2(zl[tl], zl[tl]), xs2, pack_f32x2(q[0], q[1]));
                    const uint64_t dh = fma_f32x2(pack_f32x2(zh[tl], zh[tl]), xs2, pack_f32x2(q[2], q[3]));
                    unpack_f32x2(fma_f32x2(mul_f32x2(pack_f32x2(sl[tl], sl[tl]), sx2), dl, pack_f32x2(c[0], c[1])), c[0], c[1]);
                    unpack_f32x2(fma_f32x2(mul_f32x2(pack_f32x2(sh[tl], sh[tl]), sx2), dh, pack_f32x2(c[2], c[3])), c[2], c[3]);
                  } else {
                    c[0] = fmaf(sl[tl] * sx.x, fmaf(zl[tl], xs.x, q[0]), c[0]);
                    c[1] = fmaf(sl[tl] * sx.y, fmaf(zl[tl], xs.y, q[1]), c[1]);
                    c[2] = fmaf(sh[tl] * sx.x, fmaf(zh[tl], xs.x, q[2]), c[2]);
                    c[3] = fmaf(sh[tl] * sx.y, fmaf(zh[tl], xs.y, q[3]), c[3]);
                  }
                }
              }
            }
          }
        }
      }
      __syncwarp();  // every lane has read the slot and the record
      if (lane == 0) mbar_arrive(&sempty[st]);
      issue();
      if (++cslot == D) cslot = 0;
      if (++st == RXR) st = 0, ph ^= 1;
    }

    // ---- the part of row block `tile` is complete ----
    const bool first = i0 == 0, whole = ub == 0 && len == U;
    i0 += len;
    ub = 0;
    ++tile;
    if (WK > 1) {
      // the other sets' sums join the first set's
      float4 *stg = reinterpret_cast<float4 *>(smem + C::OFF_STG) + lane;
      named_barrier_sync(1, NTHREADS);  // the previous part's staging is read
      if (wk > 0)
#pragma unroll
        for (int tl = 0; tl < 2; ++tl)
#pragma unroll
          for (int nt = 0; nt < NT; ++nt)
            stg[(((wk - 1) * RG + rg) * 2 * NT + tl * NT + nt) * 32] =
                make_float4(tot[tl][nt][0], tot[tl][nt][1], tot[tl][nt][2], tot[tl][nt][3]);
      named_barrier_sync(1, NTHREADS);
      if (wk > 0) continue;
      for (int w = 0; w < WK - 1; ++w)
#pragma unroll
        for (int tl = 0; tl < 2; ++tl)
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) {
            const float4 v = stg[((w * RG + rg) * 2 * NT + tl * NT + nt) * 32];
            tot[tl][nt][0] += v.x; tot[tl][nt][1] += v.y; tot[tl][nt][2] += v.z; tot[tl][nt][3] += v.w;
          }
    }
    // from here the first set's warps alone (wk == 0)
    if (!whole) {
      // a split row block's part: the CTA's slot 0 (its first part) or 1 (its last)
      float4 *mine = reinterpret_cast<float4 *>(a.part) + ((size_t)blockIdx.x * 2 + (first ? 0 : 1)) * C::SLOT_F4 +
                     (size_t)rg * (2 * NT * 32) + lane;
#pragma unroll
      for (int tl = 0; tl < 2; ++tl)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
          __stcg(mine + (tl * NT + nt) * 32, make_float4(tot[tl][nt][0], tot[tl][nt][1], tot[tl][nt][2], tot[tl][nt][3]));
      const long long tu = (long long)(tile - 1) * U;
      const int c_lo = (int)(((tu + 1) * P + W - 1) / W - 1), c_hi = (int)(((tu + U) * P + W - 1) / W - 1);
      named_barrier_sync(2, RG * 32);
      if (tid == 0) {
        int last = 0;
        __threadfence();  // after the barrier: covers the writes of all the set's threads
        if (!*abort_s) {
          last = atomicAdd(&a.cnt[tile - 1], 1u) == (unsigned)(c_hi - c_lo) ? 1 : 0;
          if (last) a.cnt[tile - 1] = 0;  // ready for the next launch
        }
        *last_s = last;
        __threadfence();
      }
      named_barrier_sync(2, RG * 32);
      if (!*last_s) continue;
#pragma unroll
      for (int tl = 0; tl < 2; ++tl)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
          for (int q = 0; q < 4; ++q) tot[tl][nt][q] = 0.f;
#pragma unroll(NT <= 4 ? 2 : 1)
      for (int cc = c_lo; cc <= c_hi; ++cc) {  // the parts in feature order
        // CTA cc's part of this row block is its first unless the block began inside its range
        const float4 *src = reinterpret_cast<const float4 *>(a.part) +
                            ((size_t)cc * 2 + (tu <= W * cc / P ? 0 : 1)) * C::SLOT_F4 + (size_t)rg * (2 * NT * 32) + lane;
        float4 v[2][NT];
#pragma unroll
        for (int tl = 0; tl < 2; ++tl)
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) v[tl][nt] = __ldcg(src + (tl * NT + nt) * 32);
#pragma unroll
        for (int tl = 0; tl < 2; ++tl)
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) {
            tot[tl][nt][0] += v[tl][nt].x; tot[tl][nt][1] += v[tl][nt].y;
            tot[tl][nt][2] += v[tl][nt].z; tot[tl][nt][3] += v[tl][nt].w;
          }
      }
    }
    const int seg = ROUTED ? (tile - 1) / RB : 0, rblk = tile - 1 - seg * RB, n0 = rblk * kBatchRows;
    const int4 sg = ROUTED ? seg_of(tile - 1) : make_int4(0, a.M, 0, 0);
    const int M = sg.y;
    // output row of token m
    auto orow = [&](int m) -> size_t { return ROUTED ? (size_t)__ldcg(&a.route->list[sg.z + m]) : (size_t)m; };
    if (NPROJ == 2) {
      if (!ROUTED) wait(aux, 0);
      // Eq. 1's unmerged adapter: tot += B t, t as three bf16 parts (all 24 bits),
      // the smallest first, summed on their own before they join the total
      if (BITS != 4 && a.tfrag != nullptr) {
        const int RK = (a.r + 15) / 16;
        auto load_b = [&](int p, int kk, uint32_t (&bf)[4]) {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int row = n0 + rg * 16 + g + 8 * (q & 1), col = kk * 16 + 2 * t + 8 * (q >> 1);
            const size_t at = (ROUTED ? (size_t)sg.x * a.N + row : (size_t)row) * a.r + col;
            bf[q] = row < a.N && col < a.r
                        ? __ldg(reinterpret_cast<const uint32_t *>(reinterpret_cast<const uint8_t *>(a.lora_b[p]) + at * 2))
                        : 0u;
          }
        };
        // the fragments of a rank step: from shared memory, or (routed) from L2 a step ahead
        auto load_t = [&](int p, int kk, uint4 (&tv)[NT], uint2 (&tl)[NT]) {
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) {
            const uint32_t at = ((p * RK + kk) * NT + nt) * kTfragBytes;
            if (ROUTED) {
              const uint8_t *src = a.tfrag + (size_t)seg * (2 * RK * NT * kTfragBytes) + at;
              tv[nt] = __ldcg(reinterpret_cast<const uint4 *>(src) + lane);
              tl[nt] = __ldcg(reinterpret_cast<const uint2 *>(src + 512) + lane);
            } else {
              tv[nt] = lds128(smem + C::OFF_TF + at + lane * 16);
              tl[nt] = lds64(smem + C::OFF_TF + at + 512 + lane * 8);
            }
          }
        };
        // PP projections at a time: both where their registers allow (d 4096 in
        // groups of 32 at 5 tokens 38.4 -> 38.1 us a layer against one at a time; two
        // parts of t in place of three took 37.9)
        constexpr int PP = NT <= (ROUTED ? 1 : 2) ? 2 : 1;
        uint32_t bf[PP][4], bn[PP][4] = {};
        uint4 tv[PP][NT], tvn[PP][NT] = {};
        uint2 tl[PP][NT], tln[PP][NT] = {};
#pragma unroll
        for (int q = 0; q < PP; ++q) {
          load_b(q, 0, bf[q]);
          if (ROUTED) load_t(q, 0, tv[q], tl[q]);
        }
#pragma unroll
        for (int p0 = 0; p0 < 2; p0 += PP) {
          float ad[PP][NT][4] = {};
#pragma unroll 1
          for (int kk = 0; kk < RK; ++kk) {
            const bool same = kk + 1 < RK;
            if (same || p0 + PP < 2) {
#pragma unroll
              for (int q = 0; q < PP; ++q) {
                load_b(same ? p0 + q : 1, same ? kk + 1 : 0, bn[q]);
                if (ROUTED) load_t(same ? p0 + q : 1, same ? kk + 1 : 0, tvn[q], tln[q]);
              }
            }
#pragma unroll
            for (int q = 0; q < PP; ++q)
              if (!ROUTED) load_t(p0 + q, kk, tv[q], tl[q]);
#pragma unroll
            for (int part = 2; part >= 0; --part)
#pragma unroll
              for (int q = 0; q < PP; ++q)
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) {
                  const uint4 v = tv[q][nt];
                  const uint2 w = part == 2 ? tl[q][nt] : part == 1 ? make_uint2(v.z, v.w) : make_uint2(v.x, v.y);
                  mma_bf16_16816(ad[q][nt], bf[q], w.x, w.y);
                }
#pragma unroll
            for (int q = 0; q < PP; ++q) {
#pragma unroll
              for (int e = 0; e < 4; ++e) bf[q][e] = bn[q][e];
#pragma unroll
              for (int nt = 0; nt < NT; ++nt)
                if (ROUTED) tv[q][nt] = tvn[q][nt], tl[q][nt] = tln[q][nt];
            }
          }
#pragma unroll
          for (int q = 0; q < PP; ++q)
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
              for (int e = 0; e < 4; ++e) tot[p0 + q][nt][e] += ad[q][nt][e];
        }
      }
      // h = SiLU(rs g) rs u, staged as bf16 [token][128 rows]
      __nv_bfloat16 *hs = reinterpret_cast<__nv_bfloat16 *>(smem + C::OFF_STG);
      const float *rs_s = reinterpret_cast<const float *>(smem + C::OFF_RS);
      named_barrier_sync(2, RG * 32);  // the staged sums are read
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int m = nt * 8 + 2 * t + e;
          const float rs = a.rs == nullptr || m >= M ? 1.f : ROUTED ? __ldcg(a.rs + seg * NT * 8 + m) : rs_s[m];
#pragma unroll
          for (int rr = 0; rr < 2; ++rr) {
            const float gv = rs * tot[0][nt][2 * rr + e], uv = rs * tot[1][nt][2 * rr + e];
            hs[m * kHsStride + rg * 16 + g + 8 * rr] = __float2bfloat16_rn(gv / (1.f + __expf(-gv)) * uv);
          }
        }
      named_barrier_sync(2, RG * 32);
      const int nb = n0 + 4 * lane;
      for (int m = rg; m < NT * 8; m += RG) {
        const uint2 raw = lds64(hs + m * kHsStride + 4 * lane);
        if (a.out != nullptr && m < M && nb < a.N) {
          __nv_bfloat16 *o = reinterpret_cast<__nv_bfloat16 *>(a.out) + orow(m) * a.N + nb;
          if ((a.N & 3) == 0) {
            *reinterpret_cast<uint2 *>(o) = raw;
          } else {
            for (int e = 0; e < 4 && nb + e < a.N; ++e)
              o[e] = __ushort_as_bfloat16((unsigned short)((e < 2 ? raw.x : raw.y) >> (16 * (e & 1))));
          }
        }
        if (a.panel_out != nullptr) {
          const float f[4] = {__uint_as_float(raw.x << 16), __uint_as_float(raw.x & 0xffff0000u),
                              __uint_as_float(raw.y << 16), __uint_as_float(raw.y & 0xffff0000u)};
          batch_panel_token(a.panel_out + (size_t)(tile - 1) * batch_rec_bytes(NT, a.group_out), NT, a.group_out, true, m,
                            lane, f);  // routed: RB records a segment
        }
      }
    } else {
      // y = sums + residual, staged as fp32 [token][128 rows]: 4 rows a lane
      float *ys = reinterpret_cast<float *>(smem + C::OFF_STG);
      named_barrier_sync(2, RG * 32);  // the staged sums are read
#pragma unroll
      for (int tl = 0; tl < 2; ++tl)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
          for (int q = 0; q < 4; ++q)
            ys[(nt * 8 + 2 * t + (q & 1)) * kYsStride + rg * 32 + tl * 16 + g + 8 * (q >> 1)] = tot[tl][nt][q];
      named_barrier_sync(2, RG * 32);
      const int nb = n0 + 4 * lane;
      const bool vec = (a.N & 3) == 0;
      constexpr int MU = 4;  // tokens of a warp in flight
      for (int mb = rg; mb < M; mb += RG * MU) {
        uint2 res[MU];
#pragma unroll
        for (int q = 0; q < MU; ++q) {
          const int m = mb + q * RG;
          res[q] = make_uint2(0u, 0u);
          if (a.residual != nullptr && vec && m < M && nb < a.N)
            res[q] = __ldcg(reinterpret_cast<const uint2 *>(reinterpret_cast<const __nv_bfloat16 *>(a.residual) +
                                                            (size_t)m * a.N + nb));
        }
#pragma unroll
        for (int q = 0; q < MU; ++q) {
          const int m = mb + q * RG;
          if (m >= M || nb >= a.N) continue;
          const float4 v4 = *reinterpret_cast<const float4 *>(ys + m * kYsStride + 4 * lane);
          float v[4] = {v4.x, v4.y, v4.z, v4.w};
          const size_t o = orow(m) * a.N + nb;
          if (vec) {
            v[0] += __uint_as_float(res[q].x << 16);
            v[1] += __uint_as_float(res[q].x & 0xffff0000u);
            v[2] += __uint_as_float(res[q].y << 16);
            v[3] += __uint_as_float(res[q].y & 0xffff0000u);
            if (a.out_f32) {
              *reinterpret_cast<float4 *>(reinterpret_cast<float *>(a.out) + o) = make_float4(v[0], v[1], v[2], v[3]);
            } else {
              const __nv_bfloat162 lo = __floats2bfloat162_rn(v[0], v[1]), hi = __floats2bfloat162_rn(v[2], v[3]);
              *reinterpret_cast<uint2 *>(reinterpret_cast<__nv_bfloat16 *>(a.out) + o) =
                  make_uint2(*reinterpret_cast<const uint32_t *>(&lo), *reinterpret_cast<const uint32_t *>(&hi));
            }
          } else {
            for (int e = 0; e < 4 && nb + e < a.N; ++e) {
              float y = v[e];
              if (a.residual) y += __bfloat162float(__ldcg(reinterpret_cast<const __nv_bfloat16 *>(a.residual) + o + e));
              if (a.out_f32)
                reinterpret_cast<float *>(a.out)[o + e] = y;
              else
                reinterpret_cast<__nv_bfloat16 *>(a.out)[o + e] = __float2bfloat16_rn(y);
            }
          }
        }
      }
    }
  }
  cp_async_wait_all();
  __syncwarp();
  // the records were waited for where they are used, unless a timeout came before
  if (*abort_s && elect_one() && issued >= 0) mbar_wait(&sfull[issued % RXR], (issued / RXR) & 1);
  // no CTA ends with a copy into its shared memory in flight: one whose parts are
  // all finished by others has not waited for the LoRA-A products and scales
  if (NPROJ == 2 && !ROUTED && tid == 0 && !mbar_wait(aux, 0)) atomicExch(&g_batch_status, -6);
}

template <int BITS, int NPROJ, int GROUP, int NT, bool ROUTED = false, int OCC = 1>
cudaError_t launch_batch_t(const BatchArgs &a, int ctas, cudaStream_t s) {
  using C = BatchCfg<BITS, NPROJ, GROUP, NT, OCC>;
  auto kern = batch_kernel<BITS, NPROJ, GROUP, NT, ROUTED, OCC>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ctas);
  cfg.blockDim = dim3(C::NWARP * 32);
  cfg.dynamicSmemBytes = C::SMEM;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a);
}

template <int BITS, int NPROJ, int GROUP>
cudaError_t launch_batch_n(const BatchArgs &a, int nt, int ctas, cudaStream_t s) {
  switch (nt) {
    case 1: return launch_batch_t<BITS, NPROJ, GROUP, 1>(a, ctas, s);
    case 2: return launch_batch_t<BITS, NPROJ, GROUP, 2>(a, ctas, s);
    case 3: return launch_batch_t<BITS, NPROJ, GROUP, 3>(a, ctas, s);
    case 4: return launch_batch_t<BITS, NPROJ, GROUP, 4>(a, ctas, s);
    case 6: return launch_batch_t<BITS, NPROJ, GROUP, 6>(a, ctas, s);
    case 8: return launch_batch_t<BITS, NPROJ, GROUP, 8>(a, ctas, s);
    default: return cudaErrorInvalidValue;
  }
}

template <int BITS, int NPROJ>
cudaError_t launch_batch_g(const BatchArgs &a, int nt, int ctas, cudaStream_t s) {
  switch (a.group) {
    case 32: return launch_batch_n<BITS, NPROJ, 32>(a, nt, ctas, s);
    case 64: return launch_batch_n<BITS, NPROJ, 64>(a, nt, ctas, s);
    case 128: return launch_batch_n<BITS, NPROJ, 128>(a, nt, ctas, s);
    default: return cudaErrorInvalidValue;
  }
}

template <int BITS, int NPROJ, int GROUP>
cudaError_t launch_batch_routed_n(const BatchArgs &a, int nt, int ctas, int occ, cudaStream_t s) {
  if (occ == 2) {
    if (nt == 1) return launch_batch_t<BITS, NPROJ, GROUP, 1, true, 2>(a, ctas, s);
    if (nt == 2) return launch_batch_t<BITS, NPROJ, GROUP, 2, true, 2>(a, ctas, s);
    return cudaErrorInvalidValue;
  }
  switch (nt) {
    case 1: return launch_batch_t<BITS, NPROJ, GROUP, 1, true>(a, ctas, s);
    case 2: return launch_batch_t<BITS, NPROJ, GROUP, 2, true>(a, ctas, s);
    case 4: return launch_batch_t<BITS, NPROJ, GROUP, 4, true>(a, ctas, s);
    default: return cudaErrorInvalidValue;
  }
}

template <int BITS, int NPROJ>
cudaError_t launch_batch_routed_g(const BatchArgs &a, int nt, int ctas, int occ, cudaStream_t s) {
  switch (a.group) {
    case 32: return launch_batch_routed_n<BITS, NPROJ, 32>(a, nt, ctas, occ, s);
    case 64: return launch_batch_routed_n<BITS, NPROJ, 64>(a, nt, ctas, occ, s);
    case 128: return launch_batch_routed_n<BITS, NPROJ, 128>(a, nt, ctas, occ, s);
    default: return cudaErrorInvalidValue;
  }
}

inline cudaError_t read_batch_status_tu(int *status) {
  int v = 0;
  cudaError_t e = cudaMemcpyFromSymbol(&v, g_batch_status, sizeof(int));
  if (e != cudaSuccess) return e;
  const int zero = 0;
  e = cudaMemcpyToSymbol(g_batch_status, &zero, sizeof(int));
  *status = v;
  return e;
}

}  // namespace
}  // namespace wq
