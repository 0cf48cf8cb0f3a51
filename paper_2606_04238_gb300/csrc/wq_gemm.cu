// wq_gemm.cu -- batched (prefill-size) dequant-GEMM on the 5th-generation
// tensor cores (tcgen05, accumulators in tensor memory), sm_103a.
//
// For a token batch of more than a few dozen tokens the gated MLP of the
// W4/W2-GateUp scheme (Sec. 3.3) is a real dense contraction, so the packed
// weights are dequantized to binary16 tiles in shared memory and fed to
// tcgen05.mma with fp32 accumulation in TMEM:
//   * gate/up: D_g = x deq(Wg)^T + (lora_scale x A_g^T) B_g^T, D_u likewise
//     (the unmerged LoRA path of Eq. 1 enters as two more k-steps), then
//     h = SiLU(rs D_g) * (rs D_u) with rs the RMSNorm scale of the token;
//   * down: y = residual + h deq(Wd)^T.
// A CTA computes a tile of 128 or 256 tokens x 128 output rows (x 2
// projections for gate/up; down may take 256 rows) over the whole feature axis, 64 features (half a
// block of the packed format) per pipeline stage; with 256 tokens the two
// halves of 128 multiply the same dequantized B tile into accumulators of
// their own, so each weight is dequantized once per 256 tokens.  Warp roles:
//   warps 0..15 dequantize, in two groups of 8 that take alternate stages (a
//               group's hand-overs and load latencies then have two stages):
//               code q of row n, group j gives
//               the binary16 value s_nj (q - z_nj), rounded once; they write
//               it in the tcgen05 K-major layout (8-row x 16-byte core
//               matrices), then run the epilogue from TMEM;
//   warp 16     loads the binary16 activation tile with the tensor-memory
//               accelerator (TMA; one box of 64 features x 128 tokens in the
//               128-byte swizzled layout, zero fill outside the matrix);
//   warp 17     owns the TMEM allocation; one elected lane issues the MMAs.
//               The lane is chosen by elect.sync: behind `lane == 0` each
//               tcgen05.mma took ~100 ns to issue whatever its N, longer than
//               the 62 ns the tensor pipe needs for one of 128 x 256 x 16, so
//               the issuing thread bounded the main loop (a layer of d 5120,
//               inter 17408 at 512 tokens: 327 us, with elect.sync 282 us; of
//               d 2560, inter 9728 at 3001 tokens: 512 us, then 454 us);
//   warp 18     loads the packed codes and scales/zeros of the CTA's 8 row
//               tiles (TMA, one box each per projection and block) into their
//               own ring.
// The activation tiles, the B tiles and the packed codes have rings of their
// own depths: each slot is released by what last reads it (the MMAs' commit,
// or the dequantizing warps for the codes).
// What bounds it now (clock stamps, gate/up): a stage of 64 features takes ~1100
// clocks where its MMAs need 1024, a tile ~4400 before its first MMA and ~7800
// for its epilogue, half of them the 2 x 32768 exponentials and reciprocals.
// Measured with 256-row down tiles, the reduction kernel, 3 B tiles and the
// sector-wide stores: the d 5120 layer at 512 tokens 209 us, the d 2560 layer at
// 3001 tokens 357 us.
// Stages are handed over with mbarriers; every wait is bounded (a timeout
// sets the device status word and the CTA skips the rest of its work).
#include <algorithm>
#include <cmath>
#include <mutex>

#include <cuda.h>
#include <cudaTypedefs.h>

#include "wq_internal.h"
#include "wq_ptx.cuh"

namespace wq {

// Device status word of the GEMM kernels: WQ_OK (0) or WQ_ERR_TIMEOUT (-6).
__device__ int g_gemm_status = 0;

namespace {

constexpr int kBM = 128;                         // tokens per CTA tile (MMA M)
constexpr int kBN = 128;                         // output rows per CTA tile and projection (MMA N)
constexpr int kDeqWarps = 16;                    // dequantizing warps, two groups that take alternate stages
constexpr int kDeqGroup = kDeqWarps / 2;
constexpr int kProducerWarp = kDeqWarps;         // activation tiles
constexpr int kMmaWarp = kDeqWarps + 1;          // TMEM owner and MMA issuer
constexpr int kRawWarp = kDeqWarps + 2;          // packed-code ring
constexpr int kGemmThreads = (kDeqWarps + 3) * 32;
constexpr int kTileBytes = kBM * 64 * 2;         // one 128 x 64 binary16 operand tile (a stage)
constexpr int kHalves = 2;                       // token halves of kBM a CTA can take (GemmArgs::mt)
constexpr uint32_t kSboTile = 8 * 128;           // bytes between 8-row groups of a 64-feature B tile
constexpr int kLoraK = 32;                       // LoRA rank columns a stage
constexpr uint32_t kGemmSmemLimit = 232448;      // 227 KB opt-in

// EXACT: every weight s (q - z) is written as two binary16 tiles whose sum is
// exact -- s_hi (q - z) and s_lo (q - z), s_hi the scale with its 4 lowest
// mantissa bits cleared and s_lo = s - s_hi -- and the tensor cores add both
// (two MMAs a k-step), so the products are those of the exact weights.  Used
// for fp32 output; otherwise each weight is rounded to binary16 once.
template <int BITS, int NPROJ, int GROUP, bool EXACT>
struct GemmCfg {
  static constexpr int BPK = BITS == 2 ? 512 : 1024;      // code bytes per (16-row tile, block)
  static constexpr int GPB = 128 / GROUP;
  static constexpr int NB = NPROJ * (EXACT ? 2 : 1);      // B tiles a stage
  // The ring of packed codes holds whole blocks (two stages) of 2-bit codes,
  // whose two halves interleave, and half blocks (a stage) of 4-bit codes.
  static constexpr bool HALFRAW = BITS == 4;
  static constexpr int CPR = HALFRAW ? BPK / 2 : BPK;               // code bytes of a row tile in a ring slot
  static constexpr int GPR = HALFRAW && GPB > 1 ? GPB / 2 : GPB;    // groups whose scales/zeros it holds
  static constexpr int RAW_TILE = CPR + GPR * 64;          // codes + scales/zeros of a row tile
  static constexpr int RAWP = 8 * RAW_TILE;                // a projection's: [8 tiles][codes], then [8 tiles][meta]
  static constexpr int RAW = NPROJ * RAWP;                 // a slot of the ring
  static constexpr int BT = NB * kTileBytes;               // a stage's B tiles
  static constexpr int AT = kHalves * kTileBytes;          // a stage's activation tiles (both token halves)
  // 1 KB for the barriers, 1 KB to align the tiles on 1024 bytes
  static constexpr int AVAIL = (int)kGemmSmemLimit - 2048;
  // Three rings.  B tiles: 3 (2 where 3 would leave fewer than 3 activation
  // stages) -- with 2 the dequantization of a tile and its hand-over have to
  // fit into one stage of MMAs; the third, bought with a fourth activation
  // stage, took gate/up at 3001 tokens of d 2560 from 213 to 194 us.
  // Activation tiles (from L2): what is left, at most 8; then the packed codes.
  static constexpr int SB = (AVAIL - 3 * BT - 3 * RAW) / AT >= 3 ? 3 : 2;
  // (small slots: 8, so that enough of the weights is in flight at few tokens)
  static constexpr int RMIN = HALFRAW && NB == 1 ? 8 : 3;
  static constexpr int SA = std::min(8, (AVAIL - SB * BT - RMIN * RAW) / AT);
  static constexpr int R = std::min(HALFRAW ? 12 : 6, (AVAIL - SA * AT - SB * BT) / RAW);
  static_assert(SA >= 2 && R >= 2, "GEMM pipeline does not fit");
  static constexpr int OFF_A = 0;
  static constexpr int OFF_B = SA * AT;
  static constexpr int OFF_RAW = OFF_B + SB * BT;
  static constexpr int OFF_BAR = OFF_RAW + R * RAW;
  static constexpr int SMEM = OFF_BAR + (2 * SA + 3 * SB + 3 * R + 2) * 8 + 16 + 1024;  // + alignment slack
  static constexpr int NCH = NPROJ * kBN;                  // TMEM columns of a token half (fp32 accumulators)
  static constexpr int NCOLS = kHalves * NCH;
  static_assert(SMEM <= (int)kGemmSmemLimit, "GEMM stage does not fit");
};

__device__ __forceinline__ void gemm_timeout() { atomicExch(&g_gemm_status, -6); }

// After a timeout, before the CTA ends: time for the loads and MMAs that its other
// roles issued last (microseconds each) to end, so that none reaches shared memory
// or TMEM that has changed hands.
__device__ __noinline__ void gemm_settle() {
  const unsigned long long t0 = global_timer_ns();
  for (int i = 0; i < 1 << 20 && global_timer_ns() - t0 < 2000000ull; ++i) __nanosleep(1000);
}

// Byte offset of element (row, k) in a K-major no-swizzle tile whose 8-row
// groups are `sbo` bytes apart (core matrices along K 128 bytes apart).
__device__ __forceinline__ uint32_t kmajor_off(int row, int k, uint32_t sbo) {
  return (uint32_t)(row >> 3) * sbo + (uint32_t)(k >> 3) * 128u + (uint32_t)(row & 7) * 16u + (uint32_t)(k & 7) * 2u;
}

__device__ __forceinline__ uint32_t h2bits(__half2 v) { return *reinterpret_cast<uint32_t *>(&v); }
__device__ __forceinline__ __half2 bits2h(uint32_t v) { return *reinterpret_cast<__half2 *>(&v); }

// The tensor maps of a launch: the activations, and per projection the packed
// codes viewed as [RT][KB * BPK / 128][128 bytes] and the scales/zeros as
// [RT][KB * GPB][64 bytes].
struct GemmMaps {
  CUtensorMap act, codes[2], meta[2];
};

// 3-D TMA load (coordinates innermost first), completing on `bar`.
__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map, int x, int y, int z, uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
          smem_addr(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_addr(bar))
      : "memory");
}

// 2-D TMA load of a box of the activations into shared memory, completing
// on `bar` with its byte count.  x (the feature coordinate) is a multiple of 64.
__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, int x, int y, uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_addr(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_addr(bar))
      : "memory");
}

// ---------------------------------------------------------------------------
// Pieces shared by the two kernels below.
// ---------------------------------------------------------------------------

// Dequantizes the stage hb (features 64 hb .. 64 hb + 63) of a block of
// packed codes `raw` into the B tiles `Bs`: thread dt of a group of 8 warps
// takes lane dt % 32 of the fragment layout of 16-row tile dt / 32, for every
// projection.
template <int BITS, int NPROJ, int GROUP, bool EXACT>
__device__ __forceinline__ void gemm_deq_stage(const uint8_t *raw, uint8_t *Bs, int hb, int dt) {
  using C = GemmCfg<BITS, NPROJ, GROUP, EXACT>;
  constexpr int GPB = C::GPB, GS = GROUP / 16;
#pragma unroll
  for (int p = 0; p < NPROJ; ++p) {
    const int j = dt >> 5, L = dt & 31;
    const int g = L >> 2;
    uint8_t *Bp = Bs + p * kTileBytes;
    // the lane's code words of this half block: 2-bit, words 2 hb, 2 hb + 1
    // of its 16 bytes; 4-bit, the 16 bytes of half hb
    uint32_t wds[BITS == 2 ? 2 : 4];
    const uint8_t *cb = raw + p * C::RAWP + j * C::CPR;                       // codes of tile j
    const uint8_t *mb = raw + p * C::RAWP + 8 * C::CPR + j * C::GPR * 64;  // its scales/zeros
    if (BITS == 2) {
      const uint2 w0 = lds64(cb + L * 16 + hb * 8);
      wds[0] = w0.x;
      wds[1] = w0.y;
    } else {
      const uint4 w0 = lds128(cb + L * 16);
      wds[0] = w0.x;
      wds[1] = w0.y;
      wds[2] = w0.z;
      wds[3] = w0.w;
    }
    // this stage: k-steps 4 hb .. 4 hb + 3 of the block
#pragma unroll
    for (int gl = 0; gl < (GS >= 4 ? 1 : 4 / GS); ++gl) {
      const int gi = (4 * hb) / GS + gl;
      // scales and zeros of rows g and g + 8 in group gi (zero for tiles outside the matrix)
      const uint2 sz = lds64(mb + (C::HALFRAW ? gl : gi) * 64 + g * 8);
      // scales of rows g ("lo" row) and g + 8 ("hi" row); EXACT splits each
      // into a head with the 4 lowest mantissa bits cleared and the tail
      const uint32_t sg = sz.x & 0xffffu, sg8 = sz.x >> 16;
      const __half2 s_lo = __half2half2(__ushort_as_half((unsigned short)(EXACT ? (sg & 0xfff0u) : sg)));
      const __half2 s_hi = __half2half2(__ushort_as_half((unsigned short)(EXACT ? (sg8 & 0xfff0u) : sg8)));
      const __half2 t_lo = __half2half2(
          __hsub(__ushort_as_half((unsigned short)sg), __ushort_as_half((unsigned short)(sg & 0xfff0u))));
      const __half2 t_hi = __half2half2(
          __hsub(__ushort_as_half((unsigned short)sg8), __ushort_as_half((unsigned short)(sg8 & 0xfff0u))));
      // 1024 + z: the code read as 1024 + q minus this is q - z exactly
      const __half2 z_lo =
          __half2half2(__hadd(__ushort_as_half((unsigned short)(sz.y & 0xffffu)), __float2half(1024.f)));
      const __half2 z_hi = __half2half2(__hadd(__ushort_as_half((unsigned short)(sz.y >> 16)), __float2half(1024.f)));
#pragma unroll
      for (int kk = 0; kk < (GS >= 4 ? 4 : GS); ++kk) {
        const int ks = (GS >= 4 ? 4 * hb : gi * GS) + kk;
        uint32_t q[4];  // (row g, k 2t..2t+1), (row g+8, ...), (row g, k 2t+8..), (row g+8, k 2t+8..)
        const int kl = ks - 4 * hb;  // k-step within the half block
        if (BITS == 2) {
          const uint32_t x = wds[(kl >> 1) & 1];
          const int s4 = (kl & 1) * 4;
          q[0] = (x >> s4) & 0x00030003u;
          q[1] = (x >> (s4 + 8)) & 0x00030003u;
          q[2] = (x >> (s4 + 2)) & 0x00030003u;
          q[3] = (x >> (s4 + 10)) & 0x00030003u;
        } else {
          const uint32_t x = wds[kl & 3];
          q[0] = x & 0x000F000Fu;
          q[1] = (x >> 8) & 0x000F000Fu;
          q[2] = (x >> 4) & 0x000F000Fu;
          q[3] = (x >> 12) & 0x000F000Fu;
        }
        uint32_t w[4], wl[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const __half2 v = bits2h(q[e] | 0x64006400u);  // 1024 + q, exact
          const bool hi_row = (e & 1) != 0;
          const __half2 qz = __hsub2(v, hi_row ? z_hi : z_lo);  // q - z, exact
          w[e] = h2bits(__hmul2(qz, hi_row ? s_hi : s_lo));
          if (EXACT) wl[e] = h2bits(__hmul2(qz, hi_row ? t_hi : t_lo));
        }
        // the four 8x8 blocks (rows +0/+8, k +0/+8) of this k-step are core
        // matrices of the K-major tile: one matrix store; lane L gives row
        // L % 8 of block L / 8
        const int blk = L >> 3;
        const uint32_t dst = smem_addr(Bp) + (uint32_t)(2 * j + (blk & 1)) * kSboTile +
                             (uint32_t)(2 * kl + (blk >> 1)) * 128u + (uint32_t)(L & 7) * 16u;
        stmatrix_x4(dst, w[0], w[1], w[2], w[3]);
        if (EXACT) stmatrix_x4(dst + NPROJ * kTileBytes, wl[0], wl[1], wl[2], wl[3]);
      }
    }
  }
}

// Ring slot of packed codes and scales/zeros (TMA; one thread): block kb (with
// HALFRAW its half hb) of the 8 row tiles from n0 / 16 of each projection (TALL:
// of the next 8 row tiles); row tiles past the matrix read as zeros.
template <class C, int NPROJ, bool TALL>
__device__ __forceinline__ void gemm_load_raw(const GemmMaps &tm, uint8_t *dst, int n0, int kb, int hb, uint64_t *full) {
  mbar_arrive_expect_tx(full, (uint32_t)C::RAW);
  const int y = kb * (C::BPK / 128) + (C::HALFRAW ? hb * (C::CPR / 128) : 0);
  const int ym = kb * C::GPB + (C::GPR < C::GPB ? hb * C::GPR : 0);
#pragma unroll
  for (int p = 0; p < NPROJ; ++p) {
    const int z = n0 / 16 + (TALL ? 8 * p : 0);
    tma_load_3d(dst + p * C::RAWP, &tm.codes[TALL ? 0 : p], 0, y, z, full);
    tma_load_3d(dst + p * C::RAWP + 8 * C::CPR, &tm.meta[TALL ? 0 : p], 0, ym, z, full);
  }
}

// LoRA stage l, B side: rows n0 .. n0 + 127 of B_p (bf16 [N][r]), rank
// columns 32 l .. 32 l + 31 -> binary16, zeros past r.
template <int NPROJ>
__device__ __forceinline__ void gemm_lora_b_stage(const GemmArgs &a, uint8_t *Bs, int n0, int l, int dt) {
  constexpr uint32_t sbo = 4 * 128u;
  for (int i = dt; i < NPROJ * kBN * 4; i += kDeqGroup * 32) {
    const int p = i / (kBN * 4), rem = i - p * kBN * 4;
    const int nl = rem >> 2, c = rem & 3;
    const int n = n0 + nl, col = l * kLoraK + c * 8;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (n < a.N && col < a.r)
      v = __ldg(reinterpret_cast<const uint4 *>(reinterpret_cast<const uint8_t *>(a.lora_b[p]) +
                                                ((size_t)n * a.r + col) * 2));
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    uint32_t o[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float lo = __uint_as_float(w[e] << 16), hi = __uint_as_float(w[e] & 0xffff0000u);
      o[e] = h2bits(__floats2half2_rn(lo, hi));
    }
    *reinterpret_cast<uint4 *>(Bs + p * (kBN * kLoraK * 2) + kmajor_off(nl, c * 8, sbo)) =
        make_uint4(o[0], o[1], o[2], o[3]);
  }
}

// LoRA stage l, A side (one warp): lora_scale * t, rank columns 32 l .. 32 l
// + 31 of gate (first r columns of ta) and of up (next r) for the mth token
// halves from m0, zeros past r; lane 0 arrives on `full` once all landed.
template <int NPROJ>
__device__ __forceinline__ void gemm_lora_a_stage(const GemmArgs &a, uint8_t *As, int m0, int mth, int l, int lane,
                                                  uint64_t *full) {
  for (int i = lane; i < mth * NPROJ * kBM * 4; i += 32) {
    const int h = i / (NPROJ * kBM * 4), hr = i - h * NPROJ * kBM * 4;
    const int p = hr / (kBM * 4), rem = hr - p * kBM * 4;
    const int ml = rem >> 2, c = rem & 3;
    const int m = m0 + h * kBM + ml, col = l * kLoraK + c * 8;
    const bool in = m < a.M && col < a.r;
    const uint16_t *src = in ? a.ta + (size_t)m * 2 * a.r + p * a.r + col : a.ta;
    cp_async16_zfill(As + h * kTileBytes + p * (kBM * kLoraK * 2) + kmajor_off(ml, c * 8, 4 * 128u), src,
                     in ? 16u : 0u);
  }
  // once landed, each lane fences its generic-proxy writes against the tensor
  // cores' reads, then lane 0 arrives
  cp_async_wait_all();
  fence_proxy_async_smem();
  __syncwarp();
  if (lane == 0) mbar_arrive(full);
}

// The MMAs of one stage (one thread): every token half multiplies the same B
// tile into its own accumulators; `first` starts the accumulators.
template <int NPROJ, bool EXACT>
__device__ __forceinline__ void gemm_issue_stage(uint32_t tmem, uint32_t as0, uint32_t bs, int mth, bool wstage,
                                                 bool first) {
  constexpr int NCH = NPROJ * kBN;
  // gate/up: one MMA of N = 256 a k-step (the gate tile and the up tile are
  // adjacent, 256 rows), so the activation tile is read once
  constexpr uint32_t idesc = umma_idesc_f16(kBM, kBN);
  constexpr uint32_t idesc2 = umma_idesc_f16(kBM, 2 * kBN);
  for (int h = 0; h < mth; ++h) {
    const uint32_t as = as0 + h * kTileBytes, th = tmem + h * NCH;
    if (wstage && NPROJ == 2 && !EXACT) {
#pragma unroll
      for (int ks = 0; ks < 4; ++ks)
        umma_f16(th, umma_desc_kmajor_sw128(as + ks * 32, 1024), umma_desc_kmajor(bs + ks * 256, 128, kSboTile), idesc2,
                 (first && ks == 0) ? 0u : 1u);
    } else if (wstage) {
#pragma unroll
      for (int p = 0; p < NPROJ; ++p)
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
          // A (swizzled TMA layout): k-step ks at byte 32 ks of each row
          umma_f16(th + p * kBN, umma_desc_kmajor_sw128(as + ks * 32, 1024),
                   umma_desc_kmajor(bs + p * kTileBytes + ks * 256, 128, kSboTile), idesc,
                   (first && ks == 0) ? 0u : 1u);
          if (EXACT)  // the low parts of the same weights
            umma_f16(th + p * kBN, umma_desc_kmajor_sw128(as + ks * 32, 1024),
                     umma_desc_kmajor(bs + (NPROJ + p) * kTileBytes + ks * 256, 128, kSboTile), idesc, 1u);
        }
    } else {
      constexpr uint32_t sbo = 4 * 128u;  // 32 rank columns a LoRA stage
      for (int p = 0; p < NPROJ; ++p)
        for (int ks = 0; ks < kLoraK / 16; ++ks)
          umma_f16(th + p * kBN, umma_desc_kmajor(as + p * (kBM * kLoraK * 2) + ks * 256, 128, sbo),
                   umma_desc_kmajor(bs + p * (kBN * kLoraK * 2) + ks * 256, 128, sbo), idesc,
                   (first && ks == 0) ? 0u : 1u);
    }
  }
}

// 4 x 4 transpose of 16-byte chunks over groups of 4 lanes: afterwards v[i] is
// chunk lane % 4 of lane (lane & ~3) + i.
__device__ __forceinline__ void transpose4(uint4 (&v)[4], int lane) {
#pragma unroll
  for (int st = 1; st <= 2; st <<= 1) {
    const bool hi = (lane & st) != 0;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int lo_i = st == 1 ? 2 * q : q, hi_i = lo_i + st;
      uint4 give = hi ? v[lo_i] : v[hi_i];
      give.x = __shfl_xor_sync(0xffffffffu, give.x, st);
      give.y = __shfl_xor_sync(0xffffffffu, give.y, st);
      give.z = __shfl_xor_sync(0xffffffffu, give.z, st);
      give.w = __shfl_xor_sync(0xffffffffu, give.w, st);
      if (hi) v[lo_i] = give; else v[hi_i] = give;
    }
  }
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t *>(&v);
}

// h = SiLU(rs g) (rs u) of 16 columns, in place of g.
__device__ __forceinline__ void gemm_silu16(float *g, const float (&u)[16], float rs) {
#pragma unroll
  for (int e = 0; e < 16; ++e) {
    const float gv = rs * g[e];
    g[e] = __fdividef(gv, 1.f + __expf(-gv)) * (rs * u[e]);
  }
}

// Stores 32 output rows nb .. nb + 31 of the tokens mw + lane (one a lane): v,
// for down plus the residual.  Four lanes exchange their 16-byte chunks first,
// so that a store instruction writes 64 contiguous bytes of 8 tokens (whole
// sectors) instead of 16 bytes of 32; the residual is read the same way.
template <bool GATEUP>
__device__ __forceinline__ void gemm_emit32(const GemmArgs &a, int mw, int nb, float (&v)[32], int lane) {
  const bool f32 = !GATEUP && a.out_f32;
  const size_t row = (size_t)(mw + lane) * a.N + nb;
  if ((a.N & 7) != 0) {  // ragged rows: a token a lane
    if (mw + lane >= a.M) return;
    if (!GATEUP && a.residual) {
#pragma unroll
      for (int e = 0; e < 32; ++e)
        if (nb + e < a.N) v[e] += __bfloat162float(reinterpret_cast<const __nv_bfloat16 *>(a.residual)[row + e]);
    }
#pragma unroll
    for (int e = 0; e < 32; ++e) {
      if (nb + e >= a.N) continue;
      if (f32)
        reinterpret_cast<float *>(a.out)[row + e] = v[e];
      else
        reinterpret_cast<__nv_bfloat16 *>(a.out)[row + e] = __float2bfloat16_rn(v[e]);
    }
    return;
  }
  const int col = nb + 8 * (lane & 3), m4 = mw + (lane & ~3);
  uint4 o[4];
  if (!GATEUP && a.residual) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      o[i] = m4 + i < a.M && col < a.N
                 ? *reinterpret_cast<const uint4 *>(reinterpret_cast<const __nv_bfloat16 *>(a.residual) +
                                                    (size_t)(m4 + i) * a.N + col)
                 : make_uint4(0u, 0u, 0u, 0u);
    transpose4(o, lane);  // chunk i of this lane's token
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t w[4] = {o[i].x, o[i].y, o[i].z, o[i].w};
#pragma unroll
      for (int e = 0; e < 8; ++e)
        v[8 * i + e] += __uint_as_float(e & 1 ? (w[e >> 1] & 0xffff0000u) : (w[e >> 1] << 16));
    }
  }
  if (f32) {  // 128 contiguous bytes a lane
    if (mw + lane >= a.M) return;
#pragma unroll
    for (int e = 0; e < 32; e += 4)
      if (nb + e < a.N)
        *reinterpret_cast<float4 *>(reinterpret_cast<float *>(a.out) + row + e) =
            make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
    return;
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
    o[i] = make_uint4(pack_bf16(v[8 * i], v[8 * i + 1]), pack_bf16(v[8 * i + 2], v[8 * i + 3]),
                      pack_bf16(v[8 * i + 4], v[8 * i + 5]), pack_bf16(v[8 * i + 6], v[8 * i + 7]));
  transpose4(o, lane);
#pragma unroll
  for (int i = 0; i < 4; ++i)
    if (m4 + i < a.M && col < a.N)
      *reinterpret_cast<uint4 *>(reinterpret_cast<__nv_bfloat16 *>(a.out) + (size_t)(m4 + i) * a.N + col) = o[i];
}

// A warp's share of a finished tile from TMEM: its 32 tokens of half h, 32
// columns of each accumulator (gate and up; down: one, or with TALL the two
// 128-row halves of the tile).
template <int NPROJ, bool TALL>
__device__ __forceinline__ void gemm_emit_tmem(const GemmArgs &a, uint32_t taddr, int mw, int nb, int lane) {
  const float rs = a.rs != nullptr && mw + lane < a.M ? a.rs[mw + lane] : 1.f;
#pragma unroll 1
  for (int p = 0; p < (TALL ? 2 : 1); ++p) {
    float g[32];
    tmem_ld32(taddr + p * kBN, reinterpret_cast<uint32_t(&)[32]>(g));
    if (NPROJ == 2 && !TALL) {
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        float u[16];
        tmem_ld16(taddr + kBN + 16 * q, reinterpret_cast<uint32_t(&)[16]>(u));
        tmem_ld_wait();
        gemm_silu16(g + 16 * q, u, rs);
      }
    } else {
      tmem_ld_wait();
#pragma unroll
      for (int e = 0; e < 32; ++e) g[e] *= rs;
    }
    gemm_emit32<NPROJ == 2 && !TALL>(a, mw, nb + p * kBN, g, lane);
  }
}

// Shared memory of a launch: the barriers behind the rings, then the TMEM
// base address and the abort flag.
// raw_full and b_empty have two barriers a slot, for its even and its odd uses:
// a dequantizing group waits for its own stages only, every other one, so that
// with one barrier the phase it waits for could have the parity of an earlier
// one that it never waited for.  With two, the barrier's next phase belongs to
// a use that cannot begin before this one, and its previous phase has completed
// before the group's last stage.
// acc_full is the MMAs' completion of a part, acc_empty the 16 dequantizing warps'
// reads of its accumulators: the next part's first MMA, for whose B tile one
// group of 8 suffices, starts them anew.
template <class C>
struct GemmSmem {
  uint8_t *base;
  uint64_t *raw_full, *raw_empty, *a_full, *a_empty, *b_full, *b_empty, *acc_full, *acc_empty;
  uint32_t *tmem_s;
  volatile int *abort_s;
  __device__ explicit GemmSmem(uint8_t *smem_raw) {
    // the swizzled activation tiles need 1024-byte alignment
    base = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
    raw_full = reinterpret_cast<uint64_t *>(base + C::OFF_BAR);
    raw_empty = raw_full + 2 * C::R;
    a_full = raw_empty + C::R;
    a_empty = a_full + C::SA;
    b_full = a_empty + C::SA;
    b_empty = b_full + C::SB;
    acc_full = b_empty + 2 * C::SB;
    acc_empty = acc_full + 1;
    tmem_s = reinterpret_cast<uint32_t *>(acc_empty + 1);
    abort_s = reinterpret_cast<volatile int *>(tmem_s + 1);
  }
  // thread 0: barrier initialisation; the MMA warp: TMEM allocation
  __device__ void init(int tid, int warp) {
    if (tid == 0) {
      for (int q = 0; q < C::R; ++q) {
        mbar_init(&raw_full[2 * q], 1);
        mbar_init(&raw_full[2 * q + 1], 1);
        mbar_init(&raw_empty[q], C::HALFRAW ? kDeqGroup : kDeqWarps);
      }
      for (int s = 0; s < C::SA; ++s) {
        mbar_init(&a_full[s], 1);
        mbar_init(&a_empty[s], 1);
      }
      for (int s = 0; s < C::SB; ++s) {
        mbar_init(&b_full[s], kDeqGroup);
        mbar_init(&b_empty[2 * s], 1);
        mbar_init(&b_empty[2 * s + 1], 1);
      }
      mbar_init(acc_full, 1);
      mbar_init(acc_empty, kDeqWarps);
      *abort_s = 0;
      fence_barrier_init();
    }
    if (warp == kMmaWarp) tmem_alloc(tmem_s, C::NCOLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
  }
};

// ---------------------------------------------------------------------------
// One tile a CTA: grid (token tiles, row tiles).
// ---------------------------------------------------------------------------
template <int BITS, int NPROJ, int GROUP, bool EXACT, bool TALL>
__global__ void __launch_bounds__(kGemmThreads, 1) qgemm_tile_kernel(const GemmArgs a, const __grid_constant__ GemmMaps tm) {
  using C = GemmCfg<BITS, NPROJ, GROUP, EXACT>;
  constexpr int SA = C::SA, SB = C::SB, R = C::R;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  GemmSmem<C> sm(smem_raw);
  uint8_t *smem = sm.base;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = blockIdx.x * a.mt * kBM, n0 = blockIdx.y * (TALL ? 2 * kBN : kBN);
  const int mth = min(a.mt, (a.M - m0 + kBM - 1) / kBM);  // token halves with tokens in them
  const int KB = (a.K + 127) / 128;
  const int nws = 2 * KB;  // weight stages (64 features each)
  const int nlora = NPROJ == 2 && !TALL && a.r > 0 ? (a.r + kLoraK - 1) / kLoraK : 0;
  const int nit = nws + nlora;
  sm.init(tid, warp);
  const uint32_t tmem = *sm.tmem_s;

  // bounded wait; a timeout (or an earlier one) makes the caller skip its work
  auto wait = [&](uint64_t *bar, uint32_t parity) -> bool {
    if (mbar_try_wait(bar, parity)) return true;
    if (*sm.abort_s) return false;
    if (mbar_wait_sleep(bar, parity)) return true;
    *sm.abort_s = 1;
    gemm_timeout();
    return false;
  };

  if (warp == kRawWarp) {
    // ---- packed codes and scales/zeros (TMA) into their ring; row tiles
    // past the matrix read as zeros ----
    if (elect_one())
      for (int it = 0; it < (C::HALFRAW ? nws : KB); ++it) {
        const int q = it % R;
        if (it >= R && !wait(&sm.raw_empty[q], (it / R - 1) & 1)) break;
        gemm_load_raw<C, NPROJ, TALL>(tm, smem + C::OFF_RAW + q * C::RAW, n0, C::HALFRAW ? it >> 1 : it, it & 1,
                                      &sm.raw_full[2 * q + (it / R & 1)]);
      }
    __syncwarp();
  } else if (warp == kProducerWarp) {
    // ---- activation tiles (TMA); the LoRA stages' by cp.async ----
    for (int it = 0; it < nit; ++it) {
      const int s = it % SA;
      if (it >= SA && !wait(&sm.a_empty[s], (it / SA - 1) & 1)) break;
      uint8_t *As = smem + C::OFF_A + s * C::AT;
      if (it < nws) {
        if (lane == 0) {
          // per token half one box of 64 features x 128 tokens, a 128-byte row
          // per token, swizzled (8-row groups 1 KB apart)
          mbar_arrive_expect_tx(&sm.a_full[s], (uint32_t)(mth * kTileBytes));
          for (int h = 0; h < mth; ++h) tma_load_2d(As + h * kTileBytes, &tm.act, it * 64, m0 + h * kBM, &sm.a_full[s]);
        }
      } else {
        gemm_lora_a_stage<NPROJ>(a, As, m0, mth, it - nws, lane, &sm.a_full[s]);
      }
    }
  } else if (warp == kMmaWarp) {
    // ---- MMA issue ----
    if (elect_one()) {
      for (int it = 0; it < nit; ++it) {
        const int sa = it % SA, sb = it % SB;
        if (!wait(&sm.a_full[sa], (it / SA) & 1) || !wait(&sm.b_full[sb], (it / SB) & 1)) break;
        tc_fence_after();
        gemm_issue_stage<NPROJ, EXACT>(tmem, smem_addr(smem + C::OFF_A + sa * C::AT),
                                       smem_addr(smem + C::OFF_B + sb * C::BT), mth, it < nws, it == 0);
        // both slots are free once these MMAs have read them
        umma_commit(&sm.a_empty[sa]);
        umma_commit(&sm.b_empty[2 * sb + (it / SB & 1)]);
      }
      umma_commit(sm.acc_full);
    }
    __syncwarp();
  } else {
    // ---- dequantization into the B tiles ----
    const int hb = warp / kDeqGroup, dt = tid & (kDeqGroup * 32 - 1);
    for (int it = hb; it < nit; it += 2) {
      const int s = it % SB, kr = C::HALFRAW ? it : it >> 1, q = kr % R;
      const int ur = kr / R, ub = it / SB - 1;  // the slots' uses waited for
      if (it < nws && !wait(&sm.raw_full[2 * q + (ur & 1)], (ur >> 1) & 1)) break;
      if (it >= SB && !wait(&sm.b_empty[2 * s + (ub & 1)], (ub >> 1) & 1)) break;
      uint8_t *Bs = smem + C::OFF_B + s * C::BT;
      if (it < nws)
        gemm_deq_stage<BITS, NPROJ, GROUP, EXACT>(smem + C::OFF_RAW + q * C::RAW, Bs, hb, dt);
      else
        gemm_lora_b_stage<NPROJ>(a, Bs, n0, it - nws, dt);
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&sm.b_full[s]);
        if (it < nws) mbar_arrive(&sm.raw_empty[q]);  // this warp's half of the block's codes is read
      }
    }

    // ---- epilogue: warp w reads TMEM lanes 32 (w % 4) .. 32 (w % 4) + 31
    // (the tokens of each half) and columns 32 (w / 4) .. 32 (w / 4) + 31 ----
    if (wait(sm.acc_full, 0)) {
      tc_fence_after();
      const int quarter = warp & 3, c0 = (warp >> 2) * 32;
      for (int h = 0; h < mth; ++h)
        gemm_emit_tmem<NPROJ, TALL>(a, tmem + h * C::NCH + ((uint32_t)(quarter * 32) << 16) + c0,
                                    m0 + h * kBM + quarter * 32, n0 + c0, lane);
    }
  }

  if (*sm.abort_s) gemm_settle();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == kMmaWarp) tmem_dealloc(tmem, C::NCOLS);
}

// ---------------------------------------------------------------------------
// Stream-K: gridDim.x persistent CTAs divide the T * U work units evenly.
// ---------------------------------------------------------------------------
// The tiles (mt * 128 tokens x 128 rows) are cut into units of one
// 128-feature block (plus one unit for the LoRA stages); CTA c takes units
// [c W / P, (c + 1) W / P) of the W = T * U in order, i.e. whole tiles and at
// most one part of a tile at each end of its range.

// The epilogue of one part of a tile (the 16 dequantizing warps, after the
// part's accumulators are complete; `have`: no timeout so far).  Warp w reads
// TMEM lanes 32 (w % 4) .. 32 (w % 4) + 31 (the tokens of each half) and
// columns 32 (w / 4) .. 32 (w / 4) + 31.  A whole tile is finished from TMEM;
// a part of a split tile is written to its scratch slot, and gemm_reduce_kernel
// adds a tile's parts and finishes it: with all SMs, where the CTA of the last
// part alone took 25 to 35 us for a tile of 256 tokens x 256 rows in 5 parts.
// Kept out of line so that the dequantization loop keeps its registers.
template <int BITS, int NPROJ, int GROUP, bool EXACT, bool TALL>
__device__ __noinline__ void gemm_part_epilogue(const GemmArgs &a, uint32_t tmem, int tile, int ub, int ue, int U,
                                                long long g0, bool have) {
  using C = GemmCfg<BITS, NPROJ, GROUP, EXACT>;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int quarter = warp & 3, c0 = (warp >> 2) * 32;
  const int MT = (a.M + a.mt * kBM - 1) / (a.mt * kBM);
  const int m0 = (tile % MT) * a.mt * kBM, n0 = (tile / MT) * (TALL ? 2 * kBN : kBN);
  const int mth = min(a.mt, (a.M - m0 + kBM - 1) / kBM);
  // a scratch slot: [half][accumulator][column / 4][128 tokens][4] floats, so that
  // a warp's accesses are contiguous
  constexpr int SLOT = kHalves * kBM * C::NCH;
  auto part_at = [&](float *slot, int h, int p) {
    return reinterpret_cast<float4 *>(slot) + (((size_t)h * NPROJ + p) * (kBN / 4) + c0 / 4) * kBM + quarter * 32 + lane;
  };
  const bool whole = ub == 0 && ue == U;
  // a split part's scratch slot: the CTA's first part (0) or its last (1)
  float *mine = whole ? nullptr : a.sk_part + ((size_t)blockIdx.x * 2 + ((long long)tile * U + ub == g0 ? 0 : 1)) * SLOT;
  for (int h = 0; h < mth && have; ++h) {
    const uint32_t tl = tmem + h * C::NCH + ((uint32_t)(quarter * 32) << 16) + c0;
    if (whole) {
      gemm_emit_tmem<NPROJ, TALL>(a, tl, m0 + h * kBM + quarter * 32, n0 + c0, lane);
    } else {
#pragma unroll 1
      for (int p = 0; p < NPROJ; ++p) {
        uint32_t v[32];
        tmem_ld32(tl + p * kBN, v);
        tmem_ld_wait();
        float4 *dst = part_at(mine, h, p);
#pragma unroll
        for (int q = 0; q < 8; ++q)
          __stcg(dst + q * kBM, make_float4(__uint_as_float(v[4 * q]), __uint_as_float(v[4 * q + 1]),
                                            __uint_as_float(v[4 * q + 2]), __uint_as_float(v[4 * q + 3])));
      }
    }
  }
}

template <int BITS, int NPROJ, int GROUP, bool EXACT, bool TALL>
__global__ void __launch_bounds__(kGemmThreads, 1) qgemm_sk_kernel(const __grid_constant__ GemmArgs a,
                                                                   const __grid_constant__ GemmMaps tm) {
  using C = GemmCfg<BITS, NPROJ, GROUP, EXACT>;
  constexpr int SA = C::SA, SB = C::SB, R = C::R;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  GemmSmem<C> sm(smem_raw);
  uint8_t *smem = sm.base;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int KB = (a.K + 127) / 128;
  const int nlora = NPROJ == 2 && !TALL && a.r > 0 ? (a.r + kLoraK - 1) / kLoraK : 0;
  const int U = KB + (nlora > 0 ? 1 : 0);
  constexpr int ROWS = TALL ? 2 * kBN : kBN;  // output rows of a tile
  const int MT = (a.M + a.mt * kBM - 1) / (a.mt * kBM), NT = (a.N + ROWS - 1) / ROWS;
  const long long W = (long long)MT * NT * U, P = gridDim.x;
  const long long g0 = W * blockIdx.x / P, g1 = W * (blockIdx.x + 1) / P;
  sm.init(tid, warp);
  const uint32_t tmem = *sm.tmem_s;

  auto wait = [&](uint64_t *bar, uint32_t parity) -> bool {
    if (mbar_try_wait(bar, parity)) return true;
    if (*sm.abort_s) return false;
    if (mbar_wait_sleep(bar, parity)) return true;
    *sm.abort_s = 1;
    gemm_timeout();
    return false;
  };
  // The parts of tiles in this CTA's range, in order: tile, units [ub, ue),
  // weight blocks wb, stages nit (two a block, then the LoRA stages); token
  // tiles vary fastest, so neighbouring CTAs share row tiles.
#define WQ_FOR_EACH_PART                                                         \
  for (long long g_ = g0; g_ < g1;)                                              \
    for (int tile = (int)(g_ / U), ub = (int)(g_ - (long long)tile * U),         \
             ue = (int)min((long long)U, ub + (g1 - g_)), wb = min(ue, KB) - ub, \
             nit = 2 * wb + (ue > KB ? nlora : 0), once_ = (g_ += ue - ub, 1);   \
         once_; once_ = 0)
  auto tile_m0 = [&](int tile) { return (tile % MT) * a.mt * kBM; };
  auto halves = [&](int m0) { return min(a.mt, (a.M - m0 + kBM - 1) / kBM); };

  if (warp == kRawWarp) {
    if (elect_one()) {
      int gr = 0;  // ring slots loaded so far
      bool ok = true;
      WQ_FOR_EACH_PART {
        (void)nit;  // the codes ring follows the blocks only
        const int n0 = (tile / MT) * ROWS;
        for (int r = 0; r < (C::HALFRAW ? 2 * wb : wb) && ok; ++r, ++gr) {
          const int q = gr % R;
          if (gr >= R && !wait(&sm.raw_empty[q], (gr / R - 1) & 1)) {
            ok = false;
            break;
          }
          gemm_load_raw<C, NPROJ, TALL>(tm, smem + C::OFF_RAW + q * C::RAW, n0, ub + (C::HALFRAW ? r >> 1 : r), r & 1,
                                        &sm.raw_full[2 * q + (gr / R & 1)]);
        }
      }
    }
    __syncwarp();
  } else if (warp == kProducerWarp) {
    int gs = 0;  // stages so far
    bool ok = true;
    WQ_FOR_EACH_PART {
      const int m0 = tile_m0(tile), mth = halves(m0);
      for (int it = 0; it < nit && ok; ++it, ++gs) {
        const int s = gs % SA;
        if (gs >= SA && !wait(&sm.a_empty[s], (gs / SA - 1) & 1)) {
          ok = false;
          break;
        }
        uint8_t *As = smem + C::OFF_A + s * C::AT;
        if (it < 2 * wb) {
          if (lane == 0) {
            mbar_arrive_expect_tx(&sm.a_full[s], (uint32_t)(mth * kTileBytes));
            for (int h = 0; h < mth; ++h)
              tma_load_2d(As + h * kTileBytes, &tm.act, (ub + (it >> 1)) * 128 + (it & 1) * 64, m0 + h * kBM,
                          &sm.a_full[s]);
          }
        } else {
          gemm_lora_a_stage<NPROJ>(a, As, m0, mth, it - 2 * wb, lane, &sm.a_full[s]);
        }
      }
    }
  } else if (warp == kMmaWarp) {
    if (elect_one()) {
      int gs = 0, part = 0;
      bool ok = true;
      WQ_FOR_EACH_PART {
        if (!ok) break;
        const int mth = halves(tile_m0(tile));
        // the previous part's accumulators are read
        if (part > 0 && !wait(sm.acc_empty, (part - 1) & 1)) ok = false;
        ++part;
        if (!ok) break;
        for (int it = 0; it < nit; ++it, ++gs) {
          const int sa = gs % SA, sb = gs % SB;
          if (!wait(&sm.a_full[sa], (gs / SA) & 1) || !wait(&sm.b_full[sb], (gs / SB) & 1)) {
            ok = false;
            break;
          }
          tc_fence_after();
          gemm_issue_stage<NPROJ, EXACT>(tmem, smem_addr(smem + C::OFF_A + sa * C::AT),
                                         smem_addr(smem + C::OFF_B + sb * C::BT), mth, it < 2 * wb, it == 0);
          umma_commit(&sm.a_empty[sa]);
          umma_commit(&sm.b_empty[2 * sb + (gs / SB & 1)]);
        }
        if (ok) umma_commit(sm.acc_full);  // the part's accumulators are complete
      }
    }
    __syncwarp();
  } else {
    // dequantization, then each part's epilogue; a warp that met a timeout
    // skips its work but still arrives for every part
    const int hb = warp / kDeqGroup, dt = tid & (kDeqGroup * 32 - 1);
    int gs = 0, gr = 0, part = 0;
    bool ok = true;
    WQ_FOR_EACH_PART {
      const int n0 = (tile / MT) * ROWS;
      for (int it = hb; it < nit; it += 2) {
        const int st = gs + it, s = st % SB, kr = gr + (C::HALFRAW ? it : it >> 1), q = kr % R;
        const bool wstage = it < 2 * wb;
        const int ur = kr / R, vb = st / SB - 1;  // the slots' uses waited for
        if (ok && wstage && !wait(&sm.raw_full[2 * q + (ur & 1)], (ur >> 1) & 1)) ok = false;
        if (ok && st >= SB && !wait(&sm.b_empty[2 * s + (vb & 1)], (vb >> 1) & 1)) ok = false;
        if (!ok) continue;
        uint8_t *Bs = smem + C::OFF_B + s * C::BT;
        if (wstage)
          gemm_deq_stage<BITS, NPROJ, GROUP, EXACT>(smem + C::OFF_RAW + q * C::RAW, Bs, hb, dt);
        else
          gemm_lora_b_stage<NPROJ>(a, Bs, n0, it - 2 * wb, dt);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(&sm.b_full[s]);
          if (wstage) mbar_arrive(&sm.raw_empty[q]);  // this warp's half of the block's codes is read
        }
      }
      gs += nit;
      gr += C::HALFRAW ? 2 * wb : wb;
      const bool have = ok && wait(sm.acc_full, part & 1);
      ++part;
      tc_fence_after();
      gemm_part_epilogue<BITS, NPROJ, GROUP, EXACT, TALL>(a, tmem, tile, ub, ue, U, g0, have);
      // every lane's TMEM reads are done: the next part may overwrite them
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(sm.acc_empty);
    }
  }
#undef WQ_FOR_EACH_PART

  if (*sm.abort_s) gemm_settle();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == kMmaWarp) tmem_dealloc(tmem, C::NCOLS);
}

// The split tiles of a stream-K launch of P CTAs: the parts' fp32 sums added in
// k order (their CTAs c_lo .. c_hi are consecutive), then the epilogue.  A
// thread takes one token and 16 columns of an accumulator (of gate and up):
// grid (columns / 16, halves, tiles), 128 threads a half.
template <int NPROJ, bool TALL>
__global__ void __launch_bounds__(kBM) gemm_reduce_kernel(const GemmArgs a, int U, long long W, long long P) {
  pdl_wait();
  const int tile = blockIdx.z, h = blockIdx.y, cg = blockIdx.x % (kBN / 16), p = blockIdx.x / (kBN / 16);
  const long long t0u = (long long)tile * U;
  const int c_lo = (int)(((t0u + 1) * P + W - 1) / W - 1), c_hi = (int)(((t0u + U) * P + W - 1) / W - 1);
  if (c_lo == c_hi) return;  // finished from TMEM
  const int MT = (a.M + a.mt * kBM - 1) / (a.mt * kBM);
  const int m = (tile % MT) * a.mt * kBM + h * kBM + threadIdx.x;
  const int nb = (tile / MT) * (TALL ? 2 * kBN : kBN) + p * kBN + cg * 16;
  if (m >= a.M || nb >= a.N) return;
  constexpr int SLOT = kHalves * kBM * NPROJ * kBN;
  auto sum = [&](int acc, float (&v)[16]) {
#pragma unroll
    for (int e = 0; e < 16; ++e) v[e] = 0.f;
#pragma unroll 4
    for (int cc = c_lo; cc <= c_hi; ++cc) {
      // CTA cc's part of this tile is its first (slot 0) unless the tile began inside its range
      const float4 *src = reinterpret_cast<const float4 *>(a.sk_part + ((size_t)cc * 2 + (t0u <= W * cc / P ? 0 : 1)) * SLOT) +
                          (((size_t)h * NPROJ + acc) * (kBN / 4) + cg * 4) * kBM + threadIdx.x;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 f = __ldcg(src + i * kBM);
        v[4 * i] += f.x;
        v[4 * i + 1] += f.y;
        v[4 * i + 2] += f.z;
        v[4 * i + 3] += f.w;
      }
    }
  };
  const float rs = a.rs != nullptr ? a.rs[m] : 1.f;
  float v[16];
  const size_t o = (size_t)m * a.N + nb;
  sum(p, v);
  if (NPROJ == 2 && !TALL) {
    float u[16];
    sum(1, u);
    gemm_silu16(v, u, rs);
  } else {
#pragma unroll
    for (int e = 0; e < 16; ++e) v[e] *= rs;
    const __nv_bfloat16 *res = reinterpret_cast<const __nv_bfloat16 *>(a.residual);
    if (res && (a.N & 7) == 0) {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        if (nb + 8 * i >= a.N) continue;
        const uint4 q = *reinterpret_cast<const uint4 *>(res + o + 8 * i);
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int e = 0; e < 8; ++e)
          v[8 * i + e] += __uint_as_float(e & 1 ? (w[e >> 1] & 0xffff0000u) : (w[e >> 1] << 16));
      }
    } else if (res) {
#pragma unroll
      for (int e = 0; e < 16; ++e)
        if (nb + e < a.N) v[e] += __bfloat162float(res[o + e]);
    }
  }
  const bool f32 = NPROJ == 1 && !TALL && a.out_f32;
  if (!f32 && (a.N & 7) == 0) {
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (nb + 8 * i < a.N)
        *reinterpret_cast<uint4 *>(reinterpret_cast<__nv_bfloat16 *>(a.out) + o + 8 * i) =
            make_uint4(pack_bf16(v[8 * i], v[8 * i + 1]), pack_bf16(v[8 * i + 2], v[8 * i + 3]),
                       pack_bf16(v[8 * i + 4], v[8 * i + 5]), pack_bf16(v[8 * i + 6], v[8 * i + 7]));
    return;
  }
#pragma unroll
  for (int e = 0; e < 16; ++e) {
    if (nb + e >= a.N) continue;
    if (f32)
      reinterpret_cast<float *>(a.out)[o + e] = v[e];
    else
      reinterpret_cast<__nv_bfloat16 *>(a.out)[o + e] = __float2bfloat16_rn(v[e]);
  }
}

// Per token of x [M, K] (bf16, K a multiple of 32): the binary16 copy x16
// [M][lda16] (the GEMM's A operand, zeros past K), the RMSNorm scale
// rs = 1/sqrt(mean(x^2) + eps) and, with an adapter, ta = lora_scale * x A^T
// as binary16 [M][2r] (gate rows, then up rows).
// A CTA takes 16 tokens and 16 rows of A.  The products x A^T run on m16n8k16
// bf16 MMAs (exact products, fp32 sums); the 16 warps take interleaved chunks
// of 32 features, kPrepUnroll chunks' loads in flight at a time (2, or 5 where
// the grid leaves each SM one CTA: 512 tokens of d 5120 15.8 -> 13.2 us), and
// their partial sums are added in warp order.  A lane loads 8 consecutive features of a row
// (16 bytes) and feeds features 0..3 and 4..7 of them to two k-steps in the
// slots of k 2t, 2t+1, 2t+8, 2t+9: the same permutation of k for x and A, so
// the sums are unchanged.  Every CTA sums x^2 of its tokens (row block 0
// writes rs) and converts the chunks c with c % gridDim.y == blockIdx.y.
constexpr int kPrepTok = 16, kPrepRows = 16, kPrepWarps = 16;

template <int kPrepUnroll>
__global__ void __launch_bounds__(kPrepWarps * 32) gemm_prep_kernel(const __nv_bfloat16 *x, int M, int K, int lda16,
                                                                   const __nv_bfloat16 *lora_a, int r2,
                                                                   float lora_scale, int prenorm, uint16_t *x16,
                                                                   float *rs, uint16_t *ta) {
  __shared__ float part[kPrepWarps][kPrepTok][kPrepRows + 1];
  __shared__ float ssp[kPrepWarps][kPrepTok];
  __shared__ uint32_t mxp[kPrepWarps][kPrepTok];
  __shared__ float scl[kPrepTok];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  const int m0 = blockIdx.x * kPrepTok, j0 = blockIdx.y * kPrepRows;
  const int nchunk = K / 32;
  const bool lora = r2 > 0;
  float acc[2][4];
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i >> 2][i & 3] = 0.f;
  float ss[2] = {0.f, 0.f};  // tokens g and g + 8 of the block
  uint32_t mx[2] = {0u, 0u};  // their largest |x| (bit patterns of non-negative floats order like the values)
  const auto word = [](const uint4 &v, int q) { return q == 0 ? v.x : q == 1 ? v.y : q == 2 ? v.z : v.w; };
  for (int cb = warp; cb < nchunk; cb += kPrepWarps * kPrepUnroll) {
    uint4 xa[kPrepUnroll][2], ab[kPrepUnroll][2];
#pragma unroll
    for (int u = 0; u < kPrepUnroll; ++u) {  // the loads of both chunks first
      const int c = cb + u * kPrepWarps, k = c * 32 + 8 * t;
      const bool in = c < nchunk;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int m = m0 + g + 8 * i;
        xa[u][i] = in && m < M ? __ldg(reinterpret_cast<const uint4 *>(x + (size_t)m * K + k))
                               : make_uint4(0u, 0u, 0u, 0u);
      }
#pragma unroll
      for (int n = 0; n < 2; ++n) {
        const int j = j0 + 8 * n + g;
        ab[u][n] = in && lora && j < r2 ? __ldg(reinterpret_cast<const uint4 *>(lora_a + (size_t)j * K + k))
                                        : make_uint4(0u, 0u, 0u, 0u);
      }
    }
#pragma unroll
    for (int u = 0; u < kPrepUnroll; ++u) {
      const int c = cb + u * kPrepWarps;
      if (c >= nchunk) break;  // the same for the whole warp
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const uint32_t w[4] = {xa[u][i].x, xa[u][i].y, xa[u][i].z, xa[u][i].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float lo = __uint_as_float(w[e] << 16), hi = __uint_as_float(w[e] & 0xffff0000u);
          ss[i] = fmaf(lo, lo, ss[i]);
          ss[i] = fmaf(hi, hi, ss[i]);
          mx[i] = max(mx[i], max((w[e] << 16) & 0x7fffffffu, w[e] & 0x7fff0000u));
        }
      }
      if (lora) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          // rows g, g + 8 of the m-tile are tokens g (xa[u][0]) and g + 8 (xa[u][1])
          const uint32_t af[4] = {word(xa[u][0], 2 * h), word(xa[u][1], 2 * h), word(xa[u][0], 2 * h + 1),
                                  word(xa[u][1], 2 * h + 1)};
#pragma unroll
          for (int nt = 0; nt < 2; ++nt)
            mma_bf16_16816(acc[nt], af, word(ab[u][nt], 2 * h), word(ab[u][nt], 2 * h + 1));
        }
      }
    }
  }
  // sums of squares: the quad's lanes hold disjoint features of the same tokens
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    ss[i] += __shfl_xor_sync(0xffffffffu, ss[i], 1);
    ss[i] += __shfl_xor_sync(0xffffffffu, ss[i], 2);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    mx[i] = max(mx[i], __shfl_xor_sync(0xffffffffu, mx[i], 1));
    mx[i] = max(mx[i], __shfl_xor_sync(0xffffffffu, mx[i], 2));
  }
  if (t == 0) {
    ssp[warp][g] = ss[0];
    ssp[warp][g + 8] = ss[1];
    mxp[warp][g] = mx[0];
    mxp[warp][g + 8] = mx[1];
  }
  if (lora) {
    // accumulator (row, col) of n-tile nt: rows g / g + 8, cols 2t, 2t+1
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
      part[warp][g][8 * nt + 2 * t] = acc[nt][0];
      part[warp][g][8 * nt + 2 * t + 1] = acc[nt][1];
      part[warp][g + 8][8 * nt + 2 * t] = acc[nt][2];
      part[warp][g + 8][8 * nt + 2 * t + 1] = acc[nt][3];
    }
  }
  __syncthreads();
  // Per token an exact power of two 2^e puts its largest |x| in [2^4, 2^5):
  // the binary16 copies of x and of t = lora_scale x A^T are taken of the
  // values times 2^e (no overflow: 2^11 below the binary16 maximum even for
  // |t| up to 2^10 |x|; every element within 2^-22 of the largest stays
  // exact), and the epilogue multiplies the fp32 sums by rs 2^-e, which
  // undoes it exactly.
  if (tid < kPrepTok) {
    uint32_t mxb = 0u;
    for (int w = 0; w < kPrepWarps; ++w) mxb = max(mxb, mxp[w][tid]);
    const int be = (int)(mxb >> 23);
    const int e = mxb == 0u || be >= 255 ? 0 : max(-100, min(100, 131 - be));
    scl[tid] = __int_as_float((e + 127) << 23);
    if (blockIdx.y == 0 && m0 + tid < M) {
      float tot = 0.f;
      for (int w = 0; w < kPrepWarps; ++w) tot += ssp[w][tid];
      const float r = prenorm ? __fdiv_rn(1.f, __fsqrt_rn(__fadd_rn(__fdiv_rn(tot, (float)K), kRmsEps))) : 1.f;
      rs[m0 + tid] = r * __int_as_float((127 - e) << 23);
    }
  }
  __syncthreads();
  // the binary16 copy of x (2^e x): this CTA's chunks c = blockIdx.y + cc
  // gridDim.y, 16 bytes an item, four loads in flight a thread
  {
    const int ncc = (nchunk - (int)blockIdx.y + (int)gridDim.y - 1) / (int)gridDim.y;
    const int items = kPrepTok * ncc * 4;
    constexpr int NT = kPrepWarps * 32;
    for (int i0 = tid; i0 < items; i0 += 4 * NT) {
      uint4 v[4];
      int tl[4];
      size_t dst[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = i0 + u * NT;
        tl[u] = i / (ncc * 4);
        const int rem = i % (ncc * 4), c = (int)blockIdx.y + (rem / 4) * (int)gridDim.y, k = c * 32 + 8 * (rem % 4);
        const int m = m0 + tl[u];
        const bool ok = i < items && m < M;
        dst[u] = ok ? (size_t)m * lda16 + k : ~(size_t)0;
        v[u] = ok ? __ldg(reinterpret_cast<const uint4 *>(x + (size_t)m * K + k)) : make_uint4(0u, 0u, 0u, 0u);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (dst[u] == ~(size_t)0) continue;
        const uint32_t w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
        const float sc = scl[tl[u]];
        uint32_t o[4];
#pragma unroll
        for (int e = 0; e < 4; ++e)
          o[e] = h2bits(__floats2half2_rn(__uint_as_float(w[e] << 16) * sc, __uint_as_float(w[e] & 0xffff0000u) * sc));
        *reinterpret_cast<uint4 *>(x16 + dst[u]) = make_uint4(o[0], o[1], o[2], o[3]);
      }
    }
  }
  if (lora) {
    for (int o = tid; o < kPrepTok * kPrepRows; o += kPrepWarps * 32) {
      const int tl = o / kPrepRows, jl = o % kPrepRows;
      const int m = m0 + tl, j = j0 + jl;
      if (m >= M || j >= r2) continue;
      float v = 0.f;
      for (int w = 0; w < kPrepWarps; ++w) v += part[w][tl][jl];
      ta[(size_t)m * r2 + j] = __half_as_ushort(__float2half_rn(lora_scale * v * scl[tl]));
    }
  }
  // zeros past K
  if (blockIdx.y == 0)
    for (int i = tid; i < kPrepTok * (lda16 - K); i += kPrepWarps * 32) {
      const int tl = i / (lda16 - K), k = K + i % (lda16 - K);
      if (m0 + tl < M) x16[(size_t)(m0 + tl) * lda16 + k] = 0;
    }
}

// bf16 [M, K] -> binary16 [M, lda16] (zero padded), the down GEMM's A
// operand, one CTA per token: an exact power of two 2^e puts the token's
// largest |x| in [2^4, 2^5) (no overflow, every element within 2^-22 of the
// largest exact); sx[m] = 2^-e, by which the epilogue multiplies the sums.
// K a multiple of 8.
__global__ void __launch_bounds__(256) to_f16_kernel(const __nv_bfloat16 *x, int M, int K, int lda16, uint16_t *x16,
                                                     float *sx) {
  __shared__ uint32_t wmax[8];
  const int m = blockIdx.x, tid = threadIdx.x;
  if (m >= M) return;
  const uint4 *row = reinterpret_cast<const uint4 *>(x + (size_t)m * K);
  const int n8 = K / 8;
  uint32_t mx = 0u;
  for (int i = tid; i < n8; i += blockDim.x) {
    const uint4 v = __ldg(row + i);
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) mx = max(mx, max((w[e] << 16) & 0x7fffffffu, w[e] & 0x7fff0000u));
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  if ((tid & 31) == 0) wmax[tid >> 5] = mx;
  __syncthreads();
  mx = 0u;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) mx = max(mx, wmax[w]);
  const int be = (int)(mx >> 23);
  const int e = mx == 0u || be >= 255 ? 0 : max(-100, min(100, 131 - be));
  const float sc = __int_as_float((e + 127) << 23);
  if (tid == 0) sx[m] = __int_as_float((127 - e) << 23);
  for (int i = tid; i < n8; i += blockDim.x) {
    const uint4 v = __ldg(row + i);
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    uint32_t o[4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
      o[q] = h2bits(__floats2half2_rn(__uint_as_float(w[q] << 16) * sc, __uint_as_float(w[q] & 0xffff0000u) * sc));
    *reinterpret_cast<uint4 *>(x16 + (size_t)m * lda16 + 8 * i) = make_uint4(o[0], o[1], o[2], o[3]);
  }
  for (int k = K + tid; k < lda16; k += blockDim.x) x16[(size_t)m * lda16 + k] = 0;
}

// cuTensorMapEncodeTiled from the driver (looked up once).
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static std::once_flag once;
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  std::call_once(once, [] {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

// Tensor maps of a launch (zero fill outside every tensor):
//   activations [M][lda] binary16, boxes of 64 features x 128 tokens;
//   codes [RT][KB * BPK / 128][128 B], boxes of a 2-bit block or half a 4-bit one of 8 row tiles;
//   scales/zeros [RT][KB * GPB][64 B], boxes of the groups that those codes have.
cudaError_t make_maps(const GemmArgs &a, int nproj, int bits, GemmMaps *m) {
  PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
  if (!fn) return cudaErrorNotSupported;
  const cuuint32_t e1[3] = {1, 1, 1};
  {
    const cuuint64_t dims[2] = {(cuuint64_t)a.K, (cuuint64_t)a.M};
    const cuuint64_t strides[1] = {(cuuint64_t)a.lda * 2};
    const cuuint32_t box[2] = {64, (cuuint32_t)kBM};
    if (fn(&m->act, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<uint16_t *>(a.act), dims, strides, box, e1,
           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cudaErrorInvalidValue;
  }
  const cuuint64_t RT = (cuuint64_t)(a.N + 15) / 16, KB = (cuuint64_t)(a.K + 127) / 128;
  const cuuint64_t bpk = bits == 2 ? 512 : 1024, gpb = 128 / a.group;
  for (int p = 0; p < 2; ++p) {
    const int src = p < nproj ? p : 0;  // unused second map of the down kernel: a copy of the first
    {
      const cuuint64_t dims[3] = {128, KB * bpk / 128, RT};
      const cuuint64_t strides[2] = {128, KB * bpk};
      const cuuint32_t box[3] = {128, 4, 8};  // a 2-bit block or half a 4-bit block
      if (fn(&m->codes[p], CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<uint32_t *>(a.codes[src]), dims, strides, box, e1,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    }
    {
      const cuuint64_t dims[3] = {64, KB * gpb, RT};
      const cuuint64_t strides[2] = {64, KB * gpb * 64};
      const cuuint32_t box[3] = {64, (cuuint32_t)(bits == 4 && gpb > 1 ? gpb / 2 : gpb), 8};
      if (fn(&m->meta[p], CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<uint16_t *>(a.meta[src]), dims, strides, box, e1,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    }
  }
  return cudaSuccess;
}

cudaError_t num_sms_cached(int *sms) {
  static int cached[64] = {0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (cached[dev] == 0 && (e = cudaDeviceGetAttribute(&cached[dev], cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
    return e;
  *sms = cached[dev];
  return cudaSuccess;
}

// Work split of a launch.  A CTA takes two token halves (each weight
// dequantized once for 256 tokens) whenever there are more than 128 tokens.
// Tiles are mt * 128 tokens x 128 rows (down may take 256, below), U work units
// each (128-feature blocks, plus one for the LoRA stages).  Stream-K -- P CTAs
// (one per SM at most, 4 units each at least) dividing the T * U units evenly --
// where it shortens the critical path by more than its cost in units: the split
// tiles' parts and their reduction (~8; measured d 2560 down at 2048 tokens 137
// -> 103 us, d 5120 at 1500 228 -> 216), and for gate/up, whose parts are twice
// as large, a main loop about a tenth slower (d 4096 at 700 tokens 159 -> 152
// with it, at 512 tokens 110 -> 116, d 5120 at 3001 658 -> 695; d 2560 at 65
// tokens, half the SMs without it, 39 -> 34).  Where gate/up tiles of 256 tokens
// fill one wave at most, the parts of two halves weigh more (~15; at 160 tokens
// without it -> with it d 2560 x inter 9728 39.1 -> 41.1, d 1600 x 4352 29.9 ->
// 37.5, but d 4096 x 6144 54.9 -> 51.1, d 5120 x 2048 80 -> 52).  One CTA per
// tile otherwise.
struct GemmSched {
  int mt, T, U, P;
  bool sk;
};
GemmSched gemm_schedule(int M, int N, int K, int nproj, int r, int sms, int rows = kBN) {
  GemmSched g;
  g.mt = M > kBM ? 2 : 1;
  g.T = (M + g.mt * kBM - 1) / (g.mt * kBM) * ((N + rows - 1) / rows);
  g.U = (K + 127) / 128 + (nproj == 2 && r > 0 ? 1 : 0);
  const long long W = (long long)g.T * g.U;
  const long long waves = (g.T + sms - 1) / sms, P = std::max(1LL, std::min((long long)sms, W / 4));
  const double share = (double)W / P;  // units a CTA
  const double cost = nproj == 2 ? std::max(14., 1.25 * share + (g.mt == 2 && waves == 1 ? 15 : 6)) : share + 8;
  g.sk = W >= 8 && waves * g.U > cost;
  g.P = g.sk ? (int)P : g.T;
  return g;
}

// Down launches of more than 128 tokens take tiles of 256 rows (TALL: one
// N = 256 MMA over two 128-row tiles reads 96 bytes a clock of the 128 that
// shared memory gives, an N = 128 one all 128) where they make at least
// kTallTiles of them, so that few CTAs share a split tile (us, 128-row vs
// 256-row: d 2560 at 3001 tokens 200 -> 144, d 5120 at 512 tokens 141 -> 87;
// but d 2560 at 256 tokens, 10 tiles, 37 vs 44, and at 512, 20 tiles, 46 vs 48).
constexpr int kTallTiles = 30;
bool gemm_tall(int M, int N) {
  return M > kBM && (long long)((M + 2 * kBM - 1) / (2 * kBM)) * ((N + 2 * kBN - 1) / (2 * kBN)) >= kTallTiles;
}

template <int BITS, int NPROJ, int GROUP, bool EXACT, bool TALL>
cudaError_t launch_gemm_t(const GemmArgs &a, cudaStream_t s) {
  using C = GemmCfg<BITS, NPROJ, GROUP, EXACT>;
  constexpr int ROWS = TALL ? 2 * kBN : kBN;
  auto tile_kern = qgemm_tile_kernel<BITS, NPROJ, GROUP, EXACT, TALL>;
  auto sk_kern = qgemm_sk_kernel<BITS, NPROJ, GROUP, EXACT, TALL>;
  cudaError_t e = cudaFuncSetAttribute(tile_kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(sk_kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
  if (e != cudaSuccess) return e;
  GemmMaps maps;
  if ((e = make_maps(a, TALL ? 1 : NPROJ, BITS, &maps)) != cudaSuccess) return e;
  int sms = 0;
  if ((e = num_sms_cached(&sms)) != cudaSuccess) return e;
  const GemmSched g = gemm_schedule(a.M, a.N, a.K, TALL ? 1 : NPROJ, a.r, sms, ROWS);
  GemmArgs ka = a;
  ka.mt = g.mt;
  if (g.sk && a.sk_part) {
    sk_kern<<<g.P, kGemmThreads, C::SMEM, s>>>(ka, maps);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((TALL ? 2 : 1) * kBN / 16, g.mt, g.T);
    cfg.blockDim = dim3(kBM);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, gemm_reduce_kernel<NPROJ, TALL>, ka, g.U, (long long)g.T * g.U, (long long)g.P);
  } else {
    ka.sk_part = nullptr;
    tile_kern<<<dim3((a.M + g.mt * kBM - 1) / (g.mt * kBM), (a.N + ROWS - 1) / ROWS), kGemmThreads, C::SMEM, s>>>(ka, maps);
  }
  return cudaGetLastError();
}

template <int BITS, int NPROJ, bool EXACT, bool TALL = false>
cudaError_t launch_gemm_g(const GemmArgs &a, cudaStream_t s) {
  switch (a.group) {
    case 32: return launch_gemm_t<BITS, NPROJ, 32, EXACT, TALL>(a, s);
    case 64: return launch_gemm_t<BITS, NPROJ, 64, EXACT, TALL>(a, s);
    default: return launch_gemm_t<BITS, NPROJ, 128, EXACT, TALL>(a, s);
  }
}

}  // namespace

cudaError_t launch_gemm(GemvKind kind, const GemmArgs &a, cudaStream_t s) {
  if (a.M <= 0) return cudaSuccess;
  switch (kind) {
    case kGateUpW2: return launch_gemm_g<2, 2, false>(a, s);
    case kGateUpW4: return launch_gemm_g<4, 2, false>(a, s);
    default:
      if (a.out_f32) return launch_gemm_g<4, 1, true>(a, s);
      return gemm_tall(a.M, a.N) ? launch_gemm_g<4, 2, false, true>(a, s) : launch_gemm_g<4, 1, false>(a, s);
  }
}

size_t gemm_scratch_floats(int M, int N, int K, int nproj, int num_sms) {
  if (M <= 0 || N <= 0 || K <= 0 || num_sms <= 0) return 0;
  const GemmSched g = gemm_schedule(M, N, K, nproj, kMaxRank, num_sms);
  size_t most = g.sk ? (size_t)2 * g.P * kHalves * kBM * nproj * kBN : 0;
  if (nproj == 1 && gemm_tall(M, N)) {
    const GemmSched t = gemm_schedule(M, N, K, 1, 0, num_sms, 2 * kBN);
    if (t.sk) most = std::max(most, (size_t)2 * t.P * kHalves * kBM * 2 * kBN);
  }
  return most;
}

cudaError_t launch_gemm_prep(const void *x, int M, int K, int lda16, const void *lora_a, int r2, float lora_scale,
                             int prenorm, uint16_t *x16, float *rs, uint16_t *ta, cudaStream_t s) {
  if (M <= 0) return cudaSuccess;
  if (K % 32 != 0 || lda16 < K) return cudaErrorInvalidValue;
  const dim3 grid((M + kPrepTok - 1) / kPrepTok, r2 > 0 ? (r2 + kPrepRows - 1) / kPrepRows : 1);
  int sms = 0;
  cudaError_t e = num_sms_cached(&sms);
  if (e != cudaSuccess) return e;
  auto kern = (long long)grid.x * grid.y <= sms ? gemm_prep_kernel<5> : gemm_prep_kernel<2>;
  kern<<<grid, kPrepWarps * 32, 0, s>>>(reinterpret_cast<const __nv_bfloat16 *>(x), M, K, lda16,
                                        reinterpret_cast<const __nv_bfloat16 *>(lora_a), r2, lora_scale, prenorm, x16, rs,
                                        ta);
  return cudaGetLastError();
}
cudaError_t launch_to_f16(const void *x, int M, int K, int lda16, uint16_t *x16, float *sx, cudaStream_t s) {
  if (M <= 0) return cudaSuccess;
  if (K % 8 != 0 || lda16 < K) return cudaErrorInvalidValue;
  to_f16_kernel<<<M, 256, 0, s>>>(reinterpret_cast<const __nv_bfloat16 *>(x), M, K, lda16, x16, sx);
  return cudaGetLastError();
}

cudaError_t read_gemm_status(int *status) {
  int v = 0;
  cudaError_t e = cudaMemcpyFromSymbol(&v, g_gemm_status, sizeof(int));
  if (e != cudaSuccess) return e;
  const int zero = 0;
  e = cudaMemcpyToSymbol(g_gemm_status, &zero, sizeof(int));
  *status = v;
  return e;
}

}  // namespace wq
