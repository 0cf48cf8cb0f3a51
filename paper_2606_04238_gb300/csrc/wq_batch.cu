// wq_batch.cu -- the batched-decode dequant-GEMM's inputs (activation panel,
// RMSNorm scales, LoRA-A products) and its dispatch.
#include "wq_batch.cuh"

namespace wq {
namespace {

constexpr int kPrepThreads = 512, kPrepWarps = kPrepThreads / 32;
constexpr int kPrepUnroll = 5;  // 32-feature chunks of a warp in flight

__device__ __forceinline__ uint32_t word4(const uint4 &v, int q) { return q == 0 ? v.x : q == 1 ? v.y : q == 2 ? v.z : v.w; }

// CTAs 0 .. nt * row_tiles - 1 (row_tiles > 0): 8 tokens x 16 rows of A_cat
// over all features: t = lora_scale * x A^T on bf16 mma.sync (exact products,
// fp32 sums), stored as two bf16 parts in the gate/up launch's fragment order;
// row tile 0 also the tokens' RMSNorm scales.  The 16 warps take interleaved
// chunks of 32 features and their sums are added in warp order.  A lane loads
// 8 consecutive features of a row and feeds them to two k-steps in the same
// permuted order for x and A.  The remaining CTAs convert x into the panel,
// one (128-feature block, token) a warp.  The rows of A are loaded before the
// wait on the launch that wrote x.
__global__ void __launch_bounds__(kPrepThreads) batch_prep_kernel(const __nv_bfloat16 *x, int M, int K, int wide,
                                                                 int group, const __nv_bfloat16 *lora_a, int r,
                                                                 float lora_scale, uint8_t *panel, float *rs,
                                                                 uint8_t *tfrag, int nt_total, int row_tiles) {
  __shared__ float part[kPrepWarps][16][9];
  __shared__ float ssp[kPrepWarps][8];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  pdl_launch_dependents();
  if ((int)blockIdx.x >= nt_total * row_tiles) {
    pdl_wait();
    const int item = ((int)blockIdx.x - nt_total * row_tiles) * kPrepWarps + warp;
    const int kb = item / (nt_total * 8), m = item - kb * (nt_total * 8);
    if (kb >= (K + 127) / 128) return;
    const int k = kb * 128 + 4 * lane;
    uint2 raw = make_uint2(0u, 0u);
    if (m < M && k < K) raw = ldg_cg64(x + (size_t)m * K + k);
    const float f[4] = {__uint_as_float(raw.x << 16), __uint_as_float(raw.x & 0xffff0000u),
                        __uint_as_float(raw.y << 16), __uint_as_float(raw.y & 0xffff0000u)};
    batch_panel_token(panel + (size_t)kb * batch_rec_bytes(nt_total, group), nt_total, group, wide != 0, m, lane, f);
    return;
  }
  const int jt = blockIdx.x / nt_total, nt = blockIdx.x % nt_total;
  const int r2 = tfrag != nullptr ? 2 * r : 0, j0 = jt * 16, m = nt * 8 + g;
  const int nchunk = K / 32;
  float acc[4] = {0.f, 0.f, 0.f, 0.f}, ss = 0.f;
  for (int cb = warp, round = 0; cb < nchunk; cb += kPrepWarps * kPrepUnroll, ++round) {
    uint4 av[kPrepUnroll][2], xv[kPrepUnroll];
#pragma unroll
    for (int u = 0; u < kPrepUnroll; ++u) {
      const int c = cb + u * kPrepWarps, k = c * 32 + 8 * t;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int j = j0 + g + 8 * i;
        av[u][i] = c < nchunk && j < r2 ? __ldg(reinterpret_cast<const uint4 *>(lora_a + (size_t)j * K + k))
                                        : make_uint4(0u, 0u, 0u, 0u);
      }
    }
    if (round == 0) pdl_wait();
#pragma unroll
    for (int u = 0; u < kPrepUnroll; ++u) {
      const int c = cb + u * kPrepWarps, k = c * 32 + 8 * t;
      xv[u] = c < nchunk && m < M ? ldg_cg128(x + (size_t)m * K + k) : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int u = 0; u < kPrepUnroll; ++u) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const uint32_t w = word4(xv[u], e);
        const float lo = __uint_as_float(w << 16), hi = __uint_as_float(w & 0xffff0000u);
        ss = fmaf(lo, lo, ss);
        ss = fmaf(hi, hi, ss);
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint32_t af[4] = {word4(av[u][0], 2 * h), word4(av[u][1], 2 * h), word4(av[u][0], 2 * h + 1),
                                word4(av[u][1], 2 * h + 1)};
        mma_bf16_16816(acc, af, word4(xv[u], 2 * h), word4(xv[u], 2 * h + 1));
      }
    }
  }
  if (warp >= nchunk) pdl_wait();
  ss += __shfl_xor_sync(0xffffffffu, ss, 1);
  ss += __shfl_xor_sync(0xffffffffu, ss, 2);
  if (t == 0) ssp[warp][g] = ss;
  part[warp][g][2 * t] = acc[0];
  part[warp][g][2 * t + 1] = acc[1];
  part[warp][g + 8][2 * t] = acc[2];
  part[warp][g + 8][2 * t + 1] = acc[3];
  __syncthreads();
  if (tid < 128 && r2 > 0) {
    const int jl = tid >> 3, ml = tid & 7, j = j0 + jl;
    float v = 0.f;
    for (int w = 0; w < kPrepWarps; ++w) v += part[w][jl][ml];
    if (j < r2) {
      v *= lora_scale;
      const int p = j >= r ? 1 : 0, rho = j - p * r, RK = (r + 15) / 16, c = rho & 15;
      const size_t at = ((((size_t)p * RK + (rho >> 4)) * nt_total + nt) * 32 + 4 * ml + ((c & 7) >> 1)) * 16 +
                        (c >> 3) * 4 + (c & 1) * 2;
      const __nv_bfloat16 hi = __float2bfloat16_rn(v), lo = __float2bfloat16_rn(v - __bfloat162float(hi));
      *reinterpret_cast<__nv_bfloat16 *>(tfrag + at) = hi;
      *reinterpret_cast<__nv_bfloat16 *>(tfrag + at + 8) = lo;
    }
  }
  // ranks r .. 16 RK - 1 multiply zero rows of B: zeros, not leftovers
  if (jt == 0 && r2 > 0 && (r & 15) != 0 && tid >= 128 && tid < 256) {
    const int i = tid - 128, p = i >> 6, c = 8 + ((i >> 3) & 7), ml = i & 7, RK = (r + 15) / 16;
    const size_t at = ((((size_t)p * RK + RK - 1) * nt_total + nt) * 32 + 4 * ml + ((c & 7) >> 1)) * 16 + 4 + (c & 1) * 2;
    *reinterpret_cast<uint16_t *>(tfrag + at) = 0;
    *reinterpret_cast<uint16_t *>(tfrag + at + 8) = 0;
  }
  if (jt == 0 && rs != nullptr && tid >= 256 && tid < 264) {
    const int ml = tid - 256;
    float tot = 0.f;
    for (int w = 0; w < kPrepWarps; ++w) tot += ssp[w][ml];
    if (nt * 8 + ml < M)
      rs[nt * 8 + ml] = __fdiv_rn(1.f, __fsqrt_rn(__fadd_rn(__fdiv_rn(tot, (float)K), kRmsEps)));
  }
}

cudaError_t batch_sms(int *sms) {
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

}  // namespace

cudaError_t launch_batch_prep(const void *x, int M, int K, int bits, int group, const void *lora_a, int r,
                              float lora_scale, uint8_t *panel, float *rs, uint8_t *tfrag, cudaStream_t s) {
  if (M <= 0 || M > kBatchMaxTokens || K <= 0 || K % 32 != 0) return cudaErrorInvalidValue;
  const int nt = batch_nt(M), KB = (K + 127) / 128;
  const bool lora = tfrag != nullptr && r > 0;
  const int row_tiles = lora ? (2 * r + 15) / 16 : rs != nullptr ? 1 : 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nt * row_tiles + (KB * nt * 8 + kPrepWarps - 1) / kPrepWarps);
  cfg.blockDim = dim3(kPrepThreads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, batch_prep_kernel, reinterpret_cast<const __nv_bfloat16 *>(x), M, K,
                            bits == 4 ? 1 : 0, group, reinterpret_cast<const __nv_bfloat16 *>(lora_a), r, lora_scale,
                            panel, rs, lora ? tfrag : (uint8_t *)nullptr, nt, row_tiles);
}

cudaError_t launch_batch(GemvKind kind, const BatchArgs &a, cudaStream_t s) {
  if (a.M <= 0 || a.M > kBatchMaxTokens) return cudaErrorInvalidValue;
  int sms = 0;
  cudaError_t e = batch_sms(&sms);
  if (e != cudaSuccess) return e;
  const long long W = (long long)((a.N + kBatchRows - 1) / kBatchRows) * ((a.K + 127) / 128);
  const int nt = batch_nt(a.M), ctas = (int)std::max(1LL, std::min((long long)sms, W / 2));
  switch (kind) {
    case kGateUpW2: return launch_batch_gu2(a, nt, ctas, s);
    case kGateUpW3: return launch_batch_gu3(a, nt, ctas, s);
    case kGateUpW4: return launch_batch_gu4(a, nt, ctas, s);
    case kDownW4: return launch_batch_dn4(a, nt, ctas, s);
  }
  return cudaErrorInvalidValue;
}

// Two parts a CTA: 8 (gate/up) or 4 (down) warps x 2 tiles x NT x 32 float4s.
size_t batch_scratch_floats(int M, int nproj, int num_sms) {
  return (size_t)num_sms * 2 * (nproj == 2 ? 8 : 4) * 2 * batch_nt(M) * 32 * 4;
}

size_t batch_tfrag_bytes(int M, int r) { return (size_t)2 * ((r + 15) / 16) * batch_nt(M) * 512; }

cudaError_t read_batch_status(int *status) {
  cudaError_t (*const read[4])(int *) = {read_batch_status_gu2, read_batch_status_gu3, read_batch_status_gu4,
                                         read_batch_status_dn4};
  *status = 0;
  for (auto fn : read) {
    int v = 0;
    cudaError_t e = fn(&v);
    if (e != cudaSuccess) return e;
    if (*status == 0) *status = v;
  }
  return cudaSuccess;
}

}  // namespace wq
