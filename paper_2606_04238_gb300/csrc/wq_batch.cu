// wq_batch.cu -- the batched-decode dequant-GEMM's inputs (activation panel,
// RMSNorm scales, LoRA-A products), the grouping of a mixture of experts'
// slots by expert, and the dispatch.
//
// Grouped experts: the slots kernel reads an expert's weights once for every
// token that selects it; grouped, once for up to 8 nt tokens (32 tokens of the
// GPT-OSS-20B shape, top 4 of 32: 494 -> 127 us a block, of which gate/up ~70
// and down ~40; its 334 MB of packed experts take 49 us at the copy rate).
#include "wq_batch.cuh"
#include "wq_route.cuh"

namespace wq {
namespace {

constexpr int kPrepThreads = 512, kPrepWarps = kPrepThreads / 32;
constexpr int kPrepUnroll = 5;  // 32-feature chunks of a warp in flight

__device__ __forceinline__ uint32_t word4(const uint4 &v, int q) { return q == 0 ? v.x : q == 1 ? v.y : q == 2 ? v.z : v.w; }

// CTAs 0 .. nt * row_tiles - 1 (row_tiles > 0): 8 tokens x 16 rows of A_cat
// over all features: t = lora_scale * x A^T on bf16 mma.sync (exact products,
// fp32 sums), stored as three bf16 parts in the gate/up launch's fragment order;
// row tile 0 also the tokens' RMSNorm scales.  The 16 warps take interleaved
// chunks of 32 features and their sums are added in warp order.  A lane loads
// 8 consecutive features of a row and feeds them to two k-steps in the same
// permuted order for x and A.  The remaining CTAs convert x into the panel,
// one (128-feature block, token) a warp, and zero the arrival counters of the
// launches that follow.  The rows of A are loaded before the
// wait on the launch that wrote x.
// ROUTED: the same for every segment of the route (nt_total token tiles a
// segment, max_segs segments at most); the segment's tokens are gathered and
// A_cat is the expert's.  The launch waits first: its tables come from the
// previous launch.
template <bool ROUTED>
__global__ void __launch_bounds__(kPrepThreads) batch_prep_kernel(const __nv_bfloat16 *x, int M, int K, int wide,
                                                                 int group, const __nv_bfloat16 *lora_a, int r,
                                                                 float lora_scale, uint8_t *panel, float *rs,
                                                                 uint8_t *tfrag, unsigned *cnt, int n_cnt,
                                                                 int nt_total, int row_tiles,
                                                                 const BatchRoute *route, int top_k, int max_segs) {
  __shared__ float part[kPrepWarps][16][9];
  __shared__ float ssp[kPrepWarps][8];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  if (ROUTED) pdl_wait();
  pdl_launch_dependents();
  const int nsum = nt_total * row_tiles * (ROUTED ? max_segs : 1);
  // x row of the segment's token ml, or -1
  auto xrow = [&](const int4 &sg, int ml) -> int {
    if (!ROUTED) return ml < M ? ml : -1;
    return ml < sg.y ? __ldcg(&route->list[sg.z + ml]) / top_k : -1;
  };
  if ((int)blockIdx.x >= nsum) {
    if (!ROUTED) pdl_wait();
    for (int i = ((int)blockIdx.x - nsum) * kPrepThreads + tid; i < n_cnt; i += ((int)gridDim.x - nsum) * kPrepThreads)
      cnt[i] = 0;
    int item = ((int)blockIdx.x - nsum) * kPrepWarps + warp;
    const int KB = (K + 127) / 128, per = KB * nt_total * 8;
    int4 sg = make_int4(0, M, 0, 0);
    if (ROUTED) {
      const int seg = item / per;
      if (seg >= __ldcg(&route->n_segs)) return;
      sg = __ldcg(&route->seg[seg]);
      panel += (size_t)seg * KB * batch_rec_bytes(nt_total, group);
      item -= seg * per;
    }
    const int kb = item / (nt_total * 8), m = item - kb * (nt_total * 8);
    if (kb >= KB) return;
    const int k = kb * 128 + 4 * lane, row = xrow(sg, m);
    uint2 raw = make_uint2(0u, 0u);
    if (row >= 0 && k < K) raw = ldg_cg64(x + (size_t)row * K + k);
    const float f[4] = {__uint_as_float(raw.x << 16), __uint_as_float(raw.x & 0xffff0000u),
                        __uint_as_float(raw.y << 16), __uint_as_float(raw.y & 0xffff0000u)};
    batch_panel_token(panel + (size_t)kb * batch_rec_bytes(nt_total, group), nt_total, group, wide != 0, m, lane, f);
    return;
  }
  const int seg = ROUTED ? blockIdx.x / (nt_total * row_tiles) : 0, cta = blockIdx.x - seg * nt_total * row_tiles;
  const int jt = cta / nt_total, nt = cta % nt_total;
  const int r2 = tfrag != nullptr ? 2 * r : 0, j0 = jt * 16;
  int4 sg = make_int4(0, M, 0, 0);
  if (ROUTED) {
    if (seg >= __ldcg(&route->n_segs)) return;
    sg = __ldcg(&route->seg[seg]);
    if (r2 > 0) lora_a += (size_t)sg.x * r2 * K, tfrag += (size_t)seg * 2 * ((r + 15) / 16) * nt_total * kTfragBytes;
    if (rs != nullptr) rs += seg * nt_total * 8;
  }
  const int row = xrow(sg, nt * 8 + g);
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
    if (!ROUTED && round == 0) pdl_wait();
#pragma unroll
    for (int u = 0; u < kPrepUnroll; ++u) {
      const int c = cb + u * kPrepWarps, k = c * 32 + 8 * t;
      xv[u] = c < nchunk && row >= 0 ? ldg_cg128(x + (size_t)row * K + k) : make_uint4(0u, 0u, 0u, 0u);
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
  if (!ROUTED && warp >= nchunk) pdl_wait();
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
      uint8_t *frag = tfrag + (((size_t)p * RK + (rho >> 4)) * nt_total + nt) * kTfragBytes;
      const int ln = 4 * ml + ((c & 7) >> 1), e = (c >> 3) * 4 + (c & 1) * 2;
      const __nv_bfloat16 hi = __float2bfloat16_rn(v);
      const float rest = v - __bfloat162float(hi);
      const __nv_bfloat16 mid = __float2bfloat16_rn(rest);
      *reinterpret_cast<__nv_bfloat16 *>(frag + ln * 16 + e) = hi;
      *reinterpret_cast<__nv_bfloat16 *>(frag + ln * 16 + 8 + e) = mid;
      *reinterpret_cast<__nv_bfloat16 *>(frag + 512 + ln * 8 + e) = __float2bfloat16_rn(rest - __bfloat162float(mid));
    }
  }
  // ranks r .. 16 RK - 1 multiply zero rows of B: zeros, not leftovers
  if (jt == 0 && r2 > 0 && (r & 15) != 0 && tid >= 128 && tid < 256) {
    const int i = tid - 128, p = i >> 6, c = 8 + ((i >> 3) & 7), ml = i & 7, RK = (r + 15) / 16;
    uint8_t *frag = tfrag + (((size_t)p * RK + RK - 1) * nt_total + nt) * kTfragBytes;
    const int ln = 4 * ml + ((c & 7) >> 1), e = 4 + (c & 1) * 2;
    *reinterpret_cast<uint16_t *>(frag + ln * 16 + e) = 0;
    *reinterpret_cast<uint16_t *>(frag + ln * 16 + 8 + e) = 0;
    *reinterpret_cast<uint16_t *>(frag + 512 + ln * 8 + e) = 0;
  }
  if (jt == 0 && rs != nullptr && tid >= 256 && tid < 264) {
    const int ml = tid - 256;
    float tot = 0.f;
    for (int w = 0; w < kPrepWarps; ++w) tot += ssp[w][ml];
    if (nt * 8 + ml < sg.y)
      rs[nt * 8 + ml] = __fdiv_rn(1.f, __fsqrt_rn(__fadd_rn(__fdiv_rn(tot, (float)K), kRmsEps)));
  }
}

constexpr int kRouteThreads = 1024;

// One CTA.  Warp t: the top_k experts of token t by logit and the softmax of
// the selected logits (fp32, the largest subtracted).  Then the slots of each
// expert in slot order (one warp an expert, ballots over the slots), cut into
// segments of at most `tok`.
__global__ void __launch_bounds__(kRouteThreads) batch_route_kernel(const float *logits, int m, int E, int top_k,
                                                                    int tok, int *idx_out, float *w_out,
                                                                    BatchRoute *route) {
  __shared__ int idx_s[kRouteMaxSlots], count_s[kMoeMaxExperts], first_s[kMoeMaxExperts], seg_s[kMoeMaxExperts];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = kRouteThreads / 32;
  pdl_wait();
  pdl_launch_dependents();
  for (int t = warp; t < m; t += nw) {
    RouteKeys keys;
    route_load(keys, logits + (size_t)t * E, E, lane);
    float first = 0.f, mine = 0.f, sum = 0.f;  // lane c: choice c
    int mine_e = 0;
    for (int c = 0; c < top_k; ++c) {
      float l;
      const int e = route_next(keys, lane, l);
      if (c == 0) first = l;
      const float ex = expf(l - first);
      sum += ex;
      if (lane == c) mine = ex, mine_e = e;
    }
    if (lane < top_k) {
      idx_s[t * top_k + lane] = mine_e;
      idx_out[t * top_k + lane] = mine_e;
      w_out[t * top_k + lane] = __fdiv_rn(mine, sum);
    }
  }
  __syncthreads();
  const int S = m * top_k;
  for (int e = warp; e < E; e += nw) {
    int c = 0;
    for (int b = 0; b < S; b += 32) c += __popc(__ballot_sync(0xffffffffu, b + lane < S && idx_s[b + lane] == e));
    if (lane == 0) count_s[e] = c;
  }
  __syncthreads();
  if (warp == 0) {  // exclusive sums of the counts and of the segments
    int base = 0, sbase = 0;
    for (int b = 0; b < E; b += 32) {
      const int c = b + lane < E ? count_s[b + lane] : 0, ns = (c + tok - 1) / tok;
      int a = c, q = ns;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int ua = __shfl_up_sync(0xffffffffu, a, o), uq = __shfl_up_sync(0xffffffffu, q, o);
        if (lane >= o) a += ua, q += uq;
      }
      if (b + lane < E) {
        first_s[b + lane] = base + a - c;
        seg_s[b + lane] = sbase + q - ns;
      }
      base += __shfl_sync(0xffffffffu, a, 31);
      sbase += __shfl_sync(0xffffffffu, q, 31);
    }
    if (lane == 0) route->n_segs = sbase;
  }
  __syncthreads();
  for (int e = warp; e < E; e += nw) {
    const int c = count_s[e], f = first_s[e];
    int at = f;
    for (int b = 0; b < S; b += 32) {
      const bool in = b + lane < S && idx_s[b + lane] == e;
      const uint32_t v = __ballot_sync(0xffffffffu, in);
      if (in) route->list[at + __popc(v & ((1u << lane) - 1u))] = b + lane;
      at += __popc(v);
    }
    for (int q = lane; q * tok < c; q += 32) route->seg[seg_s[e] + q] = make_int4(e, min(tok, c - q * tok), f + q * tok, 0);
  }
}

cudaLaunchConfig_t batch_config(dim3 grid, dim3 block, cudaStream_t s, cudaLaunchAttribute *attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
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
                              float lora_scale, uint8_t *panel, float *rs, uint8_t *tfrag, unsigned *cnt, int n_cnt,
                              cudaStream_t s) {
  if (M <= 0 || M > kBatchMaxTokens || K <= 0 || K % 32 != 0) return cudaErrorInvalidValue;
  const int nt = batch_nt(M), KB = (K + 127) / 128;
  const bool lora = tfrag != nullptr && r > 0;
  const int row_tiles = lora ? (2 * r + 15) / 16 : rs != nullptr ? 1 : 0;
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg = batch_config(dim3(nt * row_tiles + (KB * nt * 8 + kPrepWarps - 1) / kPrepWarps),
                                        dim3(kPrepThreads), s, attr);
  return cudaLaunchKernelEx(&cfg, batch_prep_kernel<false>, reinterpret_cast<const __nv_bfloat16 *>(x), M, K,
                            bits == 4 ? 1 : 0, group, reinterpret_cast<const __nv_bfloat16 *>(lora_a), r, lora_scale,
                            panel, rs, lora ? tfrag : (uint8_t *)nullptr, cnt, n_cnt, nt, row_tiles,
                            (const BatchRoute *)nullptr, 1, 1);
}

cudaError_t launch_batch_route(const float *logits, int m, int E, int top_k, int nt, int *idx, float *w,
                               BatchRoute *route, cudaStream_t s) {
  if (m <= 0 || E <= 0 || E > kMoeMaxExperts || top_k <= 0 || top_k > 16 || top_k > E || m * top_k > kRouteMaxSlots)
    return cudaErrorInvalidValue;
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg = batch_config(dim3(1), dim3(kRouteThreads), s, attr);
  return cudaLaunchKernelEx(&cfg, batch_route_kernel, logits, m, E, top_k, 8 * nt, idx, w, route);
}

cudaError_t launch_batch_route_prep(const void *x, int K, int bits, int group, int top_k, const void *lora_a, int r,
                                    float lora_scale, uint8_t *panel, float *rs, uint8_t *tfrag, unsigned *cnt,
                                    int n_cnt, const BatchRoute *route, int max_segs, int nt, cudaStream_t s) {
  if (K <= 0 || K % 32 != 0) return cudaErrorInvalidValue;
  const int KB = (K + 127) / 128;
  const bool lora = tfrag != nullptr && r > 0;
  const int row_tiles = lora ? (2 * r + 15) / 16 : rs != nullptr ? 1 : 0;
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg =
      batch_config(dim3(max_segs * nt * row_tiles + (max_segs * KB * nt * 8 + kPrepWarps - 1) / kPrepWarps),
                   dim3(kPrepThreads), s, attr);
  return cudaLaunchKernelEx(&cfg, batch_prep_kernel<true>, reinterpret_cast<const __nv_bfloat16 *>(x), 0, K,
                            bits == 4 ? 1 : 0, group, reinterpret_cast<const __nv_bfloat16 *>(lora_a), r, lora_scale,
                            panel, rs, lora ? tfrag : (uint8_t *)nullptr, cnt, n_cnt, nt, row_tiles, route, top_k,
                            max_segs);
}

cudaError_t launch_batch_routed(GemvKind kind, const BatchArgs &a, int max_segs, int nt, cudaStream_t s) {
  if (a.route == nullptr || max_segs <= 0 || a.N % 16 != 0) return cudaErrorInvalidValue;
  int sms = 0;
  cudaError_t e = batch_sms(&sms);
  if (e != cudaSuccess) return e;
  const long long T = (long long)max_segs * ((a.N + kBatchRows - 1) / kBatchRows), W = T * ((a.K + 127) / 128);
  const int occ = batch_routed_occ(nt, T, sms), ctas = (int)std::max(1LL, std::min((long long)sms * occ, W / 2));
  switch (kind) {
    case kGateUpW2: return launch_batch_routed_gu2(a, nt, ctas, occ, s);
    case kGateUpW4: return launch_batch_routed_gu4(a, nt, ctas, occ, s);
    case kDownW4: return launch_batch_routed_dn4(a, nt, ctas, occ, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_batch(GemvKind kind, const BatchArgs &a, cudaStream_t s) {
  if (a.M <= 0 || a.M > kBatchMaxTokens) return cudaErrorInvalidValue;
  int sms = 0;
  cudaError_t e = batch_sms(&sms);
  if (e != cudaSuccess) return e;
  const long long W = (long long)((a.N + kBatchRows - 1) / kBatchRows) * ((a.K + 127) / 128);
  const int nt = batch_nt(a.M), T = (a.N + kBatchRows - 1) / kBatchRows, U = (a.K + 127) / 128;
  int ctas = (int)std::max(1LL, std::min((long long)sms, W / 2));
  // A whole row block a CTA where that is at most 3 units longer than an equal
  // share, about what the exchange of split parts costs (us, split -> whole: gate/up
  // of d 704 x inter 10624 at 43 tokens 24.3 -> 16.8, d 512 x 2048 at 16 9.3 -> 7.8).
  if (T < ctas && U * (long long)ctas <= W + 3LL * ctas) ctas = T;
  switch (kind) {
    case kGateUpW2: return launch_batch_gu2(a, nt, ctas, s);
    case kGateUpW3: return launch_batch_gu3(a, nt, ctas, s);
    case kGateUpW4: return launch_batch_gu4(a, nt, ctas, s);
    case kDownW4: return launch_batch_dn4(a, nt, ctas, s);
  }
  return cudaErrorInvalidValue;
}

// Two parts a CTA: 8 (gate/up) or 4 (down) warps x 2 tiles x NT x 32 float4s.
size_t batch_scratch_floats(int nt, int nproj, int num_sms) {
  return (size_t)num_sms * 2 * (nproj == 2 ? 8 : 4) * 2 * nt * 32 * 4;
}

size_t batch_tfrag_bytes(int nt, int r) { return (size_t)2 * ((r + 15) / 16) * nt * kTfragBytes; }

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
