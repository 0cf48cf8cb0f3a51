// wq_attn.cu -- one decode step of grouped-query attention over a bf16 KV
// cache (sm_103a), the decoder-layer operator around the paper's MLP block
// whose cost Sec. 5 counts as independent of the weight precision.
//
// Per sequence b (one new token at position lens[b]) and kv head g:
//   1. rs = 1/sqrt(mean(x[b]^2) + eps): the layer input's RMSNorm scale,
//      applied to the projections (the normalized input is never rounded);
//   2. q heads h of the group, k and v of g: the fp32 projections x deq(W)^T
//      times rs; q and k normalized per head (unit-weight RMSNorm) and rotated
//      (RoPE, element i with i + hd/2, angle pos theta^(-2i/hd): the
//      frequencies come from the host in fp64, the angle is formed and reduced
//      modulo 2 pi in fp64 -- a few fp64 operations a CTA -- and its cosine
//      and sine taken in fp32 on the reduced argument);
//   3. k and v rounded to bf16 and appended to the cache at lens[b];
//   4. o = softmax(q K^T / sqrt(hd)) V over positions 0..lens[b].
// The context is cut into S splits (grid.y); a CTA of 4 warps takes one (b, g)
// and one split, each warp chunks of 16 positions.  A warp copies its next
// chunk's K and V rows into a shared-memory buffer of its own (cp.async,
// 16-byte chunks XOR-swizzled by the row) while it computes the current one.
// With `early` (the caller knows that nothing but qkv comes from the launch
// before, and that that launch lets this one start only after its own wait) the
// first two chunks, the layer input's norm and the RoPE angles come before the
// wait, under the projection's launch (a decoder layer of one sequence of 8192
// positions 49.0 -> 46.0 us, of 16 of 512 to 2048 79.6 -> 76.1).
//
// Scores and outputs are mma.sync products of the bf16 rows, with the fp32
// operand in three bf16 parts (8 significand bits each, 24 in all), so that
// every product is exact and the sums are fp32 as before: the 4 query heads'
// parts are the columns of Q (head h: columns 2h, 2h + 1 of the first 8-column
// tile and 2h of the second), the probabilities' parts the rows of P (row h +
// 4 part), added up at the end.  A chunk takes 16 + 16 MMAs where the lanes'
// dot products, their 31-shuffle reduction and the probabilities' 32 broadcasts
// took ~1000 instructions.  The softmax runs online (max, sum, rescaled
// accumulators) in fp32.  Parts of an infinite operand would cancel into NaN;
// a warp whose result holds a NaN therefore computes its range again with
// plain fp32 products (attn_plain).  The splits' partial results (max, sum,
// accumulator) are merged in a fixed order by a second kernel.
//
// Bound by the latency of the chunks' loads and of the steps before them (the
// layer input's norm, RoPE, the head norms); two chunks of 8 KB a warp and 12
// warps an SM keep ~190 KB in flight.  Measured (GB300, cold, us, lanes' dot
// products with 8 warps a CTA and two CTAs an SM before -> this): 16 sequences of 512
// to 2048 positions, 32 / 8 heads of 128: 39.1 -> 24.4 for 84 MB of cache rows;
// one of 8192: 17.5 -> 14.7 for 34 MB; the kept roundings of the scores (below) took
// 0.6 and 0.2 us of it back.  Share of bf16 outputs off the exact rounding 0.00027
// -> 0.00022 at 8192 positions, 0.00024 -> 0.00019 at 512 to 2048.
#include <algorithm>
#include <cmath>
#include <cstdint>

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "wq_internal.h"
#include "wq_ptx.cuh"

namespace wq {

// Status word of the attention kernels: WQ_OK (0), or WQ_ERR_ARG (-1) after a
// sequence length outside [0, max_len) was met on the device (that sequence is
// skipped).  Read and cleared by read_attn_status.
__device__ int g_attn_status = 0;

namespace {

constexpr int kAttnWarps = 4;
constexpr int kAttnOcc = 3;   // CTAs an SM holds (64 KB of K and V buffers each)
constexpr int kCombWarps = 8;
constexpr int kHG = 4;        // query heads a pass takes (padded with zero heads)
constexpr int kPos = 16;      // positions a chunk takes

__device__ __forceinline__ float bf_lo(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf_hi(uint32_t v) { return __uint_as_float(v & 0xffff0000u); }

// x = hi + mid + lo with bf16 parts (exact to 24 bits).
__device__ __forceinline__ void split3(float x, float (&p)[3]) {
  p[0] = __bfloat162float(__float2bfloat16_rn(x));
  p[1] = __bfloat162float(__float2bfloat16_rn(x - p[0]));
  p[2] = x - p[0] - p[1];
}
__device__ __forceinline__ uint32_t pack_bf2(float a, float b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t *>(&v);
}

}  // namespace

// RoPE frequencies theta^(-2i/hd), i < hd/2, computed on the host in fp64.
struct RopeFreq {
  double f[64];
};

// Copies of one chunk (positions cb .. cb + kPos - 1) of K and V rows into a
// warp's buffer ([K, V][kPos][HD], 16-byte chunk c of row r at c ^ (r % 8)):
// positions outside [p0, p1) and the new position pos are zero-filled.
template <int HD>
__device__ __forceinline__ void attn_issue(__nv_bfloat16 *buf, const __nv_bfloat16 *kbase, const __nv_bfloat16 *vbase,
                                           int lane, int cb, int p0, int p1, int pos) {
  constexpr int CPR = HD * 2 / 16;  // 16-byte copies a row
  const int c = lane % CPR;
#pragma unroll
  for (int i = 0; i < 2 * kPos * CPR / 32; ++i) {
    const int r = i * (32 / CPR) + lane / CPR;
    const int p = cb + r % kPos;
    const bool in = p < p1 && p != pos;
    const __nv_bfloat16 *src = (r < kPos ? kbase : vbase) + (size_t)(in ? p : p0) * HD + c * 8;
    cp_async16_zfill(buf + (size_t)r * HD + (c ^ (r & 7)) * 8, src, in ? 16u : 0u);
  }
}

// One warp's share of a split with plain fp32 products (a lane: HD / 32
// dimensions): the same chunks, any values.  Leaves max, sum and accumulator in
// shared memory as the fast loop does.
template <int HD>
__device__ __noinline__ void attn_plain(const float (*qs)[HD], const float (*kvn)[HD], const __nv_bfloat16 *kbase,
                                        const __nv_bfloat16 *vbase, int h0, int rep, int first, int stride, int p1,
                                        int pos, float *ws_m, float *ws_l, float (*ws_o)[HD]) {
  constexpr int E = HD / 32;
  const int lane = threadIdx.x & 31;
  for (int hq = 0; hq < kHG; ++hq) {
    float m = -INFINITY, l = 0.f, o[E];
    for (int e = 0; e < E; ++e) o[e] = 0.f;
    for (int cb = first; cb < p1; cb += stride)
      for (int p = cb; p < min(p1, cb + kPos); ++p) {
        float s = 0.f, v[E];
        for (int e = 0; e < E; ++e) {
          const int i = lane * E + e;
          const float k = p == pos ? kvn[0][i] : __bfloat162float(kbase[(size_t)p * HD + i]);
          v[e] = p == pos ? kvn[1][i] : __bfloat162float(vbase[(size_t)p * HD + i]);
          s = fmaf(h0 + hq < rep ? qs[h0 + hq][i] : 0.f, k, s);
        }
        for (int x = 16; x >= 1; x >>= 1) s += __shfl_xor_sync(0xffffffffu, s, x);
        const float mn = fmaxf(m, s), al = mn == -INFINITY ? 1.f : exp2f(m - mn);
        const float pr = s == -INFINITY ? 0.f : exp2f(s - mn);
        l = l * al + pr;
        m = mn;
        for (int e = 0; e < E; ++e) o[e] = fmaf(pr, v[e], o[e] * al);
      }
    if (lane == 0) {
      ws_m[hq] = m;
      ws_l[hq] = l;
    }
    for (int e = 0; e < E; ++e) ws_o[hq][lane * E + e] = o[e];
  }
  __syncwarp();
}

// Dynamic shared memory: per warp two chunk buffers of K and V rows,
// [warp][buffer][K, V][kPos][HD] bf16.
template <int HD>
constexpr int attn_smem_bytes() { return kAttnWarps * 2 * 2 * kPos * HD * 2; }

// grid (B * n_kv, S), block kAttnWarps * 32.  part: [B][H][S][HD + 2] fp32
// (accumulator, max, sum) of every split.
template <int HD>
__global__ void __launch_bounds__(kAttnWarps * 32, kAttnOcc) attn_split_kernel(
    const float *qkv, const __nv_bfloat16 *x, const int *lens, int d, int H, int Hkv, const RopeFreq fr,
    __nv_bfloat16 *k_cache, __nv_bfloat16 *v_cache, int max_len, float *part, int S, int early) {
  constexpr int E = HD / 32;  // dimensions a lane holds
  extern __shared__ __align__(16) uint8_t attn_dyn[];
  __shared__ __align__(16) float qs[kHG * 2][HD];  // the group's query heads (up to 8), scaled by log2(e)/sqrt(HD)
  __shared__ float kvn[2][HD];       // the new token's k (normalized, rotated, bf16-rounded) and v
  __shared__ float red[kAttnWarps];
  __shared__ float rc[HD / 2], rsn[HD / 2];  // cos, sin of the RoPE angles at this position
  __shared__ float ws_m[kAttnWarps][kHG * 2], ws_l[kAttnWarps][kHG * 2];
  __shared__ __align__(16) float ps_s[kAttnWarps][kHG][kPos];  // a chunk's probabilities
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (!early) {
    pdl_wait();
    pdl_launch_dependents();
  }
  const int b = blockIdx.x / Hkv, g = blockIdx.x % Hkv, split = blockIdx.y;
  const int rep = H / Hkv;
  const int pos = lens[b];          // the new token's position
  if (pos < 0 || pos >= max_len) {  // no room in the cache: record, skip the sequence
    if (threadIdx.x == 0 && blockIdx.y == 0 && g == 0) atomicExch(&g_attn_status, -1);
    if (early) pdl_wait();
    return;
  }
  const int L = pos + 1;            // positions attended
  const int C = (L + S - 1) / S;    // positions a split
  const int p0 = split * C, p1 = min(L, p0 + C);
  const int row = (H + 2 * Hkv) * HD;
  const size_t cache_off = ((size_t)b * Hkv + g) * max_len * HD;
  constexpr int WBYTES = 2 * 2 * kPos * HD * 2;  // a warp's buffers; after the loop its accumulator [kHG][HD]
  __nv_bfloat16 *wbuf = reinterpret_cast<__nv_bfloat16 *>(attn_dyn + warp * WBYTES);
  const __nv_bfloat16 *kbase = k_cache + cache_off, *vbase = v_cache + cache_off;
  constexpr int stride = kAttnWarps * kPos;
  const int first = p0 + warp * kPos;
  auto issue = [&](int c, int buf) {
    if (c < p1) attn_issue<HD>(wbuf + (size_t)buf * 2 * kPos * HD, kbase, vbase, lane, c, p0, p1, pos);
    cp_async_commit();
  };
  issue(first, 0);
  issue(first + stride, 1);

  // RoPE angles at the new position: pos f_i in fp64, reduced to [-pi, pi]
  if (tid < HD / 2) {
    const double a = (double)pos * fr.f[tid];
    const double k = rint(a * 0.15915494309189535);  // 1 / (2 pi)
    const double red_a = fma(-k, 6.283185307179586, a);
    const float r = (float)fma(-k, 2.4492935982947064e-16, red_a);  // 2 pi - fl(2 pi)
    float sn, cs;
    sincosf(r, &sn, &cs);
    rc[tid] = cs;
    rsn[tid] = sn;
  }
  // 1. rs of x[b]
  float ss = 0.f;
  for (int i = tid; i < d / 8; i += blockDim.x) {
    const uint4 v = *reinterpret_cast<const uint4 *>(x + (size_t)b * d + 8 * i);
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      ss = fmaf(bf_lo(w[e]), bf_lo(w[e]), ss);
      ss = fmaf(bf_hi(w[e]), bf_hi(w[e]), ss);
    }
  }
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  if (lane == 0) red[warp] = ss;
  __syncthreads();
  float tot = 0.f;
  for (int w = 0; w < kAttnWarps; ++w) tot += red[w];
  const float rs = __fdiv_rn(1.f, __fsqrt_rn(__fadd_rn(__fdiv_rn(tot, (float)d), kRmsEps)));

  if (early) {
    pdl_wait();
    pdl_launch_dependents();
  }

  // 2./3. the group's q heads, k and v: warp w takes heads w, w + 4, .. (q heads, then k, then v)
  const bool has_new = p0 <= pos && pos < p1;
  constexpr int HPW = (kHG * 2 + 2 + kAttnWarps - 1) / kAttnWarps;  // heads a warp at most, loaded in one round trip
  float raw[HPW][E];
#pragma unroll
  for (int u = 0; u < HPW; ++u) {
    const int hh = warp + u * kAttnWarps;
    const int col = hh < rep ? (g * rep + hh) * HD : hh == rep ? (H + g) * HD : (H + Hkv + g) * HD;
#pragma unroll
    for (int e = 0; e < E; ++e) raw[u][e] = hh < rep + 2 ? __ldcg(qkv + (size_t)b * row + col + lane * E + e) : 0.f;
  }
#pragma unroll
  for (int u = 0; u < HPW; ++u) {
    const int hh = warp + u * kAttnWarps;
    if (hh >= rep + 2) break;
    float v[E];
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = raw[u][e] * rs;
    if (hh <= rep) {
      // per-head RMSNorm, then RoPE: element i (< HD/2) with i + HD/2, held by lane and lane ^ 16
      float sq = 0.f;
#pragma unroll
      for (int e = 0; e < E; ++e) sq = fmaf(v[e], v[e], sq);
#pragma unroll
      for (int o = 16; o >= 1; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
      const float hn = __fdiv_rn(1.f, __fsqrt_rn(__fadd_rn(__fdiv_rn(sq, (float)HD), kRmsEps)));
#pragma unroll
      for (int e = 0; e < E; ++e) v[e] *= hn;
      float pv[E];
#pragma unroll
      for (int e = 0; e < E; ++e) pv[e] = __shfl_xor_sync(0xffffffffu, v[e], 16);
      const bool lo = lane < 16;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int i = (lane & 15) * E + e;  // index in the first half
        const float c = rc[i], s = rsn[i];
        v[e] = lo ? v[e] * c - pv[e] * s : v[e] * c + pv[e] * s;
      }
    }
    if (hh < rep) {
      const float qsc = 1.4426950408889634f * __frsqrt_rn((float)HD);  // scores in units of log 2: exp2f below
#pragma unroll
      for (int e = 0; e < E; ++e) qs[hh][lane * E + e] = v[e] * qsc;
    } else {
      const int kv = hh - rep;  // 0: k, 1: v
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const __nv_bfloat16 bv = __float2bfloat16_rn(v[e]);
        kvn[kv][lane * E + e] = __bfloat162float(bv);
        if (has_new) (kv == 0 ? k_cache : v_cache)[cache_off + (size_t)pos * HD + lane * E + e] = bv;
      }
    }
  }
  __syncthreads();

  // 4. attention over [p0, p1): per pass, 4 query heads
  const int gr = lane >> 2, tc = lane & 3;  // fragment row and column pair
  auto ws_o = [&](int w) { return reinterpret_cast<float(*)[HD]>(attn_dyn + w * WBYTES); };
  // ldmatrix row of this lane: matrices (rows 0-7, 8-15) x (16-byte chunk 2 j, 2 j + 1)
  const int lrow = (lane & 7) + (lane & 8), lchk = lane >> 4;
  for (int h0 = 0; h0 < rep; h0 += kHG) {
    if (h0 > 0) {
      issue(first, 0);
      issue(first + stride, 1);
    }
    // Q's parts as B fragments: column gr of tile 0 is part gr % 2 of head gr / 2,
    // of tile 1 (even gr) its third part
    uint32_t qb[HD / 16][2][2];
#pragma unroll
    for (int ks = 0; ks < HD / 16; ++ks)
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        float pa[3] = {0.f, 0.f, 0.f}, pb[3] = {0.f, 0.f, 0.f};
        if (h0 + (gr >> 1) < rep) {
          const float2 qv = *reinterpret_cast<const float2 *>(&qs[h0 + (gr >> 1)][16 * ks + 8 * u + 2 * tc]);
          split3(qv.x, pa);
          split3(qv.y, pb);
        }
        qb[ks][0][u] = gr & 1 ? pack_bf2(pa[1], pb[1]) : pack_bf2(pa[0], pb[0]);
        qb[ks][1][u] = gr & 1 ? 0u : pack_bf2(pa[2], pb[2]);
      }
    float m_run = -INFINITY, l_run = 0.f;  // of head h0 + tc (l_run: this lane's positions)
    float acc[HD / 8][4];                  // rows gr, gr + 8 of P V: heads' parts
#pragma unroll
    for (int j = 0; j < HD / 8; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[j][e] = 0.f;
    int bi = 0;
    for (int c0 = first; c0 < p1; c0 += stride, bi ^= 1) {
      cp_async_wait_group1();  // this chunk's rows have landed
      __syncwarp();
      __nv_bfloat16 *cur = wbuf + (size_t)bi * 2 * kPos * HD;
      if (c0 <= pos && pos < c0 + kPos) {  // the new token's rows
        const int r = pos - c0;
        for (int i = lane; i < 2 * HD; i += 32) {
          const int row = (i / HD) * kPos + r, e = i % HD;
          cur[(size_t)row * HD + ((e >> 3) ^ (row & 7)) * 8 + (e & 7)] = __float2bfloat16_rn(kvn[i / HD][e]);
        }
        __syncwarp();
      }
      const uint32_t krow = smem_addr(cur) + lrow * (HD * 2), vrow = krow + kPos * HD * 2;
      // The tensor core's own accumulation truncates, which showed as twice the
      // outputs off the exact rounding, so Q's first parts start every MMA from zero
      // and are added in fp32 here (likewise P V); the other two, 2^-8 and 2^-16 of
      // them, accumulate.  The first parts' sums are added pairwise, then with what
      // each addition rounds away kept (Knuth's two-sum).  Scores of deviation 6 (in
      // units of log 2), outputs off the exact rounding: added one by one 0.00052,
      // this 0.00033, lanes' dot products 0.00038.
      float d0[4] = {0.f, 0.f, 0.f, 0.f}, d1[4] = {0.f, 0.f, 0.f, 0.f}, pair[2] = {0.f, 0.f};
      float hi[2] = {0.f, 0.f}, rest[2] = {0.f, 0.f};
#pragma unroll
      for (int ks = 0; ks < HD / 16; ++ks) {
        uint32_t ka[4];
        ldmatrix_x4(ka, krow + (((2 * ks + lchk) ^ (lrow & 7)) << 4));
        d0[0] = d0[2] = 0.f;
        mma_bf16_16816(d0, ka, qb[ks][0][0], qb[ks][0][1]);
        mma_bf16_16816(d1, ka, qb[ks][1][0], qb[ks][1][1]);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          if (ks % 2 == 0) {
            pair[i] = d0[2 * i];
          } else {
            const float v = pair[i] + d0[2 * i], sum = __fadd_rn(hi[i], v), bb = __fsub_rn(sum, hi[i]);
            if (ks > 1) rest[i] = __fadd_rn(rest[i], __fadd_rn(__fsub_rn(hi[i], __fsub_rn(sum, bb)), __fsub_rn(v, bb)));
            hi[i] = ks > 1 ? sum : v;
          }
        }
      }
      // scores of positions c0 + gr, c0 + gr + 8 with head h0 + tc
      const float s0 = c0 + gr < p1 ? hi[0] + ((d0[1] + d1[0]) + rest[0]) : -INFINITY;
      const float s1 = c0 + gr + 8 < p1 ? hi[1] + ((d0[3] + d1[2]) + rest[1]) : -INFINITY;
      float mc = fmaxf(s0, s1);
      mc = fmaxf(mc, __shfl_xor_sync(0xffffffffu, mc, 4));
      mc = fmaxf(mc, __shfl_xor_sync(0xffffffffu, mc, 8));
      mc = fmaxf(mc, __shfl_xor_sync(0xffffffffu, mc, 16));
      const float m_new = fmaxf(m_run, mc);
      const float alpha = m_new == -INFINITY ? 1.f : exp2f(m_run - m_new);
      const float e0 = s0 == -INFINITY ? 0.f : exp2f(s0 - m_new), e1 = s1 == -INFINITY ? 0.f : exp2f(s1 - m_new);
      l_run = l_run * alpha + (e0 + e1);
      m_run = m_new;
      ps_s[warp][tc][gr] = e0;
      ps_s[warp][tc][gr + 8] = e1;
      if (__any_sync(0xffffffffu, alpha != 1.f)) {
        const float al = __shfl_sync(0xffffffffu, alpha, (lane & 28) | (gr & 3));  // of head gr % 4
#pragma unroll
        for (int j = 0; j < HD / 8; ++j)
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[j][e] *= al;
      }
      __syncwarp();
      // P's parts as the A fragment: row gr is part gr / 4 of head gr % 4, row gr
      // + 8 (gr < 4) its third part
      uint32_t pa[4];
      {
        const float2 x0 = *reinterpret_cast<const float2 *>(&ps_s[warp][gr & 3][2 * tc]);
        const float2 x1 = *reinterpret_cast<const float2 *>(&ps_s[warp][gr & 3][2 * tc + 8]);
        float q0[3], q1[3], q2[3], q3[3];
        split3(x0.x, q0);
        split3(x0.y, q1);
        split3(x1.x, q2);
        split3(x1.y, q3);
        const bool lo = gr < 4;
        pa[0] = lo ? pack_bf2(q0[0], q1[0]) : pack_bf2(q0[1], q1[1]);
        pa[1] = lo ? pack_bf2(q0[2], q1[2]) : 0u;
        pa[2] = lo ? pack_bf2(q2[0], q3[0]) : pack_bf2(q2[1], q3[1]);
        pa[3] = lo ? pack_bf2(q2[2], q3[2]) : 0u;
      }
#pragma unroll
      for (int j = 0; j < HD / 16; ++j) {
        uint32_t vb[4];
        ldmatrix_x4_trans(vb, vrow + (((2 * j + lchk) ^ (lrow & 7)) << 4));
        float t0[4] = {0.f, 0.f, 0.f, 0.f}, t1[4] = {0.f, 0.f, 0.f, 0.f};
        mma_bf16_16816(t0, pa, vb[0], vb[1]);
        mma_bf16_16816(t1, pa, vb[2], vb[3]);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          acc[2 * j][e] += t0[e];
          acc[2 * j + 1][e] += t1[e];
        }
      }
      __syncwarp();  // every lane is done with this buffer before it is filled again
      issue(c0 + 2 * stride, bi);
    }
    cp_async_wait_all();
    // the parts added up: head h0 + gr (gr < 4), dimensions 8 j + 2 tc, + 1
    bool bad = m_run != m_run;
#pragma unroll
    for (int o = 4; o <= 16; o <<= 1) l_run += __shfl_xor_sync(0xffffffffu, l_run, o);
#pragma unroll
    for (int j = 0; j < HD / 8; ++j)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float mid = __shfl_xor_sync(0xffffffffu, acc[j][e], 16);
        const float v = (acc[j][2 + e] + mid) + acc[j][e];
        bad |= gr < 4 && v != v;
        if (gr < 4) ws_o(warp)[gr][8 * j + 2 * tc + e] = v;
      }
    if (lane < kHG) {
      ws_m[warp][lane] = m_run;
      ws_l[warp][lane] = l_run;
    }
    if (__any_sync(0xffffffffu, bad || l_run != l_run))
      attn_plain<HD>(qs, kvn, kbase, vbase, h0, rep, first, stride, p1, pos, ws_m[warp], ws_l[warp], ws_o(warp));
    // merge the warps (fixed order) and write the split's partials
    __syncthreads();
    for (int i = tid; i < kHG * HD; i += blockDim.x) {
      const int hq = i / HD, e = i % HD;
      if (h0 + hq >= rep) continue;
      float M = -INFINITY;
      for (int w = 0; w < kAttnWarps; ++w) M = fmaxf(M, ws_m[w][hq]);
      float Ls = 0.f, O = 0.f;
      for (int w = 0; w < kAttnWarps; ++w) {
        const float f = ws_m[w][hq] == -INFINITY ? 0.f : exp2f(ws_m[w][hq] - M);
        Ls = fmaf(ws_l[w][hq], f, Ls);
        O = fmaf(ws_o(w)[hq][e], f, O);
      }
      const int h = g * rep + h0 + hq;
      float *pt = part + (((size_t)b * H + h) * S + split) * (HD + 2);
      pt[e] = O;
      if (e == 0) {
        pt[HD] = M;
        pt[HD + 1] = Ls;
      }
    }
    __syncthreads();
  }
}

// o[b][h * HD + e] = bf16( sum_s O_s 2^(M_s - M) / sum_s L_s 2^(M_s - M) ).
// grid B * H, 8 warps: warp w merges the splits w, w + 8, .. in order, CU at a
// time (their loads, rows of HD + 2 floats, in one round trip beside the
// length's, then their max; a decoder layer of one sequence of 8192 positions,
// 57 splits, 46.2 -> 43.7 us against a pass for the max first; CU 1 up to 8
// splits, where the seven empty places cost 1 %), lane l the features l * HD/32
// ..; then the warps' results are merged in warp order -- a fixed order, so the
// result is deterministic.
template <int HD, int CU>
__global__ void __launch_bounds__(kCombWarps * 32) attn_combine_kernel(const float *part, const int *lens, int H, int S,
                                                                       int max_len, __nv_bfloat16 *o) {
  constexpr int E = HD / 32;
  __shared__ float wm[kCombWarps], wl[kCombWarps], wo[kCombWarps][HD];
  const int bh = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  pdl_wait();
  pdl_launch_dependents();
  const int pos = lens[bh / H];
  const float *pt = part + (size_t)bh * S * (HD + 2) + lane * E;
  float M = -INFINITY, L = 0.f, O[E];
#pragma unroll
  for (int e = 0; e < E; ++e) O[e] = 0.f;
  for (int s0 = warp; s0 < S; s0 += CU * kCombWarps) {
    float2 ml[CU], ov[CU][E / 2];
    float mn = M;
#pragma unroll
    for (int u = 0; u < CU; ++u) {
      const int s = s0 + u * kCombWarps;
      const float *ps = pt + (size_t)s * (HD + 2);
      ml[u] = s < S ? *reinterpret_cast<const float2 *>(ps + HD - lane * E) : make_float2(-INFINITY, 0.f);
#pragma unroll
      for (int e = 0; e < E / 2; ++e)
        ov[u][e] = s < S ? *reinterpret_cast<const float2 *>(ps + 2 * e) : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < CU; ++u) mn = fmaxf(mn, ml[u].x);
    const float f0 = M == -INFINITY ? 0.f : exp2f(M - mn);
    M = mn;
    L *= f0;
#pragma unroll
    for (int e = 0; e < E; ++e) O[e] *= f0;
#pragma unroll
    for (int u = 0; u < CU; ++u) {
      if (s0 + u * kCombWarps >= S) break;
      const float f = ml[u].x == -INFINITY ? 0.f : exp2f(ml[u].x - M);
      L = fmaf(ml[u].y, f, L);
#pragma unroll
      for (int e = 0; e < E / 2; ++e) {
        O[2 * e] = fmaf(ov[u][e].x, f, O[2 * e]);
        O[2 * e + 1] = fmaf(ov[u][e].y, f, O[2 * e + 1]);
      }
    }
  }
  if (pos < 0 || pos >= max_len) return;  // skipped by the split kernel
  if (lane == 0) {
    wm[warp] = M;
    wl[warp] = L;
  }
#pragma unroll
  for (int e = 0; e < E; ++e) wo[warp][lane * E + e] = O[e];
  __syncthreads();
  for (int e = threadIdx.x; e < HD; e += blockDim.x) {
    float Mt = -INFINITY;
    for (int w = 0; w < kCombWarps; ++w) Mt = fmaxf(Mt, wm[w]);
    float Lt = 0.f, Ot = 0.f;
    for (int w = 0; w < kCombWarps; ++w) {
      const float f = wm[w] == -INFINITY ? 0.f : exp2f(wm[w] - Mt);
      Lt = fmaf(wl[w], f, Lt);
      Ot = fmaf(wo[w][e], f, Ot);
    }
    o[(size_t)bh * HD + e] = __float2bfloat16_rn(Ot / Lt);
  }
}

int attn_splits(int B, int Hkv, int max_len, int num_sms) {
  // as many CTAs as the SMs hold at once, at least 64 positions a split
  const int want = std::max(1, kAttnOcc * num_sms / (B * Hkv));
  return std::max(1, std::min(want, (max_len + 63) / 64));
}

long long attn_most_parts(int B, int Hkv, int max_len, int num_sms) {
  // b splits(b) is b, or at most the CTAs held (and 64 positions a split)
  return std::min(std::max((long long)B, (long long)kAttnOcc * num_sms / Hkv), (long long)B * ((max_len + 63) / 64));
}

namespace {

template <int HD>
cudaError_t launch_attn_t(const float *qkv, const __nv_bfloat16 *x, const int *lens, int B, int d, int H, int Hkv,
                          const RopeFreq &fr, __nv_bfloat16 *kc, __nv_bfloat16 *vc, int max_len, float *part, int S,
                          __nv_bfloat16 *o, bool early, cudaStream_t s) {
  constexpr int sm = attn_smem_bytes<HD>();
  cudaError_t e = cudaFuncSetAttribute(attn_split_kernel<HD>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.gridDim = dim3(B * Hkv, S);
  cfg.blockDim = dim3(kAttnWarps * 32);
  cfg.dynamicSmemBytes = sm;
  e = cudaLaunchKernelEx(&cfg, attn_split_kernel<HD>, qkv, x, lens, d, H, Hkv, fr, kc, vc, max_len, part, S,
                         early ? 1 : 0);
  if (e != cudaSuccess) return e;
  cfg.gridDim = dim3(B * H);
  cfg.blockDim = dim3(kCombWarps * 32);
  cfg.dynamicSmemBytes = 0;
  return cudaLaunchKernelEx(&cfg, S <= kCombWarps ? attn_combine_kernel<HD, 1> : attn_combine_kernel<HD, 8>,
                            (const float *)part, lens, H, S, max_len, o);
}

}  // namespace

cudaError_t launch_attn_decode(const float *qkv, const void *x, const int *lens, int B, int d, int H, int Hkv, int HD,
                               double theta, void *k_cache, void *v_cache, int max_len, float *part, int S, void *o,
                               bool early, cudaStream_t s) {
  if (HD > 128) return cudaErrorInvalidValue;
  RopeFreq fr{};
  for (int i = 0; i < HD / 2; ++i) fr.f[i] = std::pow(theta, -2.0 * i / HD);
  const auto *xb = reinterpret_cast<const __nv_bfloat16 *>(x);
  auto *kc = reinterpret_cast<__nv_bfloat16 *>(k_cache), *vc = reinterpret_cast<__nv_bfloat16 *>(v_cache);
  auto *ob = reinterpret_cast<__nv_bfloat16 *>(o);
  if (HD == 128) return launch_attn_t<128>(qkv, xb, lens, B, d, H, Hkv, fr, kc, vc, max_len, part, S, ob, early, s);
  if (HD == 64) return launch_attn_t<64>(qkv, xb, lens, B, d, H, Hkv, fr, kc, vc, max_len, part, S, ob, early, s);
  return cudaErrorInvalidValue;
}

cudaError_t read_attn_status(int *status) {
  cudaError_t e = cudaDeviceSynchronize();
  if (e != cudaSuccess) return e;
  e = cudaMemcpyFromSymbol(status, g_attn_status, sizeof(int));
  if (e != cudaSuccess) return e;
  const int zero = 0;
  return cudaMemcpyToSymbol(g_attn_status, &zero, sizeof(int));
}

}  // namespace wq
