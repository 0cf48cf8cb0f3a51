// wq_pack.cu -- Stage-1 group-wise quantizer and packer (sm_103a).
//
// Sec. 4.1 quantizes gate/up to INT2 and (Sec. 3.3, Sec. 7 step 4) every
// other linear layer to INT4.  The quantizer is asymmetric min-max
// round-to-nearest per group of `group` consecutive input features of a row,
// computed in IEEE fp32 with explicit round-to-nearest intrinsics so that the
// codes, scales and zeros are reproducible bit for bit:
//   s = fp16((max - min) / qmax) (1.0 if zero), z = clamp(rint(-min/s), 0, qmax),
//   q = clamp(rint(w/s) + z, 0, qmax).
// One kernel, one warp per packed block of 16 rows x 128 features.  A lane
// loads the features that its words of the packed layout hold (float2s; the 8
// rows' sectors of an instruction are used in full), so each weight is read
// once and the words are assembled in registers; min and max of a (row, group)
// come from its 4 lanes by two shuffles.  Bound by HBM: 4 bytes in and bits/8
// out a weight.  The per-weight division is a multiplication by the reciprocal
// of s, with the exact division only where the product lies so near a rounding
// boundary that the two could differ.  Offline work: not on the decode path.
// A second kernel merges a trained adapter into a packed matrix before it is
// quantized again (below).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>

#include "wq_internal.h"
#include "wq_launch.h"

namespace wq {
namespace {

constexpr int kPackWarps = 8;  // blocks a CTA

// rint(v / sf) as the IEEE division gives it.  p = v * rcp is within |p| 2^-22
// of the quotient (two roundings), as is the division's own result, so both
// round to the same integer unless p is that near to a half.
__device__ __forceinline__ float rint_div(float v, float sf, float rcp) {
  const float p = __fmul_rn(v, rcp), r = rintf(p);
  if (fabsf(p - r) < 0.5f - fabsf(p) * 0x1p-21f) return r;
  return rintf(__fdiv_rn(v, sf));  // also nan and infinite quotients
}

template <int BITS, int GROUP>
__global__ void __launch_bounds__(kPackWarps * 32) pack_kernel(const float *__restrict__ w, int n, int k, int RT, int KB,
                                                               uint32_t *__restrict__ codes,
                                                               uint16_t *__restrict__ meta, int *nonfinite) {
  constexpr int WPB = BITS * 64, GPB = 128 / GROUP, JG = GROUP / 8;  // code words a block, groups, 8-feature steps a group
  const long long blk = (long long)blockIdx.x * kPackWarps + (threadIdx.x >> 5);
  if (blk >= (long long)RT * KB) return;  // warp-uniform
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int rt = (int)(blk / KB), kb = (int)(blk - (long long)rt * KB);
  const int nj = min(16, (k - kb * 128) / 8);  // 8-feature steps inside the matrix (k a multiple of the group)
  // rows g and g + 8 of the tile, features 8 j + 2 t, + 1 of the block
  float2 v[2][16];
  bool in[2], bad = false;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int row = rt * 16 + g + 8 * h;
    in[h] = row < n;
    const float *src = w + (size_t)(in[h] ? row : 0) * k + kb * 128 + 2 * t;
#pragma unroll
    for (int j = 0; j < 16; ++j)
      v[h][j] = in[h] && j < nj ? __ldcs(reinterpret_cast<const float2 *>(src + 8 * j)) : make_float2(0.f, 0.f);
  }
  const float qmax = (float)((1 << BITS) - 1);
  uint32_t lo[BITS == 4 ? 8 : 4] = {}, hi[2] = {};
#pragma unroll
  for (int gi = 0; gi < GPB; ++gi) {
    unsigned short s16[2], z16[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float mn = INFINITY, mx = -INFINITY;
#pragma unroll
      for (int j = gi * JG; j < (gi + 1) * JG; ++j) {
        mn = fminf(mn, fminf(v[h][j].x, v[h][j].y));
        mx = fmaxf(mx, fmaxf(v[h][j].x, v[h][j].y));
        bad |= !isfinite(v[h][j].x) || !isfinite(v[h][j].y);
      }
#pragma unroll
      for (int o = 1; o < 4; o <<= 1) {
        mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      }
      __half sh = __float2half_rn(__fdiv_rn(__fsub_rn(mx, mn), qmax));
      if (__half2float(sh) == 0.f) sh = __float2half_rn(1.f);
      const float sf = __half2float(sh);
      const float zf = __fadd_rn(fminf(fmaxf(rintf(__fdiv_rn(-mn, sf)), 0.f), qmax), 0.f);
      const bool real = in[h] && gi * JG < nj;  // codes, scale and zero are 0 outside the matrix
      s16[h] = real ? __half_as_ushort(sh) : 0;
      z16[h] = real ? __half_as_ushort(__float2half_rn(zf)) : 0;
      const float rcp = __frcp_rn(sf);
#pragma unroll
      for (int j = gi * JG; j < (gi + 1) * JG; ++j)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const float q = fminf(fmaxf(__fadd_rn(rint_div(e ? v[h][j].y : v[h][j].x, sf, rcp), zf), 0.f), qmax);
          const uint32_t c = real ? (uint32_t)q : 0u;
          if (BITS == 4) {
            lo[j >> 1] |= c << (16 * e + 8 * h + 4 * (j & 1));
          } else {
            lo[j >> 2] |= (c & 3u) << (16 * e + 8 * h + 2 * (j & 3));
            if (BITS == 3) hi[j >> 3] |= (c >> 2) << (16 * e + 8 * ((j >> 2) & 1) + 2 * (j & 3) + h);
          }
        }
    }
    if (t == 0) {
      const uint2 m2 = make_uint2((uint32_t)s16[0] | ((uint32_t)s16[1] << 16), (uint32_t)z16[0] | ((uint32_t)z16[1] << 16));
      *reinterpret_cast<uint2 *>(meta + (((size_t)rt * KB + kb) * GPB + gi) * 32 + 4 * g) = m2;
    }
  }
  uint32_t *dst = codes + (size_t)blk * WPB;
  *reinterpret_cast<uint4 *>(dst + lane * 4) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
  if (BITS == 4) *reinterpret_cast<uint4 *>(dst + 128 + lane * 4) = make_uint4(lo[4], lo[5], lo[6], lo[7]);
  if (BITS == 3) *reinterpret_cast<uint2 *>(dst + 128 + lane * 2) = make_uint2(hi[0], hi[1]);
  if (nonfinite != nullptr && __any_sync(0xffffffffu, bad) && lane == 0) atomicOr(nonfinite, 1);
}

// Adapter merge (Sec. 4.2 lets the trained adapters be merged into the
// quantized weights; Sec. 7 step 5 deploys them merged or attached).  By
// Eq. 1 the merged matrix is deq(W) + alpha B A:
//   w[row, col] = fp32( s (q - z) + alpha * sum_rho B[row, rho] A[rho, col] ),
// evaluated in fp64 with rho ascending (a product of two bf16 values is exact)
// and rounded to fp32 once.  Every operation is an explicit round-to-nearest
// intrinsic, so no contraction changes the result.  The codes, scales and
// zeros are read from the packed layout of include/wq.h.  A CTA takes 256
// features of a row (rows strided by gridDim.y); the row of B is staged in
// shared memory as fp64.
constexpr int kMergeThreads = 256;

__global__ void __launch_bounds__(kMergeThreads)
    merge_lora_kernel(const uint32_t *__restrict__ codes, const uint16_t *__restrict__ meta, int n, int k,
                      int group, int bits, int KB, int NG, const __nv_bfloat16 *__restrict__ lora_b,
                      const __nv_bfloat16 *__restrict__ lora_a, int r, double alpha, float *__restrict__ w) {
  __shared__ double brow[kMaxRank];
  const int col = blockIdx.x * kMergeThreads + threadIdx.x;
  const int wpb = bits == 2 ? 128 : bits == 3 ? 192 : 256;
  const uint32_t mask = bits == 3 ? 3u : (1u << bits) - 1u;
  for (int row = blockIdx.y; row < n; row += gridDim.y) {
    __syncthreads();  // the previous row's B is read by every thread first
    if (threadIdx.x < r) brow[threadIdx.x] = (double)__bfloat162float(lora_b[(size_t)row * r + threadIdx.x]);
    __syncthreads();
    if (col >= k) continue;
    const int rt = row >> 4, i = row & 15, kb = col >> 7, c = col & 127;
    const int lane = (i & 7) * 4 + ((c & 7) >> 1), half = c & 1;
    int word, bit;
    if (bits != 4) {
      word = lane * 4 + (c >> 5);
      bit = 16 * half + 8 * (i >> 3) + 2 * (2 * ((c & 31) >> 4) + ((c & 15) >> 3));
    } else {
      word = (c >> 6) * 128 + lane * 4 + ((c & 63) >> 4);
      bit = 16 * half + 8 * (i >> 3) + 4 * ((c & 15) >> 3);
    }
    const uint32_t *blk = codes + ((size_t)rt * KB + kb) * wpb;
    uint32_t q = (blk[word] >> bit) & mask;
    if (bits == 3) {  // the high bit from the second plane
      const int cls = 2 * ((c & 31) >> 4) + ((c & 15) >> 3);
      q |= ((blk[128 + lane * 2 + ((c >> 5) >> 1)] >> (16 * half + 8 * ((c >> 5) & 1) + 2 * cls + (i >> 3))) & 1u) << 2;
    }
    const size_t mb = ((size_t)rt * NG + col / group) * 32 + 4 * (i & 7) + (i >> 3);
    const double sf = (double)__half2float(__ushort_as_half(meta[mb]));
    const double zf = (double)__half2float(__ushort_as_half(meta[mb + 2]));
    double ba = 0.0;
    for (int rho = 0; rho < r; ++rho)
      ba = __dadd_rn(ba, __dmul_rn(brow[rho], (double)__bfloat162float(lora_a[(size_t)rho * k + col])));
    const double v = __dadd_rn(__dmul_rn(sf, __dsub_rn((double)q, zf)), __dmul_rn(alpha, ba));
    w[(size_t)row * k + col] = __double2float_rn(v);
  }
}

}  // namespace

cudaError_t launch_merge_lora(const uint32_t *codes, const uint16_t *meta, int n, int k, int group, int bits,
                              const void *lora_b, const void *lora_a, int r, float alpha, float *w,
                              cudaStream_t stream) {
  const int KB = (k + 127) / 128, NG = KB * 128 / group;
  const dim3 grid((unsigned)((k + kMergeThreads - 1) / kMergeThreads), (unsigned)std::min(n, 65535));
  merge_lora_kernel<<<grid, kMergeThreads, 0, stream>>>(codes, meta, n, k, group, bits, KB, NG,
                                                         static_cast<const __nv_bfloat16 *>(lora_b),
                                                         static_cast<const __nv_bfloat16 *>(lora_a), r,
                                                         (double)alpha, w);
  return cudaGetLastError();
}

template <int BITS>
static void launch_pack_g(const float *w, int n, int k, int group, uint32_t *codes, uint16_t *meta, int *nonfinite,
                          cudaStream_t stream) {
  const int RT = (n + 15) / 16, KB = (k + 127) / 128;
  const unsigned ctas = (unsigned)(((long long)RT * KB + kPackWarps - 1) / kPackWarps);
  if (group == 32)
    pack_kernel<BITS, 32><<<ctas, kPackWarps * 32, 0, stream>>>(w, n, k, RT, KB, codes, meta, nonfinite);
  else if (group == 64)
    pack_kernel<BITS, 64><<<ctas, kPackWarps * 32, 0, stream>>>(w, n, k, RT, KB, codes, meta, nonfinite);
  else
    pack_kernel<BITS, 128><<<ctas, kPackWarps * 32, 0, stream>>>(w, n, k, RT, KB, codes, meta, nonfinite);
}

cudaError_t launch_pack(const float *w, int n, int k, int group, int bits, uint32_t *codes, uint16_t *meta,
                        int *nonfinite, cudaStream_t stream) {
  if (bits == 2)
    launch_pack_g<2>(w, n, k, group, codes, meta, nonfinite, stream);
  else if (bits == 3)
    launch_pack_g<3>(w, n, k, group, codes, meta, nonfinite, stream);
  else
    launch_pack_g<4>(w, n, k, group, codes, meta, nonfinite, stream);
  return cudaGetLastError();
}

}  // namespace wq
