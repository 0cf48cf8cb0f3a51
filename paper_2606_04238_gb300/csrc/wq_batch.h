// wq_batch.h -- the batched-decode dequant-GEMM (wq_batch.cuh): host interface.
#pragma once

#include <cstddef>
#include <cstdint>

#include <cuda_runtime.h>

#include "wq_internal.h"

namespace wq {

constexpr int kBatchMaxTokens = 64;  // tokens a launch can take (8 MMA tiles of 8)

// 8-token MMA tiles a launch of m tokens computes (the kernels exist for
// 1, 2, 3, 4, 6 and 8).
inline int batch_nt(int m) {
  const int n = (m + 7) / 8;
  return n <= 4 ? n : n <= 6 ? 6 : 8;
}

// Activation panel: one record per 128-feature block,
//   [NT][4][32 lanes][16 bytes]  the binary16 m16n8k16 B fragments of two
//                                16-feature steps a lane, scaled by 2^e per
//                                (block, token) -- e puts the largest |x| in
//                                [2^14, 2^15) -- and by 4^-c (2- and 3-bit
//                                codes) or 16^-c (4-bit) for the bit-position
//                                class c of the codes they meet
//   [NT * 8] fp32                2^(24 - e) per token
//   [128 / group][NT * 8] fp32   sums of x 2^(e - 24) over each quantization group
inline __host__ __device__ uint32_t batch_rec_bytes(int nt, int group) {
  return (uint32_t)nt * (2048u + 32u + 32u * (128u / (uint32_t)group));
}

// Slots of a routed call grouped by expert (written by launch_batch_route):
// segment s holds slots list[seg[s].z .. + seg[s].y) of expert seg[s].x.
constexpr int kRouteMaxSlots = 1024, kRouteMaxSegs = 1024;
struct BatchRoute {
  int n_segs;
  int4 seg[kRouteMaxSegs];
  int list[kRouteMaxSlots];
};
// Segments that m tokens of top_k choices can make at most.
inline int batch_max_segs(int slots, int experts, int nt) {
  return (slots < experts ? slots : experts) + slots / (8 * nt);
}

// CTAs an SM of a routed launch over `tiles` row blocks (of all segments at
// most).  A CTA of many row blocks finishes several, each finish a latency chain
// of one set of warps: with a second CTA of 8 warps the other computes
// meanwhile; with few row blocks twice the CTAs mean twice the split ones.
// Measured (us a block, one CTA vs two; row blocks an SM): 64 experts of 2048 x
// 768, 2.8: 61.4 vs 56.9; GPT-OSS-20B shape, 2.7: 65.6 vs 66.7, 3.3: 73.0 vs 72.2,
// 6: 123 vs 118.4; 8 experts of 4096 x 4096, 2.1: 68.1 vs 70.0, 2.9: 95.3 vs 94.8;
// 8 experts of 2048 x 2048, 1.1: 36.6 vs 40.2.
inline int batch_routed_occ(int nt, long long tiles, int num_sms) {
  return nt <= 2 && 4 * tiles >= 11LL * num_sms ? 2 : 1;
}

// A fragment of the LoRA-A products t in three bf16 parts whose sum is the fp32
// value: [32 lanes][16 bytes] the high and the middle part, then [32 lanes][8
// bytes] the low one.
constexpr uint32_t kTfragBytes = 768;

struct BatchArgs {
  const uint8_t *panel;      // [ceil(K / 128)] records
  int M, N, K, group;
  const uint32_t *codes[2];  // gate, up; or down
  const uint16_t *meta[2];
  // gate/up: lora_scale * x A^T, m16n8k16 B fragments [projection][ceil(r / 16)]
  // [NT] of kTfragBytes (null: no adapter); LoRA-B bf16 [N][r]; RMSNorm scale
  // per token (null: 1)
  const uint8_t *tfrag;
  int r;
  const void *lora_b[2];
  const float *rs;
  const void *residual;      // down: bf16 [M][N] or null
  void *out;                 // bf16 (down: or fp32) [M][N]; gate/up: may be null with panel_out
  int out_f32;
  uint8_t *panel_out;        // gate/up: also the 4-bit down launch's panel of h (null: none)
  int group_out;             // its quantization group
  float *part;               // batch_scratch_floats() fp32
  unsigned *cnt;             // [ceil(N / 128)] (routed: per segment) arrival counters, zeroed by the input launch and left at zero
  // Routed experts: the launch computes segments of up to 8 nt (token, choice)
  // slots of one expert each.  codes, meta, lora_b: the experts' matrices
  // stacked row-wise, N rows an expert (a multiple of 16); panel, tfrag, rs,
  // panel_out: one per segment; out: one row a slot.
  const BatchRoute *route;   // null: one dense matrix, M tokens
};

// Panel of x bf16 [M, K] for codes of `bits` bits and groups of `group`, and
// with rs / tfrag (either may be null) the RMSNorm scales and LoRA-A products.
// cnt [n_cnt] is zeroed: the arrival counters of the launches that follow (a
// workspace used at several token counts holds other data there in between).
cudaError_t launch_batch_prep(const void *x, int M, int K, int bits, int group, const void *lora_a, int r,
                              float lora_scale, uint8_t *panel, float *rs, uint8_t *tfrag, unsigned *cnt, int n_cnt,
                              cudaStream_t s);
cudaError_t launch_batch(GemvKind kind, const BatchArgs &a, cudaStream_t s);
// Routed: the top_k experts of each token with their softmax weights (slot
// t * top_k + j), and the slots grouped by expert in segments of 8 nt.
cudaError_t launch_batch_route(const float *logits, int m, int E, int top_k, int nt, int *idx, float *w,
                               BatchRoute *route, cudaStream_t s);
// Panels, RMSNorm scales (rs not null) and LoRA-A products (tfrag not null) of
// every segment, and cnt [n_cnt] zeroed; max_segs bounds the grid.
cudaError_t launch_batch_route_prep(const void *x, int K, int bits, int group, int top_k, const void *lora_a, int r,
                                    float lora_scale, uint8_t *panel, float *rs, uint8_t *tfrag, unsigned *cnt,
                                    int n_cnt, const BatchRoute *route, int max_segs, int nt, cudaStream_t s);
// Routed launch: nt 1, 2 or 4; max_segs for the grid.
cudaError_t launch_batch_routed(GemvKind kind, const BatchArgs &a, int max_segs, int nt, cudaStream_t s);
size_t batch_scratch_floats(int nt, int nproj, int num_sms);
size_t batch_tfrag_bytes(int nt, int r);
cudaError_t read_batch_status(int *status);

// One translation unit per kind.
cudaError_t launch_batch_gu2(const BatchArgs &a, int nt, int ctas, cudaStream_t s);
cudaError_t launch_batch_routed_gu2(const BatchArgs &a, int nt, int ctas, int occ, cudaStream_t s);
cudaError_t launch_batch_gu3(const BatchArgs &a, int nt, int ctas, cudaStream_t s);
cudaError_t launch_batch_gu4(const BatchArgs &a, int nt, int ctas, cudaStream_t s);
cudaError_t launch_batch_routed_gu4(const BatchArgs &a, int nt, int ctas, int occ, cudaStream_t s);
cudaError_t launch_batch_dn4(const BatchArgs &a, int nt, int ctas, cudaStream_t s);
cudaError_t launch_batch_routed_dn4(const BatchArgs &a, int nt, int ctas, int occ, cudaStream_t s);
cudaError_t read_batch_status_gu2(int *status);
cudaError_t read_batch_status_gu3(int *status);
cudaError_t read_batch_status_gu4(int *status);
cudaError_t read_batch_status_dn4(int *status);

}  // namespace wq
