// wq_batch_gu2.cu -- instantiations of the batched-decode dequant-GEMM: 2-bit gate/up.
#include "wq_batch.cuh"

namespace wq {

cudaError_t launch_batch_gu2(const BatchArgs &a, int nt, int ctas, cudaStream_t s) {
  return launch_batch_g<2, 2>(a, nt, ctas, s);
}

cudaError_t launch_batch_routed_gu2(const BatchArgs &a, int nt, int ctas, int occ, cudaStream_t s) {
  return launch_batch_routed_g<2, 2>(a, nt, ctas, occ, s);
}

cudaError_t read_batch_status_gu2(int *status) { return read_batch_status_tu(status); }

}  // namespace wq
