// wq_batch_dn4.cu -- instantiations of the batched-decode dequant-GEMM: 4-bit down.
#include "wq_batch.cuh"

namespace wq {

cudaError_t launch_batch_dn4(const BatchArgs &a, int nt, int ctas, cudaStream_t s) {
  return launch_batch_g<4, 1>(a, nt, ctas, s);
}

cudaError_t launch_batch_routed_dn4(const BatchArgs &a, int nt, int ctas, int occ, cudaStream_t s) {
  return launch_batch_routed_g<4, 1>(a, nt, ctas, occ, s);
}

cudaError_t read_batch_status_dn4(int *status) { return read_batch_status_tu(status); }

}  // namespace wq
