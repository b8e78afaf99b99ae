// fwd_cw_nc8.cu -- forward kernel for complex weights, with and without fixed-point dots, for plans whose largest n_f is in the
// n class 8 (one translation unit per class and kernel so they compile in parallel).
#include "fwd_impl.cuh"

namespace mhc {

cudaError_t launch_fwd_cw_nc8(const FwdArgs& a, int tile, int64_t items, size_t smem, cudaStream_t s) {
  return launch_fwd_nc<8, true, true>(a, tile, items, smem, s);
}

}  // namespace mhc
