// fwd_fx_nc18.cu -- forward kernel with fixed-point dots for plans whose largest n_f is in the
// n class 18 (one translation unit per class and kernel so they compile in parallel).
#include "fwd_impl.cuh"

namespace mhc {

cudaError_t launch_fwd_fx_nc18(const FwdArgs& a, int tile, int64_t items, size_t smem, cudaStream_t s) {
  return launch_fwd_nc<18, true, false>(a, tile, items, smem, s);
}

}  // namespace mhc
