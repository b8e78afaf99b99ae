// fwd_nc32.cu -- forward and block-factor kernels for plans whose largest n_f is in the
// n class 32 (one translation unit per class and kernel so they compile in parallel).
#include "fwd_impl.cuh"

namespace mhc {

cudaError_t launch_fwd_nc32(const FwdArgs& a, int tile, int64_t items, size_t smem, cudaStream_t s) {
  return launch_fwd_nc<32, false, true>(a, tile, items, smem, s);
}

cudaError_t launch_kfac_nc32(const FwdArgs& a, int64_t n_fam, cudaStream_t s) {
  return launch_kfac_nc<32>(a, n_fam, s);
}

}  // namespace mhc
