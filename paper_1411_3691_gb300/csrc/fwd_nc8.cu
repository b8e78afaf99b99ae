// fwd_nc8.cu -- forward and block-factor kernels for plans whose largest n_f is in the
// n class 8 (one translation unit per class and kernel so they compile in parallel).
#include "fwd_impl.cuh"

namespace mhc {

cudaError_t launch_fwd_nc8(const FwdArgs& a, int tile, int64_t items, size_t smem, cudaStream_t s) {
  if (a.w_src_im) return launch_fwd_cw_nc8(a, tile, items, smem, s);
  if (a.fx.nf > 0) return launch_fwd_fx_nc8(a, tile, items, smem, s);
  return launch_fwd_nc<8, false, false>(a, tile, items, smem, s);
}

cudaError_t launch_kfac_nc8(const FwdArgs& a, int64_t n_fam, cudaStream_t s) {
  return launch_kfac_nc<8>(a, n_fam, s);
}

}  // namespace mhc
