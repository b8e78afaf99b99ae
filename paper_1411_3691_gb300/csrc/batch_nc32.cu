// batch_nc32.cu -- batched kernels for correlators whose largest n_f is in the
// n class 32 (one translation unit per class and kernel so they compile in parallel).
#include "fwd_impl.cuh"

namespace mhc {

cudaError_t launch_batch_nc32(int grid, int T, size_t smem, cudaStream_t s, const FwdArgs* desc,
                             const BatchItem* items, int64_t n_items, unsigned long long* head,
                             const int64_t* part_off, double2* partials) {
  return launch_batch_nc<32>(grid, T, smem, s, desc, items, n_items, head, part_off, partials);
}

int batch_occupancy_nc32(int T, size_t smem) { return batch_occupancy_nc<32>(T, smem); }

cudaError_t launch_kfac_batch_nc32(const FwdArgs* desc, const int64_t* kpref, const int64_t* nfam, int count,
                                  int64_t total, int big, cudaStream_t s) {
  return launch_kfac_batch_nc<32>(desc, kpref, nfam, count, total, big, s);
}

}  // namespace mhc
