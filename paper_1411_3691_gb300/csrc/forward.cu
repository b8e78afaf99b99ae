// forward.cu -- host launchers of the forward correlator and the deterministic reduction
// of the per-work-item partial sums.
#include "kernels.cuh"
#include "trace.h"

namespace mhc {

namespace {

// Sum of the per-item partials in a fixed order: every block sums a slice of its own, the last one
// to finish (by a counter that wraps to 0) the blocks' sums.  One block took 12.5 us for the 8192
// partials of the He-4 shapes.
constexpr int kReduceBlocks = kReduceMaxBlocks, kReduceThreads = 256;
__global__ void __launch_bounds__(kReduceThreads) reduce_kernel(const double2* __restrict__ p, int64_t n, double2* blocks,
                                                                unsigned* done, double* out) {
  __shared__ double2 red[kReduceThreads / 32];
  __shared__ bool last;
  auto block_sum = [&](double2 s) {
    s = dev::warp_sum(s);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    double2 t = red[0];
    for (int w = 1; w < kReduceThreads / 32; w++) t = dev::cadd(t, red[w]);
    return t;
  };
  const int64_t per = (n + gridDim.x - 1) / gridDim.x;
  const int64_t i0 = per * blockIdx.x, i1 = i0 + per < n ? i0 + per : n;
  double2 s = make_double2(0.0, 0.0);
  for (int64_t i = i0 + threadIdx.x; i < i1; i += kReduceThreads) s = dev::cadd(s, p[i]);
  s = block_sum(s);
  if (threadIdx.x == 0) {
    blocks[blockIdx.x] = s;
    __threadfence();
    last = atomicInc(done, gridDim.x - 1) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  s = make_double2(0.0, 0.0);
  if (threadIdx.x < gridDim.x) s = __ldcg(blocks + threadIdx.x);
  s = block_sum(s);
  if (threadIdx.x == 0) {
    out[0] = s.x;
    out[1] = s.y;
  }
}

}  // namespace

// tables: the launch's work items may use fixed-point tables (their warps' scratch is larger)
size_t forward_smem_bytes(int slots, int tile, int ncmax, bool tables) {
  const size_t cache = (size_t)slots * tile * sizeof(double2);
  const size_t scratch = ncmax <= 8    ? WarpScratch<8>::bytes(slots, tables)
                         : ncmax <= 18 ? WarpScratch<18>::bytes(slots, tables)
                                       : WarpScratch<32>::bytes(slots, tables);
  return cache + (size_t)(tile / 32) * scratch;
}

// fwd_kernel over items [0, items): one launch per layout range, each with its own y
// cache, or one launch with the plan's layout (smem: its size).
static cudaError_t launch_fwd_items(const FwdArgs& a, int ncmax, int tile, int64_t items, size_t smem,
                                    cudaStream_t s) {
  auto one = [&](const FwdArgs& x, int64_t count, size_t bytes) {
    return ncmax <= 8 ? launch_fwd_nc8(x, tile, count, bytes, s)
                      : (ncmax <= 18 ? launch_fwd_nc18(x, tile, count, bytes, s)
                                     : launch_fwd_nc32(x, tile, count, bytes, s));
  };
  if (!a.fam_order || a.n_ranges <= 0) return one(a, items, smem);
  for (int r = 0; r < a.n_ranges; r++) {
    const FwdRange& g = a.ranges[r];
    if (g.count <= 0) continue;
    FwdArgs ar = a;
    ar.slots = g.slots;
    for (int f = 0; f < MHC_FMAX; f++) ar.yoff[f] = g.yoff[f];
    ar.item0 = g.first * a.n_tiles;
    const cudaError_t e = one(ar, g.count * a.n_tiles, forward_smem_bytes(g.slots, tile, ncmax, a.fx.nf > 0));
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Up to this many partials per thread the forward kernel's last block sums them instead of a launch of
// reduce_kernel.  Every block then waits for its partial to be visible, a microsecond or two per wave of
// blocks: 512 x 512 terms (444 blocks of 128 threads, one wave) 8 us faster, 1291 x 977 (1600) 1 us
// faster, 1944 x 1944 10 us and 4096 x 4096 terms (8192 blocks) 23 us slower.
constexpr int kFoldPerThread = 16;
bool forward_folds(int64_t items, int tile) { return items <= (int64_t)kFoldPerThread * tile; }

cudaError_t launch_forward(const FwdArgs& a, int ncmax, int tile, int64_t n_fam, int64_t items,
                           size_t smem, double* out, cudaStream_t s) {
  cudaError_t e = launch_fxprep(a, s);
  if (e != cudaSuccess) return e;
  if (a.snk_orig) {  // two-sided update: the LU factors of every (family, sink family) block first
    TraceRange trace("block factors");
    if (ncmax <= 8)
      e = launch_kfac_nc8(a, n_fam, s);
    else if (ncmax <= 18)
      e = launch_kfac_nc18(a, n_fam, s);
    else
      e = launch_kfac_nc32(a, n_fam, s);
    if (e != cudaSuccess) return e;
  }
  FwdArgs fa = a;
  fa.fold_items = forward_folds(items, tile) ? items : 0;
  fa.out = out;
  {
    TraceRange trace("forward kernel");
    if ((e = launch_fwd_items(fa, ncmax, tile, items, smem, s)) != cudaSuccess) {
      cudaMemsetAsync(a.reduce_done, 0, sizeof(unsigned), s);  // a range launched before the failure counts
      return e;
    }
  }
  if (fa.fold_items) return cudaSuccess;
  TraceRange trace("reduce");
  return launch_reduce(a, items, out, s);
}

cudaError_t launch_reduce(const FwdArgs& a, int64_t items, double* out, cudaStream_t s) {
  const int64_t b = (items + kReduceThreads - 1) / kReduceThreads;
  reduce_kernel<<<(unsigned)(b < kReduceBlocks ? b : kReduceBlocks), kReduceThreads, 0, s>>>(
      a.partials, items, a.reduce_blocks, a.reduce_done, out);
  return cudaGetLastError();
}

// In slices: pair_group_kernel has one block per 2, 4 or 8 (pair, flavour) units, and a grid holds
// 2^31 - 1 blocks (eight flavours of n > 18: 2^29 pairs).  A slice fills the chip many times over.
constexpr int64_t kPairSlice = (int64_t)1 << 22;
cudaError_t launch_pairs(const FwdArgs& a, int ncmax, int64_t n_pairs, int64_t n_src,
                         const int64_t* ii, const int64_t* jj, const int32_t* src_member,
                         const int32_t* mem_family, double* dets, int32_t* path, cudaStream_t s) {
  const auto slice = ncmax <= 8 ? launch_pairs_nc8 : ncmax <= 18 ? launch_pairs_nc18 : launch_pairs_nc32;
  for (int64_t p = 0; p < n_pairs; p += kPairSlice) {
    const cudaError_t e = slice(a, n_pairs - p < kPairSlice ? n_pairs - p : kPairSlice, n_src, ii + p, jj + p, src_member,
                                mem_family, dets + 2 * p * a.F, path ? path + p : nullptr, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace mhc
