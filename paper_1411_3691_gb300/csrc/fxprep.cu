// fxprep.cu -- the fixed-point tables of the member dots (fx.cuh), rebuilt by every call: they
// depend on the propagators and the weights.
//
// One launch.  Blocks [0, sum_f L_f) convert one propagator row each: the row's largest binary
// exponent, then its entries as limbs, and the limbs of the column of the same label at the
// column's exponent; the last of them to finish decides whether the call takes the fixed-point path
// (fx::Scan).  The other blocks take one source family each: a member's first row
// of the first flavour, times the member's signed weight, is stored at its own exponent, beside the
// binades by which the member's product scale lies below its family's largest: by that many the member
// loop shifts the product before it sums the members in integers (aligning the rows instead would round
// every entry of a small member, not its product).  A row with a weight of zero is stored as it is: its
// pairs pass the guards as the others, and count nothing.  A member whose rows or weight are not finite,
// or whose rows are zero, is left to the FP64 path.  The work is a pass over 2 F L^2 +
// members L entries (He-4 shapes: 206 000, 3.3 MB written).
#include "kernels.cuh"

namespace mhc {

namespace {

constexpr int kThreads = 512;  // a warp per member of a family of 16: one chain of loads each

// exponent above every used entry of a row or column (largest binary exponent + 1); one warp
__device__ __forceinline__ int row_exponent(const dev::cd* row, int pitch, int L, int lane, const int* used, int bit) {
  int e = -4096;
  for (int l = lane; l < L; l += 32)
    if (used[l] & bit) e = max(e, dev::expo(dev::ldS(row + (size_t)l * pitch)));
  return __reduce_max_sync(0xffffffffu, e) + 1;
}

// Whether the call's propagators are flat, by the last of its row blocks.
__device__ void scan_all(const FwdArgs& a) {
  __shared__ int red[kThreads / 32][6];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  bool flat = true;
  for (int f = 0; f < a.F; f++) {
    if (a.n_f[f] == 0) continue;
    fx::Scan s;
    for (int l = threadIdx.x; l < a.L_f[f]; l += kThreads) {
      const int4 v = __ldcg(a.fx.scan[f] + l);
      s.row(v.x, v.z, v.w);
      s.column(v.y);
    }
    const int v[6] = {__reduce_min_sync(0xffffffffu, s.rlo), __reduce_max_sync(0xffffffffu, s.rhi),
                      __reduce_min_sync(0xffffffffu, s.clo), __reduce_max_sync(0xffffffffu, s.chi),
                      __reduce_add_sync(0xffffffffu, s.small), __reduce_add_sync(0xffffffffu, s.total)};
    __syncthreads();
    for (int k = 0; k < 6; k++)
      if (lane == 0) red[warp][k] = v[k];
    __syncthreads();
    fx::Scan t;
    for (int q = 0; q < kThreads / 32; q++) {
      t.rlo = min(t.rlo, red[q][0]);
      t.rhi = max(t.rhi, red[q][1]);
      t.clo = min(t.clo, red[q][2]);
      t.chi = max(t.chi, red[q][3]);
      t.small += red[q][4];
      t.total += red[q][5];
    }
    flat = flat && t.flat();
  }
  if (threadIdx.x == 0) a.fx.state[0] = flat ? 1 : 0;
}

// row b and column b of flavour f
__device__ void prep_row(const FwdArgs& a, int f, int b, int n_rows) {
  __shared__ int counts[2];
  __shared__ bool last;
  const int L = a.L_f[f], lane = threadIdx.x & 31;
  const int* used = a.fx.used[f];
  const dev::cd* row = a.S[f] + (size_t)b * L;
  const int is = used[b];
  // every warp for itself: no barrier
  const int e = is & 1 ? row_exponent(row, 1, L, lane, used, 2) : -4096;
  const int ec = is & 2 ? row_exponent(a.S[f] + b, L, L, lane, used, 1) : -4096;
  if (threadIdx.x == 0) {
    const_cast<int*>(a.fx.cexp[f])[b] = ec;
    counts[0] = counts[1] = 0;
  }
  __syncthreads();
  int4* out = const_cast<int4*>(a.fx.s[f]) + (size_t)b * L;
  int4* outc = const_cast<int4*>(a.fx.sc[f]) + b;
  int small = 0, total = 0;
  for (int l = threadIdx.x; l < L; l += kThreads) {
    const int us = used[l];
    if ((is & 1) && (us & 2)) {
      const dev::cd z = dev::ldS(row + l);
      out[l] = e <= 1023 ? fx::quant(z, e, fx::kRowBits) : make_int4(0, 0, 0, 0);
      small += fx::small_entry(z, e);
      total++;
    }
    if ((is & 2) && (us & 1))
      outc[(size_t)l * L] = ec <= 1023 ? fx::quant(dev::ldS(a.S[f] + (size_t)l * L + b), ec, fx::kABits) : make_int4(0, 0, 0, 0);
  }
  small = __reduce_add_sync(0xffffffffu, small);
  total = __reduce_add_sync(0xffffffffu, total);
  if (lane == 0) {
    atomicAdd(&counts[0], small);
    atomicAdd(&counts[1], total);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const_cast<int4*>(a.fx.scan[f])[b] = make_int4(e, ec, counts[0], counts[1]);
    __threadfence();
    last = atomicInc(reinterpret_cast<unsigned*>(a.fx.state + 1), n_rows - 1) == (unsigned)n_rows - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  scan_all(a);
}

__device__ __forceinline__ bool is_zero(dev::cd w) { return w.x == 0.0 && w.y == 0.0; }
__device__ __forceinline__ dev::cd weighted(const FwdArgs& a, dev::cd w, dev::cd z) {
  if (is_zero(w)) return z;
  return a.w_src_im ? dev::cmul(w, z) : make_double2(w.x * z.x, w.x * z.y);
}

__device__ void prep_family(const FwdArgs& a, int W) {
  __shared__ int e0s[64], rest[64];
  __shared__ dev::cd ws[64];
  const int f0 = a.fx.f0, L0 = a.L_f[f0];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int mem0 = a.fam_info[4 * W], kW = a.fam_info[4 * W + 1];  // kW <= 64
  // per member: the exponent above w times its first row, and the sum of its other rows' ones
  for (int c = warp; c < kW; c += kThreads / 32) {
    const int m = mem0 + c;
    const dev::cd w = dev::source_weight<true>(a, m);
    const int32_t* lab = a.mem_lab + (int64_t)m * a.F * MHC_MAX_RANK;
    int r = 0, e0 = -4096;
    bool bad = dev::expo(w) >= 1024;
    for (int f = 0; f < a.F; f++) {
      if (a.n_f[f] == 0) continue;
      for (int t = 0; t < a.fam_rank[(int64_t)W * a.F + f]; t++) {
        const dev::cd* row = a.S[f] + (size_t)lab[f * MHC_MAX_RANK + t] * a.L_f[f];
        const bool first = f == f0 && t == 0;
        int e = -4096;
        for (int l = lane; l < a.L_f[f]; l += 32) {
          if (!(a.fx.used[f][l] & 2)) continue;
          const dev::cd z = dev::ldS(row + l);
          e = max(e, dev::expo(z));
          if (first) e0 = max(e0, dev::expo(weighted(a, w, z)));
        }
        e = __reduce_max_sync(0xffffffffu, e) + 1;
        bad |= e > 1023 || e < -1000;
        if (!first) r += e;
      }
    }
    e0 = __reduce_max_sync(0xffffffffu, e0) + 1;
    bad |= e0 > 1023 || e0 < -1000;
    if (lane == 0) {
      ws[c] = w;
      e0s[c] = bad ? -100000 : e0;
      rest[c] = r;
    }
  }
  __syncthreads();
  int X = -100000;
  for (int c = 0; c < kW; c++)
    if (e0s[c] > -100000 && !is_zero(ws[c])) X = max(X, e0s[c] + rest[c]);
  if (threadIdx.x == 0) {
    const_cast<int*>(a.fx.fexp)[W] = X;
    for (int c = kW; c & 3; c++)  // a step of four that the family does not fill
      reinterpret_cast<unsigned char*>(const_cast<unsigned*>(a.fx.align + mem0 + (c & ~3)))[c & 3] = fx::kMute;
  }
  for (int c = warp; c < kW; c += kThreads / 32) {
    const int m = mem0 + c;
    const bool bad = e0s[c] == -100000;
    if (lane == 0) {
      const int d = X - e0s[c] - rest[c];
      const_cast<int*>(a.fx.below)[m] = d;
      reinterpret_cast<unsigned char*>(const_cast<unsigned*>(a.fx.align + mem0 + (c & ~3)))[c & 3] =
          bad ? fx::kOnlyFp64 : is_zero(ws[c]) ? fx::kMute : d > fx::kMaxAlign ? fx::kFar : d;
    }
    const int32_t lab = a.mem_lab[((int64_t)m * a.F + f0) * MHC_MAX_RANK];
    const dev::cd* row = a.S[f0] + (size_t)lab * L0;
    int4* out = const_cast<int4*>(a.fx.ws) + (size_t)m * L0;
    for (int l = lane; l < L0; l += 32) {
      if (!(a.fx.used[f0][l] & 2)) continue;
      dev::cd z = make_double2(0.0, 0.0);
      if (!bad) z = weighted(a, ws[c], dev::ldS(row + l));
      out[l] = fx::quant(z, bad ? 0 : e0s[c], fx::kRowBits);
    }
  }
}

__device__ void prep_block(const FwdArgs& a, int64_t b) {
  if (a.fx.nf == 0) return;
  int n_rows = 0;
  for (int f = 0; f < a.F; f++) n_rows += a.n_f[f] > 0 ? a.L_f[f] : 0;
  for (int f = 0; f < a.F; f++) {
    if (a.n_f[f] == 0) continue;
    if (b < a.L_f[f]) {
      prep_row(a, f, (int)b, n_rows);
      return;
    }
    b -= a.L_f[f];
  }
  if (b < a.n_fam) prep_family(a, (int)b);
}

__global__ void __launch_bounds__(kThreads) fxprep_kernel(const FwdArgs a) { prep_block(a, blockIdx.x); }

__global__ void __launch_bounds__(kThreads) fxprep_batch_kernel(const FwdArgs* __restrict__ desc,
                                                                const int64_t* __restrict__ pref, int count) {
  int lo = 0, hi = count - 1;
  while (lo < hi) {  // last k with pref[k] <= block
    const int mid = (lo + hi + 1) >> 1;
    if (pref[mid] <= (int64_t)blockIdx.x) lo = mid; else hi = mid - 1;
  }
  prep_block(desc[lo], (int64_t)blockIdx.x - pref[lo]);
}

}  // namespace

int64_t fxprep_blocks(const FwdArgs& a) {
  if (a.fx.nf == 0) return 0;
  int64_t n = a.n_fam;
  for (int f = 0; f < a.F; f++) n += a.n_f[f] > 0 ? a.L_f[f] : 0;
  return n;
}

cudaError_t launch_fxprep(const FwdArgs& a, cudaStream_t s) {
  const int64_t n = fxprep_blocks(a);
  if (n == 0) return cudaSuccess;
  fxprep_kernel<<<(unsigned)n, kThreads, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_fxprep_batch(const FwdArgs* desc, const int64_t* pref, int count, int64_t total, cudaStream_t s) {
  if (total == 0) return cudaSuccess;
  fxprep_batch_kernel<<<(unsigned)total, kThreads, 0, s>>>(desc, pref, count);
  return cudaGetLastError();
}

}  // namespace mhc
