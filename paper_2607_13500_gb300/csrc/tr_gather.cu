// Gather of the kept tokens: y[r] = x[row_off(b) + idx[r]] for the image b
// that owns output row r (cu_k[b] <= r < cu_k[b+1]), a bit copy of d * elem
// bytes per row (Eq. 7: X* is made of the original token vectors).  One warp
// per output row, 16-byte loads that skip L1 and streaming stores.
#include "tr_internal.cuh"

namespace tr {
namespace {

__device__ __forceinline__ uint4 ld_nc(const uint4 *p) {
  uint4 r;
  asm("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
      : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
      : "l"(p));
  return r;
}
__device__ __forceinline__ void st_cs(uint4 *p, const uint4 &v) {
  asm volatile("st.global.cs.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
               : "memory");
}

template <int kU>
__global__ void __launch_bounds__(kGatherWarps * 32)
    k_gather(const uint4 *__restrict__ x, long long total_rows, int batch, int n_uniform,
             const int32_t *__restrict__ cu_seqlens, const int32_t *__restrict__ cu_k,
             const int32_t *__restrict__ idx, int total_k, int nchunks, uint4 *__restrict__ y) {
  // idx comes from the kernel before this one.  No early trigger here: the next
  // call's score CTAs, placed a few at a time as this grid drains, would start
  // unevenly spread over the SMs (12 ragged images: 449 us a pass against 433)
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const int row = blockIdx.x * kGatherWarps + (threadIdx.x >> 5);
  if (row >= total_k) return;
  // image b: the last b with cu_k[b] <= row (skipping images with K_b = 0)
  int lo = 0, hi = batch;  // invariant: cu_k[lo] <= row < cu_k[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (__ldg(cu_k + mid) <= row) lo = mid; else hi = mid;
  }
  const long long first = cu_seqlens ? (long long)__ldg(cu_seqlens + lo) : (long long)lo * n_uniform;
  const long long n_b = cu_seqlens ? (long long)__ldg(cu_seqlens + lo + 1) - first : (long long)n_uniform;
  const int local = __ldcg(idx + row);  // through L2: idx may come from the kernel before
  const long long g = first + local;
  uint4 *dst = y + (long long)row * nchunks;
  // an index outside its own image's tokens (or an image outside x) writes
  // zeros: never a row of another image, never an address outside x
  if (local < 0 || local >= n_b || first < 0 || g >= total_rows) {
    for (int c = lane; c < nchunks; c += 32) st_cs(dst + c, make_uint4(0u, 0u, 0u, 0u));
    return;
  }
  const uint4 *src = x + (long long)g * nchunks;
  for (int c0 = lane; c0 < nchunks; c0 += 32 * kU) {  // kU loads in flight per lane
    uint4 v[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u)
      if (c0 + 32 * u < nchunks) v[u] = ld_nc(src + c0 + 32 * u);
#pragma unroll
    for (int u = 0; u < kU; ++u)
      if (c0 + 32 * u < nchunks) st_cs(dst + c0 + 32 * u, v[u]);
  }
}

}  // namespace

cudaError_t launch_gather(const void *x, long long total_rows, int dtype, int d, int batch, int n_uniform,
                          const int32_t *cu_seqlens, const int32_t *cu_k, const int32_t *idx, int total_k, void *y,
                          cudaStream_t st, bool pdl, bool beside_scoring) {
  if (total_k == 0) return cudaSuccess;
  const int nchunks = d * elem_bytes(dtype) / 16;
  const int grid = (total_k + kGatherWarps - 1) / kGatherWarps;
  auto launch = [&](auto kernel) {
    return launch_kernel(kernel, dim3(grid), dim3(kGatherWarps * 32), 0, st, pdl, static_cast<const uint4 *>(x),
                         total_rows, batch, n_uniform, cu_seqlens, cu_k, idx, total_k, nchunks,
                         static_cast<uint4 *>(y));
  };
  // A row's chunks dealt evenly over as few rounds as eight loads a lane allow
  // (14 per lane: two of seven), none alone: what a round costs is its latency.
  // (Four a round and the rest one by one took 55.5 us on 12 ragged images of
  // 3584 bf16 channels, 322 MB, against 51.8, and 10.2 against 8.2 for a clip's
  // 784 rows, launch included.)  Beside another batch's scoring (the pipeline)
  // four loads a round: there its own latency is hidden and its
  // bursts hold the scoring up (64 images of 576 x 4096 bf16, a third kept,
  // 168.2 us a batch against 168.6; 32 images, a third kept, 85.6 against 85.9).
  const int per_lane = (nchunks + 31) / 32;
  const int most = beside_scoring ? 4 : 8;
  const int rounds = (per_lane + most - 1) / most;
  switch ((per_lane + rounds - 1) / rounds) {
    case 1: return launch(k_gather<1>);
    case 2: return launch(k_gather<2>);
    case 3: return launch(k_gather<3>);
    case 4: return launch(k_gather<4>);
    case 5: return launch(k_gather<5>);
    case 6: return launch(k_gather<6>);
    case 7: return launch(k_gather<7>);
    default: return launch(k_gather<8>);
  }
}

}  // namespace tr
