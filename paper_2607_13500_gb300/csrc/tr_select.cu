// The selection kernels (Algorithm 1) on statistics left by the scoring kernel:
// k_select runs one CTA per image (or several images in turn when the launch
// caps the grid, as the pipeline does), by the fast path of
// tr_select_cluster.cuh up to kSoloMaxN tokens and by select_image
// (tr_select_dev.cuh) above and for what that path leaves open;
// k_select_cluster shares each image among the CTAs of a cluster
// (select_cluster_ctas: large images of small batches).
//
// k_select_gather (tr_reduce on uniform batches that take no clusters) also
// copies the kept rows.
// With fewer images than SMs it runs R replica CTAs per image: each makes
// the same deterministic selection (only replica 0 writes idx and the status
// words) and copies its 1/R share of the image's kept rows, so the copies of
// one image overlap the selections of the others on SMs that would be idle.
#include <algorithm>
#include <atomic>

#include "tr_select_cluster.cuh"
#include "tr_select_dev.cuh"

namespace tr {
namespace {

// CTA c selects images c, c + gridDim.x, ... (one image per CTA unless the
// launch caps the grid below the batch).
__global__ void __launch_bounds__(kSelectThreads, 1) k_select(const SelectArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  pdl_trigger();
  pdl_wait();  // the statistics come from the kernel before this one
  for (int b = blockIdx.x; b < a.batch; b += gridDim.x) select_image_solo(a, b, smem, true);
}

// A cluster of c CTAs per image (large images of small batches).
__global__ void __launch_bounds__(kSelectThreads, 1) k_select_cluster(const SelectArgs a, const int c) {
  extern __shared__ __align__(16) unsigned char smem[];
  pdl_trigger();
  pdl_wait();  // the statistics come from the kernel before this one
  const int b = blockIdx.x / c, rank = (int)tc::cluster_rank();
  if (select_image_cluster<true>(a, b, c, rank, smem, true, nullptr)) return;
  cluster_barrier();  // nobody reads this CTA's shared memory any more
  if (rank == 0) select_image(a, b, smem);
}

__device__ __forceinline__ uint4 ld_nc16(const uint4 *p) {
  uint4 r;
  asm("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
      : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
      : "l"(p));
  return r;
}

// Replica r of `replicas` copies its share of image b's kept rows, whose
// local indices select_image left in this CTA's shared memory.
__device__ __forceinline__ void copy_kept(const SelectArgs &a, const int b, const int r, const int replicas,
                                          const int nchunks, uint4 *__restrict__ y, const uint16_t *kept) {
  long long off;
  int n;
  if (a.cu_seqlens) {
    off = a.cu_seqlens[b];
    n = a.cu_seqlens[b + 1] - a.cu_seqlens[b];
  } else {
    off = (long long)b * a.n_uniform;
    n = a.n_uniform;
  }
  const int k = a.k[b], k1 = a.k1[b], ko = a.cu_k[b];
  if (n <= 0 || n > a.max_n || off < 0 || off + n > a.total_rows || k < 0 || k > n || k1 < 0 || k1 > k)
    return;  // counted by select_image
  // this replica's share of the image's kept rows
  const int j0 = (int)((long long)r * k / replicas), j1 = (int)((long long)(r + 1) * k / replicas);
  const uint4 *x = static_cast<const uint4 *>(a.x);
  // one warp per row, eight 16-byte loads in flight per lane, streaming stores
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int kU = 8;
  for (int j = j0 + warp; j < j1; j += kWarps) {
    const uint4 *src = x + (off + kept[j]) * nchunks;
    uint4 *dst = y + (long long)(ko + j) * nchunks;
    for (int c0 = lane; c0 < nchunks; c0 += 32 * kU) {
      uint4 v[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int c = c0 + 32 * u;
        if (c < nchunks) v[u] = ld_nc16(src + c);
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int c = c0 + 32 * u;
        if (c < nchunks) __stcs(dst + c, v[u]);
      }
    }
  }
}

__global__ void __launch_bounds__(kSelectThreads, 1)
    k_select_gather(const SelectArgs a, const int replicas, const int nchunks, uint4 *__restrict__ y) {
  extern __shared__ __align__(16) unsigned char smem[];
  pdl_wait();  // the statistics come from the kernel before this one
  const int b = blockIdx.x / replicas, r = blockIdx.x % replicas;
  const uint16_t *kept = select_image_solo(a, b, smem, r == 0);
  copy_kept(a, b, r, replicas, nchunks, y, kept);
}

// Per device (index & 63): dynamic shared memory limit already raised (bit 0
// k_select, bit 1 k_select_gather, bit 2 k_select_cluster), and the SM count.
// Atomic so that first calls from several host threads are well defined
// (raising the limit twice is harmless).
std::atomic<int> g_smem_set[64];
std::atomic<int> g_sms[64];

}  // namespace

size_t select_smem_bytes(int max_n) {
  const size_t cap = (size_t)row_capacity(max_n > 0 ? max_n : 1);
  return cap * (sizeof(uint32_t) + 3 * sizeof(uint16_t) + sizeof(uint8_t)) + kWarps * 256 * sizeof(uint32_t);
}

// Dynamic shared memory of one CTA per image: both its paths.
size_t solo_smem_bytes(int max_n) {
  const size_t general = select_smem_bytes(max_n);
  return max_n <= kSoloMaxN ? std::max(general, cluster_smem_bytes(max_n > 0 ? max_n : 1, 1)) : general;
}

template <typename K>
cudaError_t raise_smem_limit(K kernel, int dev) {
  int optin = 0;
  cudaError_t err = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (err != cudaSuccess) return err;
  cudaFuncAttributes fa;
  err = cudaFuncGetAttributes(&fa, kernel);
  if (err != cudaSuccess) return err;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
}

// A cluster per image pays from about 5000 tokens on (below, its barriers
// cost more than the split passes save) and while the clusters run at once;
// more CTAs than that only queue, and two pay only where one CTA is left with
// select_image.  Reduction of B images, us with 1 / 2 / 4 / 8 CTAs per image
// (bf16, D 512, K = N / 8):
//   N 2880:  B 1   19.8 / 22.9 / 21.8 / 21.5     B 64  179 / 186 / 201 / 243
//   N 4096:  B 1   23.5 / 26.0 / 23.9 / 23.3     B 16  80.9 / 86.0 / 84.0 / 91.5
//   N 6272:  B 1   32.4 / 32.3 / 28.3 / 26.9     B 12  101 / 104 / 100 / 99.0
//            B 16  122 / 125 / 121 / 129         B 32  205 / 208 / 205 / 230
//   N 8192:  B 1   45.9 / 44.5 / 39.7 / 37.3     B 32  264 / 263 / 258 / 285
//   N 16384: B 1    100 / 72.1 / 58.2 / 51.5     B 16  324 / 282 / 268 / 288
int select_cluster_ctas(int batch, int max_n) {
  if (batch <= 0 || max_n < 5120) return 1;
  if (batch <= 36) return batch <= 12 ? 8 : 4;
  return batch <= 72 && max_n > kSoloMaxN ? 2 : 1;
}

cudaError_t launch_select(const SelectArgs &a, cudaStream_t st, int max_ctas, bool pdl) {
  if (a.batch == 0) return cudaSuccess;
  int dev = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err != cudaSuccess) return err;
  const int c = max_ctas > 0 ? 1 : select_cluster_ctas(a.batch, a.max_n);
  if (c > 1) {
    if (!(g_smem_set[dev & 63].load() & 4)) {
      if ((err = raise_smem_limit(k_select_cluster, dev)) != cudaSuccess) return err;
      g_smem_set[dev & 63].fetch_or(4);
    }
    const size_t need = std::max(cluster_smem_bytes(a.max_n, c), select_smem_bytes(a.max_n));
    return launch_kernel_cluster(k_select_cluster, dim3(a.batch * c), dim3(kSelectThreads), c, need, st, pdl, a, c);
  }
  const size_t smem = solo_smem_bytes(a.max_n);
  if (!(g_smem_set[dev & 63].load() & 1)) {
    if ((err = raise_smem_limit(k_select, dev)) != cudaSuccess) return err;
    g_smem_set[dev & 63].fetch_or(1);
  }
  const int grid = max_ctas > 0 && max_ctas < a.batch ? max_ctas : a.batch;
  return launch_kernel(k_select, dim3(grid), dim3(kSelectThreads), smem, st, pdl, a);
}

int sm_count() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (!g_sms[dev & 63].load()) {
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    g_sms[dev & 63].store(sms);
  }
  return g_sms[dev & 63].load();
}

cudaError_t launch_select_gather(const SelectArgs &a, void *y, cudaStream_t st, bool pdl) {
  if (a.batch == 0) return cudaSuccess;
  int dev = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err != cudaSuccess) return err;
  if (!(g_smem_set[dev & 63].load() & 2)) {
    if ((err = raise_smem_limit(k_select_gather, dev)) != cudaSuccess) return err;
    g_smem_set[dev & 63].fetch_or(2);
  }
  const int sms = sm_count();
  if (sms <= 0) return cudaErrorInvalidDevice;
  const size_t smem = solo_smem_bytes(a.max_n);
  const int nchunks = a.d * elem_bytes(a.dtype) / 16;
  const int replicas = max(1, min(16, sms / a.batch));
  return launch_kernel(k_select_gather, dim3(a.batch * replicas), dim3(kSelectThreads), smem, st, pdl, a, replicas,
                       nchunks, static_cast<uint4 *>(y));
}

}  // namespace tr
