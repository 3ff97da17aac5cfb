// The fast path of the selection, over one CTA or a thread-block cluster of C
// CTAs (2, 4 or 8; large images).  In a cluster CTA r holds rows [r cap,
// (r + 1) cap) of the image, and every pass over the rows is split over the
// cluster.  What select_image does in passes over n rows is, per CTA, a pass
// over n / C rows between cluster barriers:
//
//   keys      range of R and of s over the image (each CTA sends its own to
//             all);
//   Stage I   a histogram of R over kClBuckets value buckets per CTA, summed
//             by every CTA through distributed shared memory, gives the
//             bucket of the K1-th key; the rows of that bucket and of the
//             occupied buckets on either side go to CTA 0, which sorts them,
//             certifies or settles the cut and returns the marks;
//   Stage II  the same histogram of s over X_rem gives each row's bucket
//             start, so each CTA scatters its rows straight to the CTA that
//             owns that stretch of the sorted order; owners rank their
//             buckets, certify their picks (reading neighbours across a
//             boundary from the CTA that has them) and settle their runs;
//   output    kept counts are exchanged and each CTA writes its indices.
//
// Near-ties are settled by the double-float keys, else by exact sums, exactly
// as in tr_select_dev.cuh (of 16384 tokens about one image in six has a pair
// at a pick that only exact sums separate).  What is left to select_image --
// rows outside the fp32 error model, values crowded into one bucket, long or
// very many runs -- is decided by the whole cluster alike (flags exchanged
// before a barrier), and CTA 0 then makes the selection anew.
//
// With one CTA the same code runs without the exchanges (block barriers, plain
// shared memory): the selection of every image up to kSoloMaxN tokens that no
// cluster takes.  It beats select_image's fast path by keeping the s keys from
// the one load of the records, by ranking buckets instead of sorting, and by
// fewer passes: passes of one 576-token fp32 image 17.1 us with select_image
// alone and 13.6 with the fast path before it, tr_select on 64 x 576 tokens 11.8
// and 9.5, on a 2880-token image 20.0 and 15.2.
//
// What bounds it: a chain of about ten short phases, each ending in a cluster
// barrier (0.5-0.6 us) and spending as much on its own latencies; a run to
// settle adds 8-9 us.  6272 tokens, eight CTAs: 27.6 us from the first
// instruction to the last (17 us for 2880 tokens without a run), against 43
// us in one CTA; 16384 tokens 34 us against about 140.
#pragma once

#include "tr_select_dev.cuh"
#include "tr_tc.cuh"

namespace tr {
namespace {

constexpr int kClMax = 8;          // CTAs of a cluster at most
constexpr int kClBuckets = 1024;   // value buckets, two 16-bit counters to a word
constexpr int kClWords = kClBuckets / 2;
static_assert(kClWords == kSelectThreads, "one histogram word per thread");
constexpr int kClWindow = 512;     // rows near the top-K1 cut that CTA 0 sorts
constexpr int kClBucketMax = 256;  // rows of X_rem in one bucket
constexpr int kRunExact = 1 << 30;  // with a run's place in the row list: ranked by exact sums

// Rows per CTA (a multiple of 16), and the sorted stretch a CTA may own.
__host__ __device__ inline int cluster_rows(int max_n, int c) { return ((max_n + c - 1) / c + 15) / 16 * 16; }
__host__ __device__ inline int cluster_slots(int max_n, int c) { return cluster_rows(max_n, c) + kClBucketMax; }
// Dynamic shared memory of the cluster path (also enough for select_image).
__host__ __device__ inline size_t cluster_smem_bytes(int max_n, int c) {
  return (size_t)cluster_rows(max_n, c) * 9 + (size_t)cluster_slots(max_n, c) * 12;
}

// ---------------------------------------------------------------- distributed shared memory
// Barrier over every thread of the cluster (also a block barrier); callable
// from diverged warps.
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ uint32_t ld_cl_u32(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t ld_cl_u16(uint32_t addr) {
  uint16_t v;
  asm volatile("ld.shared::cluster.u16 %0, [%1];" : "=h"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void st_cl_u32(uint32_t addr, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void st_cl_u16(uint32_t addr, uint32_t v) {
  asm volatile("st.shared::cluster.u16 [%0], %1;" ::"r"(addr), "h"((uint16_t)v) : "memory");
}
__device__ __forceinline__ void st_cl_u8(uint32_t addr, uint32_t v) {
  asm volatile("st.shared::cluster.u8 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t atom_cl_add(uint32_t addr, uint32_t v) {
  uint32_t r;
  asm volatile("atom.shared::cluster.add.u32 %0, [%1], %2;" : "=r"(r) : "r"(addr), "r"(v) : "memory");
  return r;
}

// The two halves of the barrier.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// Phases whose failure (anything the fast path leaves to select_image) is
// exchanged; each has its own flag, set before a barrier and read after it.
enum { kFailKeys = 0, kFailCut = 1, kFailPicks = 2, kFailPhases = 3 };

struct ClusterShared {
  float4 range[kClMax];            // per CTA: min, max of -R; min, max of s
  uint32_t fail[kFailPhases];
  uint32_t kept[kClMax];           // per CTA: kept rows
  uint32_t hist_r[kClWords], hist_s[kClWords];  // this CTA's rows per bucket, two 16-bit counts a word
  uint32_t start[kClBuckets + 1];  // sorted position where a bucket of s begins
  uint32_t base[kClBuckets];       // next sorted position for a row of this CTA's in the bucket
  int own[kClMax + 1];             // CTA c owns sorted positions [own[c], own[c + 1])
  int bucket[3], before, flag;
  // CTA 0: the rows near the cut
  uint32_t win_key[kClWindow];
  uint16_t win_row[kClWindow], win_ord[kClWindow];
  uint32_t win_count;
  int lo, hi;
  float wr[kWarps][4];
  // runs around picks (RunPlace, where this CTA's rows are few)
  uint32_t run[kMaxRuns];
  int first[kMaxRuns];
  int runs, run_rows, exact_rows, exact_total;
  uint16_t list[kPendCap], xlist[kPendCap];
  alignas(16) unsigned long long scratch[kSelectThreads];
};

// Double-float keys of rows[0..cnt) (mode 0: R, 1: s) into their records, up
// to four rows at a time by groups of warps.  A row that does not qualify gets
// a NaN key, which compares as undecided with any other, so its run, and no
// other, is left open.  Called by the whole block; ends with a barrier.
__device__ __noinline__ void refine_df(const SelectArgs &a, long long off, const uint16_t *rows, int cnt, int mode,
                                       ExactRec *rec) {
  __shared__ PartDf pdf;
  const int groups = cnt >= 4 ? 4 : (cnt >= 2 ? 2 : 1);
  const int gsize = (int)blockDim.x / groups;
  const int gi = (int)threadIdx.x / gsize;
  const Group g{gi * gsize, gsize, 1 + gi};
  for (int base = 0; base < cnt; base += groups)
    if (base + gi < cnt) {
      const int row = rows[base + gi];
      if (!df_row_any(a, off + row, mode, rec + row, pdf, g) && g.tid() == 0)
        (mode == 0 ? rec[row].r_hi : rec[row].s_hi) = __int_as_float(0x7fc00000);
    }
  __syncthreads();
}

// Exact sums of rows[0..cnt) into their records, in the same way, with the H2
// (mode 0) or s (mode 1) outputs rewritten from them; false (block-uniform)
// when a row's sums do not fit the exact representation.
__device__ __noinline__ bool refine_exact(const SelectArgs &a, long long off, const uint16_t *rows, int cnt, int mode,
                                          ExactRec *rec, const bool primary) {
  __shared__ Part128 part;
  const int groups = cnt >= 4 ? 4 : (cnt >= 2 ? 2 : 1);
  const int gsize = (int)blockDim.x / groups;
  const int gi = (int)threadIdx.x / gsize;
  const Group g{gi * gsize, gsize, 1 + gi};
  for (int base = 0; base < cnt; base += groups)
    if (base + gi < cnt) {
      const int row = rows[base + gi];
      exact_row_any(a, off + row, mode, a.stats + (off + row) * TR_STATS_WORDS, rec + row, part, g);
    }
  __syncthreads();
  bool ok = true;
  for (int i = threadIdx.x; i < cnt; i += blockDim.x) {
    const ExactRec &r = rec[rows[i]];
    const bool fine = (mode == 0 ? r.flags_l : r.flags_s) == 0u;
    ok &= fine;
    if (fine && primary && mode == 0 && a.h2) a.h2[off + rows[i]] = exact_h2(r);
    if (fine && primary && mode == 1 && a.s) a.s[off + rows[i]] = exact_s_key(r);
  }
  return !__syncthreads_or(!ok);
}

// What a CTA knows of its image, and the cluster's memory: with kMany = false
// one CTA has the image to itself.
template <bool kMany>
struct SplitImage {
  long long off;
  int n, k, k1, k2, ko;
  int c, rank;            // CTAs of the cluster, this one
  int cap, first, rows;   // rows per CTA; this CTA's first row and number of rows
  bool primary;           // writes the outputs
  uint32_t *keyr, *keys, *sk, *sk2;
  uint16_t *sr, *sr2;
  uint8_t *fl;
  ExactRec *rec;
  static __device__ __forceinline__ void barrier() {
    if (kMany)
      cluster_barrier();
    else
      __syncthreads();
  }
  static __device__ __forceinline__ uint32_t at(const void *p, int cta) {
    return tc::map_shared(tc::smem_u32(p), (uint32_t)cta);
  }
  // *p in CTA `cta`
  static __device__ __forceinline__ void put(uint32_t *p, int cta, uint32_t v) {
    if (kMany)
      st_cl_u32(at(p, cta), v);
    else
      *p = v;
  }
  static __device__ __forceinline__ void put(uint16_t *p, int cta, uint32_t v) {
    if (kMany)
      st_cl_u16(at(p, cta), v);
    else
      *p = (uint16_t)v;
  }
  static __device__ __forceinline__ uint32_t add(uint32_t *p, int cta, uint32_t v) {
    return kMany ? atom_cl_add(at(p, cta), v) : atomicAdd(p, v);
  }
  __device__ __forceinline__ int ctas() const { return kMany ? c : 1; }
  // marks image row `row` in its CTA's flags
  __device__ __forceinline__ void mark(int row, uint32_t f) const {
    if (kMany) {
      const int o = row / cap;
      st_cl_u8(at(fl + (row - o * cap), o), f);
    } else {
      fl[row] = (uint8_t)f;
    }
  }
};

// Sums the cluster's histogram word `w` (this thread's two buckets) over the
// CTAs; *mine: the part of the CTAs before this one.
template <bool kMany>
__device__ __forceinline__ uint32_t sum_words(const SplitImage<kMany> &im, const uint32_t *hist, int w,
                                              uint32_t *mine) {
  if (!kMany) {
    *mine = 0u;
    return hist[w];
  }
  const uint32_t local = tc::smem_u32(hist + w);
  uint32_t v[kClMax], total = 0u, before = 0u;
#pragma unroll
  for (int o = 0; o < kClMax; ++o) v[o] = o < im.c ? ld_cl_u32(tc::map_shared(local, (uint32_t)o)) : 0u;
#pragma unroll
  for (int o = 0; o < kClMax; ++o) {
    total += v[o];
    if (o < im.rank) before += v[o];
  }
  *mine = before;
  return total;
}

// Bucket of an importance key (value -R) or consistency key (value s).
struct BucketMap {
  float vmin, scale;
  bool complemented;
  __device__ __forceinline__ int operator()(uint32_t key) const {
    return min(kClBuckets - 1, max(0, (int)((key_value(key, complemented) - vmin) * scale)));
  }
};
__device__ __forceinline__ bool bucket_map(float vmin, float vmax, bool complemented, BucketMap &m) {
  const float span = vmax - vmin;
  m.vmin = vmin;
  m.scale = (float)kClBuckets / span;
  m.complemented = complemented;
  return span > 0.f && isfinite(span) && isfinite(m.scale);
}

// Stage I across the cluster; marks X_imp in the rows' flags.  False
// (cluster-uniform) when it is left to select_image.  On return the marks of
// every CTA are in place.
template <bool kMany>
__device__ __forceinline__ bool cluster_stage_one(const SelectArgs &a, const SplitImage<kMany> &im, ClusterShared &sh,
                                                  float vmin, float vmax) {
  const int tid = threadIdx.x, nthr = blockDim.x;
  BucketMap map;
  if (!bucket_map(vmin, vmax, true, map)) return false;  // the same in every CTA
  for (int i = tid; i < im.rows; i += nthr) {
    const int b = map(im.keyr[i]);
    atomicAdd(&sh.hist_r[b >> 1], 1u << (16 * (b & 1)));
  }
  im.barrier();
  uint32_t unused;
  const uint32_t w = sum_words(im, sh.hist_r, tid, &unused);
  const int c0 = (int)(w & 0xffffu), c1 = (int)(w >> 16);
  int total = 0;
  const int pre = block_exclusive_scan(c0 + c1, &total);
  // the occupied buckets holding positions k1 - 1, and the last before and the
  // first after that bucket
  if (tid < 3) sh.bucket[tid] = -1;
  __syncthreads();
  auto holds = [&](int pos, int slot, bool set_before) {
    if (pos >= pre && pos < pre + c0 + c1) {
      const bool second = pos >= pre + c0;
      sh.bucket[slot] = 2 * tid + (second ? 1 : 0);
      if (set_before) {
        sh.before = pre + (second ? c0 : 0);  // rows before the bucket
        sh.flag = second ? c1 : c0;           // rows in it
      }
    }
  };
  holds(im.k1 - 1, 1, true);
  __syncthreads();
  const int before = sh.before, count = sh.flag;
  __syncthreads();
  holds(before - 1, 0, false);
  holds(before + count, 2, false);
  __syncthreads();
  const int bl = sh.bucket[0], bm = sh.bucket[1], bh = sh.bucket[2];
  // rows of the window: from bucket bl (or bm) to bucket bh (or bm)
  const int wlo = bl >= 0 ? bl : bm, whi = bh >= 0 ? bh : bm;
  int in0 = (2 * tid >= wlo && 2 * tid <= whi) ? c0 : 0, in1 = (2 * tid + 1 >= wlo && 2 * tid + 1 <= whi) ? c1 : 0;
  int lt0 = 2 * tid < wlo ? c0 : 0, lt1 = 2 * tid + 1 < wlo ? c1 : 0;
  int both = 0;  // each total is at most n < 2^16
  block_exclusive_scan((in0 + in1) | ((lt0 + lt1) << 16), &both);
  const int len = both & 0xffff, n_lt = (int)((unsigned)both >> 16);
  if (len > kClWindow) return false;  // the same in every CTA
  for (int i = tid; i < im.rows; i += nthr) {
    const uint32_t key = im.keyr[i];
    const int b = map(key);
    if (b < wlo) {
      im.fl[i] = F_IMP;  // R above the whole window's
    } else if (b <= whi) {
      const uint32_t slot = im.add(&sh.win_count, 0, 1u);
      if (slot < (uint32_t)kClWindow) {
        im.put(&sh.win_key[slot], 0, key);
        im.put(&sh.win_row[slot], 0, (uint32_t)(im.first + i));
      }
    }
  }
  im.barrier();
  if (im.rank == 0) {
    // sorted by key (equal keys in any order: they are never certified)
    for (int i = tid; i < len; i += nthr) sh.win_ord[i] = (uint16_t)i;
    __syncthreads();
    if (len <= kCountSortMax)
      sort_count(sh.win_key, sh.win_ord, len, sh.scratch);
    else
      sort_small<1>(sh.win_key, sh.win_ord, len, sh.scratch);
    // the uncertain run around position p, as in resolve_cut
    const int p = im.k1 - n_lt;
    if (tid == 0) {
      sh.lo = 0;
      sh.hi = len;
    }
    __syncthreads();
    int my_lo = 0, my_hi = len;
    for (int q = 1 + tid; q < len; q += nthr)
      if (cert_r(sh.win_key, sh.win_ord, q, a.bounds)) {
        if (q <= p) my_lo = q;
        if (q >= p && my_hi == len) my_hi = q;
      }
    if (my_lo > 0) atomicMax(&sh.lo, my_lo);
    if (my_hi < len) atomicMin(&sh.hi, my_hi);
    __syncthreads();
    const int lo = sh.lo, hi = sh.hi;
    // a run that may go on outside the window, or is long, is left to select_image
    bool ok = p >= 1 && p < len && !(lo == 0 && n_lt > 0 && hi > lo) && !(hi == len && n_lt + len < im.n && hi > lo) &&
              hi - lo <= kDfRunMax;
    if (ok) {  // uniform
      for (int q = tid; q < lo; q += nthr) im.mark(sh.win_row[sh.win_ord[q]], F_IMP);
      if (hi > lo) {
        for (int q = lo + tid; q < hi; q += nthr) sh.list[q - lo] = sh.win_row[sh.win_ord[q]];
        __syncthreads();
        const int len = hi - lo;
        refine_df(a, im.off, sh.list, len, 0, im.rec);
        bool open = false;
        int rank = 0;
        if (tid < len)
          for (int j = 0; j < len; ++j) {
            if (j == tid) continue;
            const int c = df_cmp_r(im.rec[sh.list[j]], im.rec[sh.list[tid]], a.bounds);
            open |= c == 0;
            rank += c > 0;
          }
        if (__syncthreads_or(open)) {
          ok = refine_exact(a, im.off, sh.list, len, 0, im.rec, im.primary);
          rank = 0;
          if (ok && tid < len) {
            const int r = sh.list[tid];
            for (int j = 0; j < len; ++j) {
              if (j == tid) continue;
              const int c = cmp_r(im.rec[sh.list[j]], im.rec[r]);
              rank += c > 0 || (c == 0 && sh.list[j] < r);
            }
          }
          if (tid == 0) sh.exact_total += len;
        }
        if (ok && tid < len && n_lt + lo + rank < im.k1) im.mark(sh.list[tid], F_IMP);
        __syncthreads();
      }
    }
    if (!ok && tid < im.ctas()) im.put(&sh.fail[kFailCut], tid, 1u);
  }
  im.barrier();
  return sh.fail[kFailCut] == 0u;
}

// Where a CTA lists the runs around its picks: [lo, hi) packed, the place of
// their rows in the list, the list, and that of the rows for exact sums.  A CTA
// with many rows lists them in the memory of its R keys, which Stage I was the
// last to read (half of it is taken): an eighth as many runs as rows, and twice
// as many rows of runs.  Keys of a narrow band have some hundred near-ties at
// one pick in two (8192 tokens of 1544 channels, half of them kept: 191 runs),
// and an image with more runs than are listed is selected anew by select_image.
constexpr int kWideRows = 2048;
struct RunPlace {
  uint32_t *run;
  int *first;
  uint16_t *list, *xlist;
  int max_runs, max_rows;
};
// Out of line and asked for only where a run is: inlined ahead of the picks it
// took 0.2 us of a 576-token image's 13.3, runs or none.
__device__ __noinline__ RunPlace run_place(uint32_t *keyr, int cap, ClusterShared &sh) {
  if (cap < kWideRows) return RunPlace{sh.run, sh.first, sh.list, sh.xlist, kMaxRuns, kPendCap};
  const int w = cap / 8;
  uint16_t *list = reinterpret_cast<uint16_t *>(keyr + 2 * w);
  return RunPlace{keyr, reinterpret_cast<int *>(keyr + w), list, list + 2 * w, w, 2 * w};
}

// Element q of X_rem sorted by s, wherever it is.
struct SortedRow {
  float s;
  int row;
};
template <bool kMany>
__device__ __forceinline__ SortedRow sorted_row(const SplitImage<kMany> &im, const ClusterShared &sh, int q) {
  if (!kMany) return SortedRow{unord32(im.sk2[q]), im.sr2[q]};
  int o = im.rank;
  if (q < sh.own[o] || q >= sh.own[o + 1]) {
    o = 0;
    while (q >= sh.own[o + 1]) ++o;
  }
  const int i = q - sh.own[o];
  if (o == im.rank) return SortedRow{unord32(im.sk2[i]), im.sr2[i]};
  return SortedRow{unord32(ld_cl_u32(im.at(im.sk2 + i, o))), (int)ld_cl_u16(im.at(im.sr2 + i, o))};
}
// Cut between sorted positions q - 1 and q certain (as cert_s).
template <bool kMany>
__device__ __forceinline__ bool cluster_cert_s(const SplitImage<kMany> &im, const ClusterShared &sh, int q,
                                               const Bounds &bd) {
  const float sa = sorted_row(im, sh, q - 1).s, sb = sorted_row(im, sh, q).s;
  const float hi_a = __fadd_ru(sa, __fmaf_ru(bd.s_rel, fabsf(sa), bd.s_abs));
  const float lo_b = __fsub_rd(sb, __fmaf_ru(bd.s_rel, fabsf(sb), bd.s_abs));
  return lo_b > hi_a;
}

// Stage II across the cluster: marks X_div.  False (cluster-uniform) when it
// is left to select_image.
template <bool kMany>
__device__ __forceinline__ bool cluster_stage_two(const SelectArgs &a, const SplitImage<kMany> &im, ClusterShared &sh,
                                                  float vmin, float vmax, int slots) {
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int m = im.n - im.k1, t = max(1, m / im.k2);
  BucketMap map;
  if (!bucket_map(vmin, vmax, false, map)) return false;
  for (int i = tid; i < im.rows; i += nthr)
    if (!(im.fl[i] & F_IMP)) {
      const int b = map(im.keys[i]);
      atomicAdd(&sh.hist_s[b >> 1], 1u << (16 * (b & 1)));
    }
  const int nc = im.ctas();
  if (tid <= nc) sh.own[tid] = tid < nc && !kMany ? 0 : m;
  im.barrier();
  uint32_t mine;
  const uint32_t w = sum_words(im, sh.hist_s, tid, &mine);
  const int c0 = (int)(w & 0xffffu), c1 = (int)(w >> 16);
  int total = 0;
  const int pre = block_exclusive_scan(c0 + c1, &total);
  sh.start[2 * tid] = (uint32_t)pre;
  sh.start[2 * tid + 1] = (uint32_t)(pre + c0);
  sh.base[2 * tid] = (uint32_t)pre + (mine & 0xffffu);
  sh.base[2 * tid + 1] = (uint32_t)(pre + c0) + (mine >> 16);
  if (tid == 0) sh.start[kClBuckets] = (uint32_t)m;
  // a bucket belongs to the CTA whose m / C stretch its start lies in
  if (kMany && c0) atomicMin(&sh.own[pre * nc / m], pre);
  if (kMany && c1) atomicMin(&sh.own[(pre + c0) * nc / m], pre + c0);
  if (__syncthreads_or(max(c0, c1) > kClBucketMax)) return false;  // the same in every CTA
  if (kMany) {
    if (tid == 0)
      for (int o = nc - 1; o >= 0; --o) sh.own[o] = min(sh.own[o], sh.own[o + 1]);
    __syncthreads();
  }
  for (int i = tid; i < im.rows; i += nthr)
    if (!(im.fl[i] & F_IMP)) {
      const uint32_t key = im.keys[i];
      const int b = map(key);
      const int o = kMany ? (int)sh.start[b] * nc / m : 0;
      const int at = (int)atomicAdd(&sh.base[b], 1u) - sh.own[o];
      if (at < slots) {  // always: a stretch is at most m / C + kClBucketMax rows
        im.put(im.sk + at, o, key);
        im.put(im.sr + at, o, (uint32_t)(im.first + i));
      }
    }
  im.barrier();
  const int q0 = sh.own[im.rank], q1 = sh.own[im.rank + 1];
  for (int i = tid; i < q1 - q0; i += nthr) {
    const uint32_t key = im.sk[i];
    const uint16_t row = im.sr[i];
    const int b = map(key);
    const int lo = (int)sh.start[b] - q0, hi = (int)sh.start[b + 1] - q0;
    const unsigned long long kk = ((unsigned long long)key << 16) | row;
    int rank = 0;
    for (int j = lo; j < hi; ++j) rank += (((unsigned long long)im.sk[j] << 16) | im.sr[j]) < kk;
    im.sk2[lo + rank] = key;
    im.sr2[lo + rank] = row;
  }
  im.barrier();
  // the picks inside this CTA's stretch
  bool bad = false, marked = false;
  for (int j = tid; j < im.k2; j += nthr) {
    const int p = pick_position(j, m, im.k2, t, a.stride_interval);
    if (p < q0 || p >= q1) continue;
    const bool cut0 = p == 0 || cluster_cert_s(im, sh, p, a.bounds);
    const bool cut1 = p + 1 >= m || cluster_cert_s(im, sh, p + 1, a.bounds);
    if (cut0 && cut1) {
      im.mark(im.sr2[p - q0], F_DIV);
      continue;
    }
    int lo = p, hi = p + 1;
    while (lo > 0 && hi - lo <= kDfRunMax && !cluster_cert_s(im, sh, lo, a.bounds)) --lo;
    while (hi < m && hi - lo <= kDfRunMax && !cluster_cert_s(im, sh, hi, a.bounds)) ++hi;
    if (hi - lo > kDfRunMax) {
      bad = true;
      continue;
    }
    marked = true;
    // every pick inside a run finds the same run; the first one records it
    if (j == 0 || pick_position(j - 1, m, im.k2, t, a.stride_interval) < lo) {
      const RunPlace place = run_place(im.keyr, im.cap, sh);
      const int slot = atomicAdd(&sh.runs, 1);
      const int at = atomicAdd(&sh.run_rows, hi - lo);
      if (slot < place.max_runs && at + (hi - lo) <= place.max_rows) {
        place.run[slot] = ((uint32_t)lo << 16) | (uint32_t)hi;
        place.first[slot] = at;
        for (int q = lo; q < hi; ++q) place.list[at + q - lo] = (uint16_t)sorted_row(im, sh, q).row;
      } else {
        bad = true;
      }
    }
  }
  bad = __syncthreads_or(bad) != 0;
  if (__syncthreads_or(marked) && !bad) {
    const int runs = sh.runs;
    const RunPlace place = run_place(im.keyr, im.cap, sh);
    // a run that the double-float keys leave open anywhere (a pair they do not
    // separate, or a row that does not qualify) is ranked by exact sums as a whole
    if (runs > 0) refine_df(a, im.off, place.list, sh.run_rows, 1, im.rec);
    for (int r = tid; r < runs; r += nthr) {
      const int len = (int)(place.run[r] & 0xffffu) - (int)(place.run[r] >> 16);
      const uint16_t *rows = place.list + place.first[r];
      bool open = false;
      for (int i = 0; i < len && !open; ++i)
        for (int j = i + 1; j < len && !open; ++j) open = df_cmp_s(im.rec[rows[j]], im.rec[rows[i]], a.bounds) == 0;
      if (open) {
        const int at = atomicAdd(&sh.exact_rows, len);
        for (int i = 0; i < len; ++i) place.xlist[at + i] = rows[i];
        place.first[r] |= kRunExact;
      }
    }
    __syncthreads();
    if (sh.exact_rows > 0) bad = !refine_exact(a, im.off, place.xlist, sh.exact_rows, 1, im.rec, im.primary);
    if (!bad) {
      for (int r = tid; r < runs; r += nthr) {
        const int lo = (int)(place.run[r] >> 16), len = (int)(place.run[r] & 0xffffu) - lo;
        const bool exact = (place.first[r] & kRunExact) != 0;
        const uint16_t *rows = place.list + (place.first[r] & ~kRunExact);
        for (int i = 0; i < len; ++i) {
          int rank = 0;
          for (int j = 0; j < len; ++j) {
            if (j == i) continue;
            const int c = exact ? cmp_s(im.rec[rows[j]], im.rec[rows[i]])
                                : df_cmp_s(im.rec[rows[j]], im.rec[rows[i]], a.bounds);
            rank += c < 0 || (c == 0 && rows[j] < rows[i]);
          }
          if (is_pick(lo + rank, m, im.k2, t, a.stride_interval)) im.mark(rows[i], F_DIV);
        }
      }
    }
    if (tid == 0) sh.exact_total += sh.exact_rows;
  }
  if (bad && tid < im.ctas()) im.put(&sh.fail[kFailPicks], tid, 1u);
  im.barrier();
  return sh.fail[kFailPicks] == 0u;
}

// Selection of image b by a cluster of c CTAs (kMany; this one: rank) or by
// this CTA.  False (cluster-uniform, nothing written) when the image is left
// to select_image: another barrier is then due before a CTA's shared memory is
// reused or gone.  Only a primary CTA writes outputs; *kept (one CTA): the kept
// local indices in shared memory.
template <bool kMany>
__device__ bool select_image_cluster(const SelectArgs &a, const int b, const int c, const int rank,
                                     unsigned char *smem, const bool primary, const uint16_t **kept) {
  __shared__ ClusterShared sh;
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5;
  SplitImage<kMany> im;
  if (a.cu_seqlens) {
    im.off = a.cu_seqlens[b];
    im.n = a.cu_seqlens[b + 1] - a.cu_seqlens[b];
  } else {
    im.off = (long long)b * a.n_uniform;
    im.n = a.n_uniform;
  }
  im.k = a.k[b];
  im.k1 = a.k1[b];
  // what select_image refuses or skips, it also reports (cluster-uniform)
  if (im.n <= 0 || im.n > a.max_n || im.off < 0 || im.off + im.n > a.total_rows || im.k < 0 || im.k > im.n ||
      im.k1 < 0 || im.k1 > im.k)
    return false;
  im.k2 = im.k - im.k1;
  im.ko = a.cu_k[b];
  im.c = c;
  im.rank = kMany ? rank : 0;
  im.primary = primary;
  im.cap = cluster_rows(a.max_n, c);
  im.first = im.rank * im.cap;
  im.rows = max(0, min(im.cap, im.n - im.first));
  const int slots = cluster_slots(a.max_n, c);
  im.keyr = reinterpret_cast<uint32_t *>(smem);
  im.keys = im.keyr + im.cap;
  im.sk = im.keys + im.cap;
  im.sk2 = im.sk + slots;
  im.sr = reinterpret_cast<uint16_t *>(im.sk2 + slots);
  im.sr2 = im.sr + slots;
  im.fl = reinterpret_cast<uint8_t *>(im.sr2 + slots);
  im.rec = a.exact + im.off;
  for (int i = tid; i < kClWords; i += nthr) sh.hist_r[i] = sh.hist_s[i] = 0u;
  if (tid < kFailPhases) sh.fail[tid] = 0u;
  if (tid == 0) {
    sh.win_count = 0u;
    sh.runs = sh.run_rows = sh.exact_rows = sh.exact_total = 0;
  }
  if (kMany) cluster_arrive();  // this CTA runs and has its counters cleared
  const bool need_r = im.k1 > 0 && im.k1 < im.n, need_s = im.k2 > 0;
  const float *st = a.stats + (im.off + im.first) * TR_STATS_WORDS;
  float4 range = make_float4(INFINITY, -INFINITY, INFINITY, -INFINITY);
  bool bad = false;
  for (int i0 = tid; i0 < im.rows; i0 += kKeyIlp * nthr) {
    float2 kk[kKeyIlp];
#pragma unroll
    for (int u = 0; u < kKeyIlp; ++u) {
      const int i = i0 + u * nthr;
      kk[u] = i < im.rows ? key_rs(st + (long long)i * TR_STATS_WORDS) : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < kKeyIlp; ++u) {
      const int i = i0 + u * nthr;
      if (i < im.rows) {
        bad |= ((need_r || a.h2) && isnan(kk[u].x)) || ((need_s || a.s) && isnan(kk[u].y));
        im.fl[i] = im.k1 == im.n ? F_IMP : 0;
        im.keyr[i] = ~ord32(kk[u].x);
        im.keys[i] = ord32(kk[u].y);
        range.x = fminf(range.x, -kk[u].x);
        range.y = fmaxf(range.y, -kk[u].x);
        range.z = fminf(range.z, kk[u].y);
        range.w = fmaxf(range.w, kk[u].y);
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    range.x = fminf(range.x, __shfl_xor_sync(0xffffffffu, range.x, o));
    range.y = fmaxf(range.y, __shfl_xor_sync(0xffffffffu, range.y, o));
    range.z = fminf(range.z, __shfl_xor_sync(0xffffffffu, range.z, o));
    range.w = fmaxf(range.w, __shfl_xor_sync(0xffffffffu, range.w, o));
  }
  if (lane == 0) {
    sh.wr[warp][0] = range.x;
    sh.wr[warp][1] = range.y;
    sh.wr[warp][2] = range.z;
    sh.wr[warp][3] = range.w;
  }
  bad = __syncthreads_or(bad) != 0;
  if (kMany) cluster_wait();  // and so do the others: their shared memory may be written
  if (tid < im.ctas()) {
    range = make_float4(INFINITY, -INFINITY, INFINITY, -INFINITY);
    for (int w = 0; w < kWarps; ++w) {
      range.x = fminf(range.x, sh.wr[w][0]);
      range.y = fmaxf(range.y, sh.wr[w][1]);
      range.z = fminf(range.z, sh.wr[w][2]);
      range.w = fmaxf(range.w, sh.wr[w][3]);
    }
    if (kMany)
      tc::st_cluster_v4(im.at(&sh.range[rank], tid), __float_as_uint(range.x), __float_as_uint(range.y),
                        __float_as_uint(range.z), __float_as_uint(range.w));
    else
      sh.range[0] = range;
    if (bad) im.put(&sh.fail[kFailKeys], tid, 1u);
  }
  im.barrier();
  if (sh.fail[kFailKeys]) return false;
  range = sh.range[0];
  for (int o = 1; o < im.ctas(); ++o) {
    const float4 v = sh.range[o];
    range.x = fminf(range.x, v.x);
    range.y = fmaxf(range.y, v.y);
    range.z = fminf(range.z, v.z);
    range.w = fmaxf(range.w, v.w);
  }
  if (need_r && !cluster_stage_one(a, im, sh, range.x, range.y)) return false;
  if (need_s && !cluster_stage_two(a, im, sh, range.z, range.w, slots)) return false;
  // kept rows in ascending order: this CTA's are one stretch of the output
  const int per = (im.rows + nthr - 1) / nthr;
  const int i0 = min(im.rows, tid * per), i1 = min(im.rows, i0 + per);
  int cnt = 0;
  for (int i = i0; i < i1; ++i) cnt += (im.fl[i] & (F_IMP | F_DIV)) != 0;
  int total = 0;
  int pos = block_exclusive_scan(cnt, &total);
  int all = total;
  if (kMany) {
    if (tid < c) im.put(&sh.kept[rank], tid, (uint32_t)total);
    im.barrier();
    all = 0;
    for (int o = 0; o < c; ++o) {
      if (o < rank) pos += (int)sh.kept[o];
      all += (int)sh.kept[o];
    }
  }
  for (int i = i0; i < i1; ++i) {
    const uint8_t f = im.fl[i];
    if ((f & (F_IMP | F_DIV)) && pos < im.k) {  // never past this image's slots
      if (primary) a.idx[im.ko + pos] = im.first + i;
      if (!kMany) im.sr[pos] = (uint16_t)i;
      ++pos;
    }
    if (primary && a.role) a.role[im.off + im.first + i] = (f & F_IMP) ? 1 : ((f & F_DIV) ? 2 : 0);
  }
  if (tid == 0 && primary && a.status) {
    if (im.rank == 0 && all != im.k) atomicAdd(&a.status[3], 1);
    if (sh.exact_total) atomicAdd(&a.status[2], sh.exact_total);
  }
  if (!kMany) {
    *kept = im.sr;
    __syncthreads();  // the list is complete, and the arrays may serve the next image
  }
  return true;
}

// Images up to this size take the fast path in one CTA (its arrays fit beside
// what select_image needs).
constexpr int kSoloMaxN = 8192;

// The selection of image b by this CTA; returns the kept local indices in
// shared memory.
__device__ __forceinline__ const uint16_t *select_image_solo(const SelectArgs &a, const int b, unsigned char *smem,
                                                             const bool primary) {
  const uint16_t *kept = kept_rows(a, smem);
  if (a.max_n <= kSoloMaxN) {
    if (select_image_cluster<false>(a, b, 1, 0, smem, primary, &kept)) return kept;
    __syncthreads();
  }
  select_image(a, b, smem, primary);
  return kept_rows(a, smem);
}

}  // namespace
}  // namespace tr
