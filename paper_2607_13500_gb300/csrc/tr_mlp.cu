// The vision encoder's final-layer MLP, x'' = W2 sigma(W1 x') (Eq. 5), on
// the 5th-generation tensor cores, with ALTR's token scoring (Eq. 3-4 and
// Eq. 6) fused into the epilogue of its second GEMM.
//
// The paper takes x' and x'' from the encoder's forward pass "at no extra
// cost" (Section IV-B).  Here the second GEMM's epilogue, which produces
// x'' anyway, rounds each element to bf16, stores it, forms the block
// output x = bf16(resid + x'') and accumulates the five row sums of the
// selection -- L1 = sum|x|, S2 = sum x^2, A = sum x'^2, B = sum x''^2,
// P = sum x'x'' -- from the stored values, so a separate scoring pass over
// x, x', x'' is not needed and the selection stays a function of the stored
// tensors.  The row records it writes are the ones tr_score writes.
//
// One kernel serves both GEMMs (C[m, n] = A[m, k] B[n, k]^T, bf16 operands,
// fp32 accumulation): a persistent grid of one CTA per SM, in pairs, walks
// output tiles of 256 rows x bn columns, bn 64 to 256 by size (gemm_shape;
// tile t: row block t / n_tiles, column block t % n_tiles, so the pairs
// running at one time share row blocks of A in L2).  Per CTA:
//   warp 0      TMA producer: A and B k-blocks (64 wide, 128-byte swizzle)
//               into a 6-stage shared-memory ring;
//   warp 1      allocates 512 TMEM columns (two fp32 accumulators of 128 rows
//               and up to 256 columns); in the pair's even CTA it issues
//               tcgen05.mma (M 256, N bn, K 16) from one thread, committing
//               each stage back to the producers and each finished
//               accumulator to the epilogues;
//   warps 2-    epilogue: one thread per accumulator row (TMEM lane: a
//               warp reads the lane quarter warp % 4); the tile's bn / 32
//               blocks of 32 columns are dealt to the two or four warps of
//               each quarter in turn.  Outputs leave through TMA stores of
//               32 x 32 blocks staged in shared memory; the score mode's x'
//               and residual come in the same way.
// K is summed in one order whatever the number of rows, the tile width and the
// mode, so a row's outputs do not depend on the batch it is in.
// The projector mode (tr_project_kept) is the hidden GEMM with its A rows
// gathered: A row j is token idx[j] of the image that owns kept slot j, so
// the first projector layer reads X* = X_imp union X_div (Eq. 7) straight
// from x without a gathered copy.  It runs 8 epilogue warps, and four more
// (10-13) bring those rows with TMA tile::gather4 loads (four 64-element rows
// of x by index, one-row box, 128-byte swizzle -- the rows land in the layout
// the tensor cores read: the swizzle follows the shared-memory address); a
// group with a row past the kept slots (or a k-block past x's columns) takes
// four one-row tiled loads instead, an outside row at coordinate -1, which
// reads zeros.
//
// The epilogue of tile i overlaps the main loop of tile i + 1 (two TMEM
// accumulators).  It does its fp32 arithmetic on packed pairs (add / mul /
// fma.f32x2, one instruction per two columns).
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>
#include <climits>
#include <mutex>

#include "tr_internal.cuh"
#include "tr_record.cuh"
#include "tr_tc.cuh"

namespace tr {
namespace {

constexpr int kBM = 128, kBN = 256, kBK = 64;  // a CTA's rows, a tile's columns at most, a k-block
enum { kModeHidden = 0, kModeScore = 1, kModeProject = 2 };
// Epilogue warps per mode: four per lane quarter for the hidden GEMM, whose
// main loop is short, so that they hide the latencies of one another's TMEM
// loads and arithmetic; two for the score GEMM (64 images x 576 tokens, D
// 1024, hidden 4096, both GEMMs: 437 us, with four 446 us -- the main loop
// covers this epilogue, and the staging it saves is a sixth operand stage) and
// for the projector, whose threads include its row loaders.
__host__ __device__ constexpr int epi_warps(int mode) { return mode == kModeHidden ? 16 : 8; }
__host__ __device__ constexpr int epi_parts(int mode) { return epi_warps(mode) / 4; }
// producer, MMA issuer, epilogue (+ the A-row loader warps of the projector mode)
constexpr int kLoadWarps = 4;  // projector: loader warps, 32 of a CTA's 128 rows each
__host__ __device__ constexpr int gemm_threads(int mode) {
  return 64 + 32 * epi_warps(mode) + (mode == kModeProject ? 32 * kLoadWarps : 0);
}
constexpr int kTmemCols = 2 * kBN;                // two accumulators
constexpr int kPartWords = 10;                    // hi, lo of L1, S2, A, B, P
// The epilogue's unit: a block of 32 rows (one warp's TMEM lanes) x 32
// columns in bf16, 2 KiB with 64-byte rows and the 64-byte swizzle (16-byte
// unit u of row r at r * 64 + ((u ^ (r / 2 % 4)) << 4): the 32 lanes' 16-byte
// accesses take the fewest shared-memory wavefronts).
constexpr int kBlk = 32;
constexpr int kBlkBytes = 32 * kBlk * 2;
// Staging per epilogue warp: the output block (the projector's warps two of
// them); the score mode's blocks of x' and of the residual, loaded by TMA
// ahead of their use and overwritten in place by x'' and x.
__host__ __device__ constexpr int stage_blks(int mode) { return mode == kModeHidden ? 1 : 2; }
__host__ __device__ constexpr int stage_bytes(int mode) { return stage_blks(mode) * kBlkBytes; }
// The score mode's partial row sums per tile and lane quarter: one for each of
// its warps, of an equal share of the tile's blocks.  certification_bounds
// counts on these numbers.
constexpr int kRowParts = kMlpRowParts;
constexpr int kWidths[] = {kMlpMaxColumns, 192, 128, kMlpMinColumns};  // a tile's columns
static_assert(kRowParts == epi_parts(kModeScore) && kBN == kMlpMaxColumns, "layout of the row partials");
static_assert(kWidths[1] % (kRowParts * kBlk) == 0 && kWidths[2] % (kRowParts * kBlk) == 0 &&
                  kMlpMinColumns == kRowParts * kBlk,
              "equal shares of every tile's blocks");

struct GemmArgs {
  int m, n, k;          // C[m, n] = A[m, k] B[n, k]^T
  int bn;               // tile columns: 256, 192, 128 or 64
  int n_tiles, tiles, kblocks;
  const float *bias;    // [n] or NULL
  int act;              // hidden GEMM: TR_ACT_*
  bool has_resid;       // score: x = x'' + residual
  float *part;          // score: [row blocks][n_tiles][kRowParts][4][kPartWords][32] partial sums
  int32_t *err;         // optional: set when a pipeline wait timed out
  // projector mode: A row j = x[first row of the image owning kept slot j + idx[j]]
  long long total_rows;
  int batch, n_uniform;
  const int32_t *cu_seqlens, *cu_k, *idx;
};

// Tensor maps of one launch: the operands, the output (hidden, projector: the
// activations; score: x''), and for the score mode x', the residual and x.
struct GemmMaps {
  CUtensorMap a, b, out, p, r, x;
};

__device__ __forceinline__ float bf16_val(uint32_t bits16) { return __uint_as_float(bits16 << 16); }

// 2^x and 1/x by the hardware approximations (PTX ex2.approx, rcp.approx:
// relative error about 2^-22 and 2^-23), a few fp32 ulp, far inside the bf16
// rounding of the activations below.
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Packed fp32 pairs (one instruction for two lanes of arithmetic, each
// rounded to nearest like its scalar form).
__device__ __forceinline__ float2 f2(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {  // a - b, one rounding
  return __ffma2_rn(b, f2(-1.f), a);
}
__device__ __forceinline__ float2 ex2_2(float2 x) { return make_float2(ex2_approx(x.x), ex2_approx(x.y)); }
__device__ __forceinline__ float2 rcp_2(float2 x) { return make_float2(rcp_approx(x.x), rcp_approx(x.y)); }

// erf(z) for z >= 0 by Abramowitz and Stegun, Handbook of Mathematical
// Functions (1964), formula 7.1.26: 1 - (a1 t + ... + a5 t^5) exp(-z^2) with
// t = 1 / (1 + p z), |error| <= 1.5e-7; with the approximate exponential and
// reciprocal GELU below stays within ~2e-7 |v| of x Phi(x), far inside the
// bf16 rounding of its result.  Two arguments at a time.
__device__ __forceinline__ float2 erf_as2(float2 z) {
  const float2 t = rcp_2(__ffma2_rn(z, f2(0.3275911f), f2(1.f)));
  float2 poly = __ffma2_rn(t, f2(1.061405429f), f2(-1.453152027f));
  poly = __ffma2_rn(t, poly, f2(1.421413741f));
  poly = __ffma2_rn(t, poly, f2(-0.284496736f));
  poly = __ffma2_rn(t, poly, f2(0.254829592f));
  poly = __fmul2_rn(t, poly);
  const float2 ez = ex2_2(__fmul2_rn(__fmul2_rn(z, z), f2(-1.4426950408889634f)));  // exp(-z^2)
  return sub2(f2(1.f), __fmul2_rn(poly, ez));
}

// The activation sigma of the hidden layer (and the projector) on a pair of
// pre-activations.
__device__ __forceinline__ float2 activate2(float2 v, int act) {
  if (act == TR_ACT_GELU) {  // v Phi(v) = v (1 + erf(v / sqrt 2)) / 2
    const float2 e = erf_as2(__fmul2_rn(make_float2(fabsf(v.x), fabsf(v.y)), f2(0.70710678118654752f)));
    return __fmul2_rn(__fmul2_rn(v, f2(0.5f)), __fadd2_rn(f2(1.f), make_float2(copysignf(e.x, v.x), copysignf(e.y, v.y))));
  }
  if (act == TR_ACT_QUICK_GELU) {  // v sigma(1.702 v) = v / (1 + 2^(-1.702 log2(e) v)), the exponent capped
    float2 z = __fmul2_rn(v, f2(-2.4554669595930156f));
    z.x = fminf(z.x, 126.f);
    z.y = fminf(z.y, 126.f);
    return __fmul2_rn(v, rcp_2(__fadd2_rn(ex2_2(z), f2(1.f))));
  }
  return v;
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t *>(&h);
}

__device__ __forceinline__ void flag_error(const GemmArgs &g, int code) {
  if (g.err) atomicOr(g.err, code);
}

// The score epilogue keeps its five double-float sums as fp32 pairs:
// component x takes the even columns, component y the odd ones, merged once
// per tile.
__device__ __forceinline__ float2 bf16x2_f2(uint32_t w) {  // the two bf16 of a word as fp32
  return make_float2(bf16_val(w & 0xffffu), bf16_val(w >> 16));
}
struct DF2 {
  float2 hi, lo;
};
struct Acc2 {
  DF2 l1, s2, a, b, p;
};
// acc += v with Knuth's TwoSum per component: s = hi + v, and the rounding
// error (hi - (s - (s - hi))) + (v - (s - hi)) joins lo.  With nb = hi - s
// (= -(s - hi) exactly, rounding being symmetric) the steps are the scalar
// df_add's, two lanes at a time.
__device__ __forceinline__ void df2_add(DF2 &acc, float2 v) {
  const float2 s = __fadd2_rn(acc.hi, v);
  const float2 nb = sub2(acc.hi, s);
  const float2 aa = __fadd2_rn(s, nb);
  acc.lo = __fadd2_rn(acc.lo, __fadd2_rn(sub2(acc.hi, aa), __fadd2_rn(v, nb)));
  acc.hi = s;
}
// acc += u v for products exact in fp32 (bf16 times bf16): the fused
// multiply-add rounds hi + u v once, as the sum of the exact product would.
__device__ __forceinline__ void df2_add_prod(DF2 &acc, float2 u, float2 v) {
  const float2 s = __ffma2_rn(u, v, acc.hi);
  const float2 nb = sub2(acc.hi, s);
  const float2 aa = __fadd2_rn(s, nb);
  acc.lo = __fadd2_rn(acc.lo, __fadd2_rn(sub2(acc.hi, aa), __ffma2_rn(u, v, nb)));
  acc.hi = s;
}
__device__ __forceinline__ void df2_fold(DF &out, const DF2 &in) {  // even + odd columns
  out.hi = in.hi.x;
  out.lo = in.lo.x;
  df_merge(out, in.hi.y, in.lo.y);
}

// The epilogues work on one 16-byte unit (8 columns) of a lane's row at a
// time, in loops that stay rolled: a tile's epilogue is short beside what it
// takes to fetch its code (unrolled over a block, the scoring arithmetic ran
// 17,000 clocks however few blocks a warp had).
// acc + bias of 8 columns, as pairs.
__device__ __forceinline__ void add_bias(const GemmArgs &g, int col0, const uint32_t (&v)[8], float2 (&a)[4]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) a[i] = make_float2(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
  if (g.bias) {  // the same 8 values in every lane: two broadcast loads
    const float4 *bp = reinterpret_cast<const float4 *>(g.bias + col0);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const float4 b = __ldg(bp + i);
      a[2 * i] = __fadd2_rn(a[2 * i], make_float2(b.x, b.y));
      a[2 * i + 1] = __fadd2_rn(a[2 * i + 1], make_float2(b.z, b.w));
    }
  }
}

// Hidden / projector epilogue for 8 columns of one row: bf16(act(acc + bias))
// to the staged unit at `addr`.
__device__ __forceinline__ void epi_act(const GemmArgs &g, int col0, const uint32_t (&v)[8], uint32_t addr) {
  float2 a[4];
  add_bias(g, col0, v, a);
  uint32_t w[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 h = activate2(a[i], g.act);
    w[i] = pack_bf16x2(h.x, h.y);
  }
  tc::st_shared_v4(addr, w[0], w[1], w[2], w[3]);
}

// Score epilogue for 8 columns of one row: x'' = bf16(acc + b2),
// x = bf16(resid + x''); the five sums take the rounded values (products and
// squares of bf16 values are exact in fp32; each term enters its double-float
// sum through TwoSum).  x' and the residual come from this warp's staged
// blocks (the unit at `addr` and kBlkBytes further) and x'' and x take their
// places.
__device__ __forceinline__ void epi_score(const GemmArgs &g, int col0, const uint32_t (&v)[8], uint32_t addr,
                                          Acc2 &acc) {
  uint32_t pw[4], rw[4], qo[4], xo[4];
  tc::ld_shared_v4(addr, pw[0], pw[1], pw[2], pw[3]);
  if (g.has_resid) tc::ld_shared_v4(addr + kBlkBytes, rw[0], rw[1], rw[2], rw[3]);
  float2 a[4];
  add_bias(g, col0, v, a);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    qo[i] = pack_bf16x2(a[i].x, a[i].y);  // x''
    const float2 q = bf16x2_f2(qo[i]);
    if (g.has_resid) {
      const float2 xs = __fadd2_rn(bf16x2_f2(rw[i]), q);
      xo[i] = pack_bf16x2(xs.x, xs.y);
    } else {
      xo[i] = qo[i];
    }
    const float2 xa = bf16x2_f2(xo[i] & 0x7fff7fffu);  // |x|
    const float2 p = bf16x2_f2(pw[i]);                 // x'
    df2_add(acc.l1, xa);
    df2_add_prod(acc.s2, xa, xa);
    df2_add_prod(acc.a, p, p);
    df2_add_prod(acc.b, q, q);
    df2_add_prod(acc.p, p, q);
  }
  tc::st_shared_v4(addr, qo[0], qo[1], qo[2], qo[3]);
  tc::st_shared_v4(addr + kBlkBytes, xo[0], xo[1], xo[2], xo[3]);
}

// One epilogue warp's place: its lane quarter, its blocks of a tile (first,
// first + parts, ... below end) and its staging.
struct EpiWarp {
  int first, end;      // blocks of a tile
  uint32_t buf, bar;   // staging, and the score mode's mbarrier of its loads
  uint32_t loads;      // score: blocks requested so far
  uint32_t used;       // score: blocks waited for so far
  int tile, blk;       // score: the next block to request
};

// Score mode: requests the x' and residual blocks of the warp's next block
// (every lane keeps the place; lane 0 issues).  The staged block must have
// been stored (bulk_wait_read).  row_of(rb): first of this warp's 32 rows in
// row tile rb.
template <int kParts, typename RowOf>
__device__ __forceinline__ void score_load_next(const GemmArgs &g, const GemmMaps &maps, EpiWarp &w, int step,
                                                RowOf row_of) {
  int nt = 0;
  while (w.tile < g.tiles) {
    nt = w.tile % g.n_tiles;
    if (w.blk < w.end && nt * g.bn + w.blk * kBlk < g.n) break;
    w.tile += step;
    w.blk = w.first;
  }
  if (w.tile >= g.tiles) return;
  if ((threadIdx.x & 31) == 0) {
    const int col = nt * g.bn + w.blk * kBlk, row = row_of(w.tile / g.n_tiles);
    tc::mbar_expect_tx(w.bar, g.has_resid ? 2 * kBlkBytes : kBlkBytes);
    tc::tma_load_2d(w.buf, &maps.p, col, row, w.bar);
    if (g.has_resid) tc::tma_load_2d(w.buf + kBlkBytes, &maps.r, col, row, w.bar);
  }
  ++w.loads;
  w.blk += kParts;
}

// The epilogue of one tile for this warp: for each of its blocks, the
// accumulator columns from TMEM, the mode's arithmetic into the staged block
// and the TMA store(s).  Rows and columns past the output are computed from
// zero operands and clipped by the store.  False when the score mode's loads
// timed out.  (Score: with x' and the residual loaded straight from global
// memory, 32 rows per warp load and one chunk ahead, a tile's epilogue took
// 24,000-33,000 clocks.)
template <int kMode, typename RowOf>
__device__ __forceinline__ bool epilogue_tile(const GemmArgs &g, const GemmMaps &maps, EpiWarp &w, uint32_t taddr,
                                              int nt, int row0, int step, RowOf row_of, Acc2 &acc2) {
  constexpr int kParts = epi_parts(kMode);
  constexpr int kUnits = 2;  // 8-column units in flight
  const int lane = threadIdx.x & 31;
  const uint32_t sw = (uint32_t)((lane >> 1) & 3);  // the 64-byte swizzle's row term
  for (int blk = w.first; blk < w.end; blk += kParts) {
    const int col = nt * g.bn + blk * kBlk;
    if (col >= g.n) break;
    uint32_t buf = w.buf;
    if (kMode == kModeScore) {
      const bool ok = tc::mbar_wait(w.bar, w.used & 1u);
      ++w.used;
      if (!__all_sync(0xffffffffu, ok)) return false;
    } else {  // the block's previous store must have been read
      buf += (w.used % stage_blks(kMode)) * kBlkBytes;
      ++w.used;
      if (lane == 0) tc::bulk_wait_read<stage_blks(kMode) - 1>();
      __syncwarp();
    }
    const uint32_t rowbuf = buf + (uint32_t)(lane * kBlk * 2);
#pragma unroll 1
    for (int u0 = 0; u0 < kBlk / 8; u0 += kUnits) {
      if (col + 8 * u0 >= g.n) break;  // n is a multiple of 16
      uint32_t v[kUnits][8];
#pragma unroll
      for (int i = 0; i < kUnits; ++i) tc::tmem_ld8(taddr + (uint32_t)(blk * kBlk + 8 * (u0 + i)), v[i]);
#pragma unroll
      for (int i = 0; i < kUnits; ++i) {
        const int u = u0 + i;
        const uint32_t addr = rowbuf + (((uint32_t)u ^ sw) << 4);
        if (kMode == kModeScore)
          epi_score(g, col + 8 * u, v[i], addr, acc2);
        else
          epi_act(g, col + 8 * u, v[i], addr);
      }
    }
    tc::fence_async_shared();
    __syncwarp();
    if (lane == 0) {
      if (row0 < g.m) {  // a block wholly past the last row is not stored
        tc::tma_store_2d(&maps.out, col, row0, buf);
        if (kMode == kModeScore) tc::tma_store_2d(&maps.x, col, row0, buf + kBlkBytes);
      }
      tc::bulk_commit();
      if (kMode == kModeScore) tc::bulk_wait_read<0>();  // the next loads overwrite the block
    }
    if (kMode == kModeScore) {
      __syncwarp();
      score_load_next<kParts>(g, maps, w, step, row_of);
    }
  }
  return true;
}

// This warp's 32 rows are done for its blocks of a tile: their partial sums
// go to the scratch; k_score_rows merges them once the GEMM has finished.
__device__ __forceinline__ long long part_slot(const GemmArgs &g, int rb, int nt, int part, int q) {
  return (((long long)(rb * g.n_tiles + nt) * kRowParts + part) * 4 + q) * (kPartWords * 32);
}
__device__ __forceinline__ void publish_rows(float *dst, const Acc2 &acc2) {
  Acc acc{{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
  df2_fold(acc.l1, acc2.l1);
  df2_fold(acc.s2, acc2.s2);
  df2_fold(acc.a, acc2.a);
  df2_fold(acc.b, acc2.b);
  df2_fold(acc.p, acc2.p);
  const float vals[kPartWords] = {acc.l1.hi, acc.l1.lo, acc.s2.hi, acc.s2.lo, acc.a.hi,
                                  acc.a.lo,  acc.b.hi,  acc.b.lo,  acc.p.hi,  acc.p.lo};
#pragma unroll
  for (int j = 0; j < kPartWords; ++j) __stcg(dst + 32 * j, vals[j]);
}

// The rows' records from the partial sums the score GEMM left: a CTA per 32
// rows, warp w of its kRowWarps merging parts w, w + kRowWarps, ... in turn
// and a warp for each of the five sums then the warps' (one warp for all five:
// passes of 576 rows 32.06 us against 31.78), so that the record does not
// depend on which CTA made which part; four parts' loads are in flight at a
// time (one warp walking all parts with its loads one part ahead of their use
// took 19 us on 36,864 rows).  A kernel of
// its own, begun while the GEMM drains: arrival counters inside the GEMM cost
// each tile a fence over its stores, an atomic and, for the last warp, this
// same merge in series (about 5,000 clocks a tile, and a memset before every
// launch).
constexpr int kRowWarps = 8;
__device__ __forceinline__ void merge_part(Acc &tot, const float (&w)[kPartWords]) {
  df_merge(tot.l1, w[0], w[1]);
  df_merge(tot.s2, w[2], w[3]);
  df_merge(tot.a, w[4], w[5]);
  df_merge(tot.b, w[6], w[7]);
  df_merge(tot.p, w[8], w[9]);
}
__global__ void __launch_bounds__(kRowWarps * 32) k_score_rows(const GemmArgs g, float4 *__restrict__ stats,
                                                               float *__restrict__ h2, float *__restrict__ s_out) {
  __shared__ float sh[kRowWarps][kPartWords][32];
  pdl_trigger();
  pdl_wait();  // the partial sums come from the GEMM before this kernel
  const int rb = blockIdx.x >> 2, q = blockIdx.x & 3, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int total = kRowParts * g.n_tiles;
  const float *src = g.part + part_slot(g, rb, 0, 0, q) + lane;
  constexpr int kStep = 4 * kPartWords * 32;  // floats from one part to the next (the four quarters between)
  constexpr int kU = 4;
  Acc tot{{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
  for (int t0 = warp; t0 < total; t0 += kU * kRowWarps) {
    float w[kU][kPartWords];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int t = t0 + u * kRowWarps;
      // past the last part: its values again, dropped below (no branch holds up the loads)
      const float *p = src + (long long)(t < total ? t : t0) * kStep;
#pragma unroll
      for (int j = 0; j < kPartWords; ++j) w[u][j] = __ldcg(p + 32 * j);
    }
#pragma unroll
    for (int u = 0; u < kU; ++u)
      if (t0 + u * kRowWarps < total) merge_part(tot, w[u]);  // uniform
  }
  const float vals[kPartWords] = {tot.l1.hi, tot.l1.lo, tot.s2.hi, tot.s2.lo, tot.a.hi,
                                  tot.a.lo,  tot.b.hi,  tot.b.lo,  tot.p.hi,  tot.p.lo};
#pragma unroll
  for (int j = 0; j < kPartWords; ++j) sh[warp][j][lane] = vals[j];
  __syncthreads();
  if (warp < kPartWords / 2) {  // sum number `warp` of the five, over the warps
    DF v{sh[0][2 * warp][lane], sh[0][2 * warp + 1][lane]};
#pragma unroll
    for (int w = 1; w < kRowWarps; ++w) df_merge(v, sh[w][2 * warp][lane], sh[w][2 * warp + 1][lane]);
    if (warp) {
      sh[0][2 * warp][lane] = v.hi;  // read by this warp alone until here
      sh[0][2 * warp + 1][lane] = v.lo;
    } else {
      tot.l1 = v;
    }
  }
  __syncthreads();
  if (warp) return;
  tot.s2 = DF{sh[0][2][lane], sh[0][3][lane]};
  tot.a = DF{sh[0][4][lane], sh[0][5][lane]};
  tot.b = DF{sh[0][6][lane], sh[0][7][lane]};
  tot.p = DF{sh[0][8][lane], sh[0][9][lane]};
  const long long row = (long long)rb * kBM + 32 * q + lane;
  if (row < g.m) write_record(tot, row, stats, h2, s_out);
}

// Row of x that kept slot j names (projector mode), or -1: the image b with
// cu_k[b] <= j < cu_k[b + 1], its local index idx[j] checked against the
// image's tokens (an index outside them gives a zero row, never another
// image's token or an address outside x).
__device__ __forceinline__ long long kept_source_row(const GemmArgs &g, long long j) {
  if (j >= g.m) return -1;
  int lo = 0, hi = g.batch;  // cu_k[lo] <= j < cu_k[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (__ldg(g.cu_k + mid) <= j) lo = mid; else hi = mid;
  }
  const long long first = g.cu_seqlens ? (long long)__ldg(g.cu_seqlens + lo) : (long long)lo * g.n_uniform;
  const long long n_b = g.cu_seqlens ? (long long)__ldg(g.cu_seqlens + lo + 1) - first : (long long)g.n_uniform;
  const int local = __ldg(g.idx + j);
  if (local < 0 || local >= n_b || first < 0 || first + local >= g.total_rows) return -1;
  return first + local;
}

// ---------------------------------------------------------------- the SM-pair kernel
// tcgen05's 2-SM MMA: a cluster of two CTAs shares each output tile of 256
// rows x bn columns (tile t: row block t / n_tiles).  CTA rank r loads A rows
// 128 r .. 128 r + 127 of the tile and its half of the tile's B rows (output
// columns) into its own shared memory -- 32 KiB per k-block stage, six stages
// -- and both CTAs' loads complete on the even CTA's stage barrier.  The even
// CTA alone issues the pair's MMAs (M 256, N bn, K 16), which read both
// CTAs' stages and write each CTA's 128 accumulator rows into its own TMEM;
// its commits reach the same barriers in both CTAs (multicast).  Each CTA's
// epilogue drains its own rows and releases the accumulator on the even
// CTA's barrier.  Per SM a k-block of 256 columns brings 32 KiB of operands
// for a 128 x 256 x 64 product, against 48 KiB on one SM.  A batch of at most 128
// rows runs here too, the odd CTA's rows read as zeros: what such a batch
// waits for is W, and a pair brings each half of it into its own SM (128 rows,
// D 1024, hidden 4096, both GEMMs: 57.4 us with a one-SM kernel, 55.3 here).
constexpr int kStagesP = 6;
constexpr int kHalfTile = 128 * kBK * 2;          // 128 rows of a k-block (A or B)
constexpr int kStagePBytes = 2 * kHalfTile;       // this CTA's A rows + B rows
__host__ __device__ constexpr int gemm_smem(int mode) {  // + alignment, barriers
  return kStagesP * kStagePBytes + epi_warps(mode) * stage_bytes(mode) + 1024 + 512;
}

template <int kMode>
__global__ void __launch_bounds__(gemm_threads(kMode), 1)
    k_mlp_gemm(const __grid_constant__ GemmMaps maps, const GemmArgs g) {
  pdl_trigger();
  extern __shared__ unsigned char smem_raw[];
  unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                          ~static_cast<uintptr_t>(1023));
  const uint32_t out_stage = tc::smem_u32(smem + (size_t)kStagesP * kStagePBytes);  // epilogue staging
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem + (size_t)kStagesP * kStagePBytes + epi_warps(kMode) * stage_bytes(kMode));
  constexpr int kBlkBars = kMode == kModeScore ? epi_warps(kMode) : 0;  // the score epilogue's staged blocks
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * kStagesP + 5 + kBlkBars);
  const uint32_t sbase = tc::smem_u32(smem);
  const uint32_t b0 = tc::smem_u32(bars);
  auto full = [&](int s) { return b0 + 8u * s; };
  auto empty = [&](int s) { return b0 + 8u * (kStagesP + s); };
  auto tfull = [&](int a) { return b0 + 8u * (2 * kStagesP + a); };
  auto tempty = [&](int a) { return b0 + 8u * (2 * kStagesP + 2 + a); };
  const uint32_t done = b0 + 8u * (2 * kStagesP + 4);
  auto blk_bar = [&](int w) { return b0 + 8u * (2 * kStagesP + 5 + w); };  // of epilogue warp w
  auto sa = [&](int s) { return sbase + (uint32_t)(s * kStagePBytes); };
  auto sb = [&](int s) { return sbase + (uint32_t)(s * kStagePBytes + kHalfTile); };

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = tc::cluster_rank();
  const bool leader = rank == 0;
  const int pair = blockIdx.x / 2, pairs = gridDim.x / 2;
  // operand bytes landing on the even CTA's stage barrier per k-block (both CTAs)
  const uint32_t b_bytes = (uint32_t)g.bn * kBK * 2u;  // of B per k-block, both CTAs
  const uint32_t tx = b_bytes + (kMode == kModeProject ? 0u : 2u * kHalfTile);
  const uint32_t idesc = tc::idesc_bf16(2 * kBM, g.bn);
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStagesP; ++s) {
      tc::mbar_init(full(s), kMode == kModeProject ? 1 + kLoadWarps : 1);  // + the even CTA's loader warps
      tc::mbar_init(empty(s), 1);
    }
    for (int a = 0; a < 2; ++a) {
      tc::mbar_init(tfull(a), 1);
      tc::mbar_init(tempty(a), 2 * epi_warps(kMode));  // one arrival per epilogue warp of either CTA
    }
    tc::mbar_init(done, 1);
    for (int i = 0; i < kBlkBars; ++i) tc::mbar_init(blk_bar(i), 1);
    tc::mbar_fence_init();
    tc::tma_prefetch_map(&maps.a);
    tc::tma_prefetch_map(&maps.b);
  }
  if (warp == 1) {
    tc::tmem_alloc_pair(tc::smem_u32(tmem_slot), kTmemCols);
    tc::tmem_relinquish_pair();
  }
  tc::fence_before_sync();
  tc::cluster_sync();  // barriers initialised and TMEM allocated in both CTAs
  tc::fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  pdl_wait();  // operands come from, and outputs may still be read by, the kernels before this one
  constexpr uint16_t both = 0x3;  // the CTAs that a commit reaches
  auto full_even = [&](int s) { return tc::map_shared(full(s), 0u); };
  auto tempty_even = [&](int a) { return tc::map_shared(tempty(a), 0u); };
  const int tiles = g.tiles;

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer (both CTAs)
    if (tc::elect_one()) {
      int stage = 0;
      uint32_t phase = 0, filled = 0, last_parity = 0;
      bool ok = true;
      for (int tile = pair; tile < tiles && ok; tile += pairs) {
        const int rb = tile / g.n_tiles, nt = tile - rb * g.n_tiles;
        for (int kb = 0; kb < g.kblocks; ++kb) {
          if (!tc::mbar_wait(empty(stage), phase ^ 1u)) {
            ok = false;
            break;
          }
          const uint32_t bar = full_even(stage);
          if (leader) tc::mbar_expect_tx(full(stage), tx);
          if (kMode != kModeProject)
            tc::tma_load_2d_pair(sa(stage), &maps.a, kb * kBK, rb * 2 * kBM + (int)rank * kBM, bar);
          tc::tma_load_2d_pair(sb(stage), &maps.b, kb * kBK, nt * g.bn + (int)rank * (g.bn / 2), bar);
          filled |= 1u << stage;
          last_parity = (last_parity & ~(1u << stage)) | (phase << stage);
          if (++stage == kStagesP) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
      if (!ok) flag_error(g, 1);
      // every load of either CTA lands on the even CTA's barriers: it waits for
      // them before the final cluster barrier, so no CTA exits with loads in flight
      if (leader)
        for (int s = 0; s < kStagesP; ++s)
          if (filled & (1u << s)) tc::mbar_wait(full(s), (last_parity >> s) & 1u);
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer (even CTA)
    if (leader && tc::elect_one()) {
      int stage = 0, acc = 0;
      uint32_t phase = 0, acc_phase = 0;
      bool ok = true;
      for (int tile = pair; tile < tiles && ok; tile += pairs) {
        if (!tc::mbar_wait(tempty(acc), acc_phase ^ 1u)) {
          ok = false;
          break;
        }
        tc::fence_after_sync();
        const uint32_t d = tmem + (uint32_t)(acc * kBN);
        for (int kb = 0; kb < g.kblocks; ++kb) {
          if (!tc::mbar_wait(full(stage), phase)) {
            ok = false;
            break;
          }
          tc::fence_after_sync();
          const uint64_t da = tc::sw128_desc(sa(stage)), db = tc::sw128_desc(sb(stage));
#pragma unroll
          for (int k = 0; k < kBK / 16; ++k)
            tc::mma_bf16_pair(d, da + 2u * k, db + 2u * k, idesc, (kb | k) != 0);
          tc::mma_commit_pair(empty(stage), both);  // both CTAs' stage is free once these MMAs read it
          if (++stage == kStagesP) {
            stage = 0;
            phase ^= 1u;
          }
        }
        if (!ok) break;
        tc::mma_commit_pair(tfull(acc), both);
        acc ^= 1;
        if (acc == 0) acc_phase ^= 1u;
      }
      if (!ok) flag_error(g, 2);
      tc::mma_commit_pair(done, both);
    }
    __syncwarp();
    tc::mbar_wait_warp(done, 0);  // every pair MMA has completed (both CTAs' TMEM)
  } else if (kMode == kModeProject && warp >= 2 + epi_warps(kMode)) {
    // ---------------------------------------------------------------- A rows (projector mode)
    // loader warp w brings rows 32 w .. 32 w + 31 of this CTA's half of the
    // pair's rows of each A k-block with eight tile::gather4 loads; a group
    // with a row outside x (past the kept slots) or a k-block past x's
    // columns takes four one-row loads instead, an outside row at coordinate
    // -1, which reads zeros.  The loads land on the even CTA's barrier, whose
    // loader warps expect both CTAs' bytes (the odd CTA's loader warps do not
    // arrive).  Each lane looks up one row; one thread issues.
    const int lw = warp - 2 - epi_warps(kMode);
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    for (int tile = pair; tile < tiles && ok; tile += pairs) {
      const int rb = tile / g.n_tiles;
      const long long src = kept_source_row(g, (long long)rb * 2 * kBM + (long long)rank * kBM + 32 * lw + lane);
      const int mine = src >= 0 ? (int)src : -1;
      const uint32_t inside = __ballot_sync(0xffffffffu, mine >= 0);
      int srow[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) srow[i] = __shfl_sync(0xffffffffu, mine, i);
      if (tc::elect_one()) {
        for (int kb = 0; kb < g.kblocks; ++kb) {
          if (!tc::mbar_wait(empty(stage), phase ^ 1u)) {
            ok = false;
            break;
          }
          if (leader) tc::mbar_expect_tx(full(stage), 2 * kHalfTile / kLoadWarps);
          const uint32_t dst = sa(stage) + (uint32_t)(32 * lw * kBK * 2);
          const uint32_t bar = full_even(stage);
          const bool cols = (kb + 1) * kBK <= g.k;  // the k-block lies inside x's columns
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            if (cols && ((inside >> (4 * j)) & 0xfu) == 0xfu) {
              tc::tma_gather4_pair(dst + (uint32_t)(4 * j * kBK * 2), &maps.a, kb * kBK, srow[4 * j], srow[4 * j + 1],
                                   srow[4 * j + 2], srow[4 * j + 3], bar);
            } else {
#pragma unroll
              for (int i = 4 * j; i < 4 * j + 4; ++i)
                tc::tma_load_2d_pair(dst + (uint32_t)(i * kBK * 2), &maps.a, kb * kBK, srow[i], bar);
            }
          }
          if (++stage == kStagesP) {
            stage = 0;
            phase ^= 1u;
          }
        }
        if (!ok) flag_error(g, 8);
      }
      ok = __all_sync(0xffffffffu, ok) != 0;  // (stage and phase live in the elected thread, the same one every time)
    }
  } else {
    // ---------------------------------------------------------------- epilogue (both CTAs)
    const int q = warp & 3;            // TMEM lane quadrant this warp may read
    const int part = (warp - 2) >> 2;  // which of the quadrant's warps
    // first of this warp's 32 rows in row tile rb
    auto row_of = [&](int rb) { return (2 * rb + (int)rank) * kBM + 32 * q; };
    EpiWarp w{part, g.bn / kBlk, out_stage + (uint32_t)((warp - 2) * stage_bytes(kMode)),
              blk_bar(warp - 2), 0u, 0u, pair, part};
    if (kMode == kModeScore) score_load_next<epi_parts(kMode)>(g, maps, w, pairs, row_of);
    int acc = 0;
    uint32_t acc_phase = 0;
    for (int tile = pair; tile < tiles; tile += pairs) {
      const int rb = tile / g.n_tiles, nt = tile - rb * g.n_tiles;
      if (g.bias)  // the first blocks' bias on its way to L1 while the main loop runs
        for (int blk = w.first; blk < w.end; blk += epi_parts(kMode))
          if (nt * g.bn + blk * kBlk + lane < g.n) tc::touch(g.bias + nt * g.bn + blk * kBlk + lane);
      bool ok = tc::mbar_wait_warp(tfull(acc), acc_phase);
      if (!ok && lane == 0) flag_error(g, 4);
      tc::fence_after_sync();
      const uint32_t taddr = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(acc * kBN);
      Acc2 sums{};
      if (ok && !epilogue_tile<kMode>(g, maps, w, taddr, nt, row_of(rb), pairs, row_of, sums)) {
        ok = false;
        if (lane == 0) flag_error(g, 16);
      }
      if (!ok) break;
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive_cluster(tempty_even(acc));  // this warp is done with the accumulator
      const int rb128 = 2 * rb + (int)rank;
      if (kMode == kModeScore && rb128 * kBM < g.m)
        publish_rows(g.part + part_slot(g, rb128, nt, part, q) + lane, sums);
      acc ^= 1;
      if (acc == 0) acc_phase ^= 1u;
    }
    if (lane == 0) {
      if (kMode == kModeScore && w.used != w.loads)  // a block requested and not used (after a timeout) lands first
        tc::mbar_wait(w.bar, w.used & 1u);
      tc::bulk_wait();  // this warp's output stores have completed
    }
    __syncwarp();
  }

  tc::fence_before_sync();
  tc::cluster_sync();  // neither CTA leaves while the other may still signal its barriers
  if (warp == 1) {
    tc::fence_after_sync();
    tc::tmem_dealloc_pair(tmem, kTmemCols);
  }
}

// ---------------------------------------------------------------- host side
using EncodeTiled = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                 const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiled encode_fn() {
  static std::once_flag once;
  static EncodeTiled fn = nullptr;
  std::call_once(once, [] {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiled>(p);
  });
  return fn;
}

// A bf16 [rows, cols] row-major tensor in boxes of box_rows x box_cols
// (box_cols x 2 bytes = the swizzle span: 64 columns with the 128-byte
// swizzle for operands, 32 with the 64-byte swizzle for the output staging);
// out-of-range rows and columns read as zeros.
bool make_map(CUtensorMap *map, const void *base, long long rows, long long cols, int box_rows, int box_cols = kBK,
              CUtensorMapSwizzle swizzle = CU_TENSOR_MAP_SWIZZLE_128B) {
  EncodeTiled fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
  const cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Per device (index & 63): bit `mode` set once the mode's shared-memory limit
// is raised and its co-resident pairs are counted.
std::atomic<int> g_gemm_set[64];
std::atomic<int> g_gemm_pairs[64][3];

template <int kMode>
cudaError_t launch_gemm(const GemmMaps &maps, const GemmArgs &g, cudaStream_t st) {
  int dev = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err != cudaSuccess) return err;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(gemm_threads(kMode));
  cfg.dynamicSmemBytes = gemm_smem(kMode);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (!(g_gemm_set[dev & 63].load() & (1 << kMode))) {
    err = cudaFuncSetAttribute(k_mlp_gemm<kMode>, cudaFuncAttributeMaxDynamicSharedMemorySize, gemm_smem(kMode));
    if (err != cudaSuccess) return err;
    int pairs = 0;
    cfg.gridDim = dim3(2 * 64);
    err = cudaOccupancyMaxActiveClusters(&pairs, k_mlp_gemm<kMode>, &cfg);
    if (err != cudaSuccess) return err;
    if (pairs <= 0) return cudaErrorInvalidConfiguration;
    g_gemm_pairs[dev & 63][kMode].store(pairs);
    g_gemm_set[dev & 63].fetch_or(1 << kMode);
  }
  cfg.gridDim = dim3(2 * std::min(g.tiles, g_gemm_pairs[dev & 63][kMode].load()));
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, k_mlp_gemm<kMode>, maps, g);
}

inline int row_tiles(int m) { return (int)(((long long)m + 2 * kBM - 1) / (2 * kBM)); }

// How a GEMM is laid out on the 76 SM pairs: its tile columns.
struct GemmShape {
  int bn, n_tiles, kblocks;
};
// The cheapest width by a model in clocks; a function of the sizes alone (it
// also sizes tr_mlp_score's scratch), whatever the device has free: the waves
// of tiles times the longer of a tile's main loop and its epilogue, and among
// equals the narrowest, whose last epilogue ends sooner.
//   A k-block takes the larger of its MMAs (2 clocks a column) and the operands
//   into each SM at 63 bytes a clock, A's 16 KiB and B's 64 bytes a column:
//   520 clocks for 256 columns, 455, 390 and 325 for 192, 128 and 64; the
//   projector's row gather 1065 whatever the columns.  An epilogue takes a
//   fixed part and one for each round of blocks over its warps: score 18,500
//   clocks for 256 columns and 9,500 for 64, projector 7,500 and 3,750.  The
//   hidden GEMM's, shared by twice the warps, shrinks with the width no more
//   than its main loop does (5,400 to 8,700 clocks by activation for 256
//   columns, 3,200 to 4,000 for 64), so the main loop ranks the widths at any K.
// Against the best of the four widths, each measured on 1419 sizes (K 64 to
// 4096, 256 to 4096 columns, 192 to 36,864 rows, three modes): within 0.1 % on
// average and 5.2 % at most.  (An epilogue in proportion to the columns gave
// few k-blocks narrow tiles whatever the rows: 36,864 rows, K 64, 4096 columns
// 255 us in 64-column tiles, 138 in 256.)
// With 256 columns throughout and with the width chosen: 192 rows, 1024 ->
// 4096, 12.3 and 8.4 us a pass (16 tiles, 64 of 64 columns); both GEMMs of 2885
// rows, 1152 -> 4304 -> 1152, 63.4 and 58.9 (60 score tiles, 72 of 192
// columns); both of 576 rows, 1024 -> 4096 -> 1024, 53.7 and 33.5 (12 score
// tiles, 48 of 64), of 48 rows 51 and 27.7.
// K is not shared among pairs where tiles are few: clusters that split it and
// exchanged partial accumulators took 32.3 us for the 576 rows and 24.5 for the
// 48, but then the order of an output element's sum, and so its last bits,
// followed the number of rows; in one order a row gives the same H, x'' and z
// alone, in any batch and with any scratch.
inline GemmShape gemm_shape(int m, int n, int k, int mode) {
  constexpr long long kPairs = 76;
  const int kb = (k + kBK - 1) / kBK;
  const long long rows = row_tiles(m);
  auto cost = [&](int bn) {
    const long long waves = (rows * ((n + bn - 1) / bn) + kPairs - 1) / kPairs;
    const int main = kb * (mode == kModeProject ? 1065 : std::max(2 * bn + 8, (16384 + 64 * bn) / 63));
    const int epi = mode == kModeScore ? 6500 + 3000 * bn / 64 : (mode == kModeProject ? 2500 + 1250 * bn / 64 : 0);
    return waves * std::max(main, epi);
  };
  int best = kBN;
  for (const int bn : kWidths)
    if (cost(bn) <= cost(best)) best = bn;
  return GemmShape{best, (n + best - 1) / best, kb};
}

inline void set_shape(GemmArgs &g, const GemmShape &sh) {
  g.bn = sh.bn;
  g.n_tiles = sh.n_tiles;
  g.tiles = row_tiles(g.m) * sh.n_tiles;
  g.kblocks = sh.kblocks;
}

bool misaligned16(const void *p) { return p && (reinterpret_cast<uintptr_t>(p) & 15u) != 0; }

tr_status check_mlp(const tr_mlp *m) {
  if (!m || !m->x_pre || !m->w1 || !m->w2) return TR_ERR_ARG;
  if (m->t < 0 || m->d <= 0 || m->d_hidden <= 0) return TR_ERR_ARG;
  if (m->act != TR_ACT_GELU && m->act != TR_ACT_QUICK_GELU && m->act != TR_ACT_NONE) return TR_ERR_ARG;
  if (m->d % 16 != 0 || m->d_hidden % 16 != 0) return TR_ERR_ALIGN;
  if (m->d > TR_MAX_D || m->d_hidden > TR_MLP_MAX_HIDDEN) return TR_ERR_UNSUPPORTED;
  const long long rblocks = ((long long)m->t + kBM - 1) / kBM;  // tile counts stay in int
  if (rblocks * ((m->d_hidden + kBN - 1) / kBN) > INT_MAX) return TR_ERR_UNSUPPORTED;
  if (misaligned16(m->x_pre) || misaligned16(m->resid) || misaligned16(m->w1) || misaligned16(m->w2) ||
      misaligned16(m->b1) || misaligned16(m->b2))
    return TR_ERR_ALIGN;
  return TR_OK;
}

// Bytes of the score mode's partial sums in one layout, and the layout that
// tr_mlp_score takes with `bytes` of them: the one gemm_shape chooses, or with
// fewer (a workspace sized for another batch: the narrow tiles of few rows may
// want more than the 256-column tiles of many) 256-column tiles.
size_t part_bytes(const tr_mlp *m, const GemmShape &sh) {
  const long long rblocks = ((long long)m->t + kBM - 1) / kBM;
  return align_up((size_t)rblocks * sh.n_tiles * kRowParts * 4 * kPartWords * 32 * sizeof(float), 256);
}
GemmShape score_shape(const tr_mlp *m, size_t bytes) {
  const GemmShape sh = gemm_shape(m->t, m->d, m->d_hidden, kModeScore);
  return part_bytes(m, sh) <= bytes ? sh : GemmShape{kBN, (m->d + kBN - 1) / kBN, sh.kblocks};
}

// out = act(a W^T + bias) for dense bf16 rows a [rows, k] and W [n, k]: the
// hidden-mode GEMM (bias + activation epilogue, TMA stores), arguments
// checked by the caller.
tr_status dense_act_gemm(const void *a, int rows, int k, const void *w, const float *bias, int n, int act, void *out,
                         int32_t *d_error, cudaStream_t st) {
  if (rows == 0) return TR_OK;
  GemmArgs g{};
  g.m = rows;
  g.n = n;
  g.k = k;
  const GemmShape sh = gemm_shape(g.m, g.n, g.k, kModeHidden);
  set_shape(g, sh);
  g.bias = bias;
  g.act = act;
  g.err = d_error;
  GemmMaps maps{};
  if (!make_map(&maps.a, a, rows, k, kBM) || !make_map(&maps.b, w, n, k, sh.bn / 2) ||
      !make_map(&maps.out, out, rows, n, 32, kBlk, CU_TENSOR_MAP_SWIZZLE_64B))
    return TR_ERR_CUDA;
  return launch_gemm<kModeHidden>(maps, g, st) == cudaSuccess ? TR_OK : TR_ERR_CUDA;
}

}  // namespace
}  // namespace tr

using namespace tr;

extern "C" {

tr_status tr_mlp_hidden(const tr_mlp *m, void *h, int32_t *d_error, void *stream) {
  tr_status rc = check_mlp(m);
  if (rc != TR_OK) return rc;
  if (!h) return TR_ERR_ARG;
  if (misaligned16(h)) return TR_ERR_ALIGN;
  return dense_act_gemm(m->x_pre, m->t, m->d, m->w1, m->b1, m->d_hidden, m->act, h, d_error,
                        static_cast<cudaStream_t>(stream));
}

tr_status tr_project(const void *y, int32_t rows, int32_t d, const void *w, const float *bias, int32_t d_out,
                     int32_t act, void *z, int32_t *d_error, void *stream) {
  if (!y || !w || !z || rows < 0 || d <= 0 || d_out <= 0) return TR_ERR_ARG;
  if (act != TR_ACT_GELU && act != TR_ACT_QUICK_GELU && act != TR_ACT_NONE) return TR_ERR_ARG;
  if (d % 16 != 0 || d_out % 16 != 0) return TR_ERR_ALIGN;
  if (d > TR_MAX_D || d_out > TR_MLP_MAX_HIDDEN) return TR_ERR_UNSUPPORTED;
  if (((long long)rows + kBM - 1) / kBM * ((d_out + kBN - 1) / kBN) > INT_MAX) return TR_ERR_UNSUPPORTED;
  if (misaligned16(y) || misaligned16(w) || misaligned16(bias) || misaligned16(z)) return TR_ERR_ALIGN;
  return dense_act_gemm(y, rows, d, w, bias, d_out, act, z, d_error, static_cast<cudaStream_t>(stream));
}

int32_t tr_gemm_columns(int32_t rows, int32_t n, int32_t k, int32_t kind) {
  if (rows <= 0 || n <= 0 || k <= 0 || kind < kModeHidden || kind > kModeProject) return 0;
  return gemm_shape(rows, n, k, kind).bn;
}

size_t tr_mlp_workspace_bytes(const tr_mlp *m) {
  if (check_mlp(m) != TR_OK) return 0;
  return part_bytes(m, score_shape(m, SIZE_MAX));
}

tr_status tr_mlp_score(const tr_mlp *m, const void *h, void *x_post, void *x, float *stats, float *h2, float *s,
                       void *ws, size_t ws_bytes, int32_t *d_error, void *stream) {
  tr_status rc = check_mlp(m);
  if (rc != TR_OK) return rc;
  if (!h || !x_post || !x || !stats) return TR_ERR_ARG;
  if (misaligned16(h) || misaligned16(x_post) || misaligned16(x) || misaligned16(stats) ||
      (reinterpret_cast<uintptr_t>(h2) & 3u) || (reinterpret_cast<uintptr_t>(s) & 3u))
    return TR_ERR_ALIGN;
  const GemmShape sh = score_shape(m, ws_bytes);
  if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255u) || ws_bytes < part_bytes(m, sh)) return TR_ERR_WORKSPACE;
  if (m->t == 0) return TR_OK;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  GemmArgs g{};
  g.m = m->t;
  g.n = m->d;
  g.k = m->d_hidden;
  set_shape(g, sh);
  g.bias = m->b2;
  g.has_resid = m->resid != nullptr;
  g.part = static_cast<float *>(ws);
  g.err = d_error;
  GemmMaps maps{};
  auto block_map = [&](CUtensorMap *map, const void *p) {  // the epilogue's 32 x 32 blocks
    return make_map(map, p, m->t, m->d, 32, kBlk, CU_TENSOR_MAP_SWIZZLE_64B);
  };
  if (!make_map(&maps.a, h, m->t, m->d_hidden, kBM) || !make_map(&maps.b, m->w2, m->d, m->d_hidden, sh.bn / 2) ||
      !block_map(&maps.p, m->x_pre) || (m->resid && !block_map(&maps.r, m->resid)) || !block_map(&maps.out, x_post) ||
      !block_map(&maps.x, x))
    return TR_ERR_CUDA;
  if (launch_gemm<kModeScore>(maps, g, st) != cudaSuccess) return TR_ERR_CUDA;
  const cudaError_t err = launch_kernel(k_score_rows, dim3((g.m + kBM - 1) / kBM * 4), dim3(kRowWarps * 32), 0, st, true,
                                        g, reinterpret_cast<float4 *>(stats), h2, s);
  return err == cudaSuccess ? TR_OK : TR_ERR_CUDA;
}

tr_status tr_project_kept(const tr_tokens *in, const int32_t *d_cu_k, const int32_t *idx, int32_t total_k,
                          const void *w, const float *bias, int32_t d_out, int32_t act, void *z, int32_t *d_error,
                          void *stream) {
  if (!in || !in->x || !w || !z) return TR_ERR_ARG;
  if (in->dtype != TR_BF16) return TR_ERR_DTYPE;
  if (in->d <= 0 || d_out <= 0 || in->batch < 0) return TR_ERR_ARG;
  if (act != TR_ACT_GELU && act != TR_ACT_QUICK_GELU && act != TR_ACT_NONE) return TR_ERR_ARG;
  if (in->d % 16 != 0 || d_out % 16 != 0) return TR_ERR_ALIGN;
  if (in->d > TR_MAX_D || d_out > TR_MLP_MAX_HIDDEN) return TR_ERR_UNSUPPORTED;
  if (misaligned16(in->x) || misaligned16(w) || misaligned16(bias) || misaligned16(z)) return TR_ERR_ALIGN;
  long long total_rows;
  if (in->cu_seqlens) {
    if (in->total < 0) return TR_ERR_ARG;
    total_rows = in->total;
  } else {
    if (in->n < 0) return TR_ERR_ARG;
    total_rows = (long long)in->batch * in->n;
  }
  if (total_k < 0 || total_k > total_rows) return TR_ERR_BUDGET;
  if (total_rows > INT_MAX) return TR_ERR_UNSUPPORTED;  // TMA row coordinates are 32-bit
  if (total_k == 0) return TR_OK;
  if (in->batch == 0 || !d_cu_k || !idx) return TR_ERR_ARG;
  const long long rblocks = ((long long)total_k + kBM - 1) / kBM;
  if (rblocks * ((d_out + kBN - 1) / kBN) > INT_MAX) return TR_ERR_UNSUPPORTED;
  GemmArgs g{};
  g.m = total_k;
  g.n = d_out;
  g.k = in->d;
  const GemmShape sh = gemm_shape(g.m, g.n, g.k, kModeProject);
  set_shape(g, sh);
  g.bias = bias;
  g.act = act;
  g.err = d_error;
  g.total_rows = total_rows;
  g.batch = in->batch;
  g.n_uniform = in->cu_seqlens ? 0 : in->n;
  g.cu_seqlens = in->cu_seqlens;
  g.cu_k = d_cu_k;
  g.idx = idx;
  // A: x, one row per box (the loaders gather rows by kept index)
  GemmMaps maps{};
  if (!make_map(&maps.a, in->x, total_rows, in->d, 1) || !make_map(&maps.b, w, d_out, in->d, sh.bn / 2) ||
      !make_map(&maps.out, z, total_k, d_out, 32, kBlk, CU_TENSOR_MAP_SWIZZLE_64B))
    return TR_ERR_CUDA;
  return launch_gemm<kModeProject>(maps, g, static_cast<cudaStream_t>(stream)) == cudaSuccess ? TR_OK : TR_ERR_CUDA;
}

}  // extern "C"
