// argus_aggregate.cu — argus_aggregate: intervals (+ ambiguity records) -> per-(scope, region) tables.
//
//   k_agg_streams_digest : argus_synthesize's pass: one CTA per stream reads the 8-byte digests the pairing
//                   kernel wrote beside the interval records (not the records) and gathers the stream's row
//                   in 124-byte shared-memory cells, with per-lane copies of the most frequent regions' cells;
//   k_agg_streams_records : the same over the 48-byte records, without the overlap selection;
//   k_agg_streams_compact : the same over the records that a scope selects: that stream's row in
//                   a compact shared-memory form (112 B per region: sums, min, max, a 16-bin window, so
//                   several CTAs fit an SM), for up to kAggCompactRegions regions;
//   k_agg_streams : the same on the global row itself, for more regions than that. Integer atomics only: the
//                   result does not depend on thread order.
//   k_agg_rollup  : CTA-scope and warp-role cells = reductions over the warps of each CTA and over the CTAs; SM-scope and
//                   kernel-scope cells by atomic add/min/max of CTA cells.
//   k_agg_iter_windows, k_agg_iter : per-iteration cells (key = ctx - ctx_lo) of the intervals of a scope.
// A scope (iteration window, warp mask, SM mask, region mask) filters what the kernels over intervals
// take in; without one everything is selected.
#include "argus_bulk.cuh"
#include "argus_internal.cuh"

#include <mutex>
#include <type_traits>

namespace {

constexpr int kAggThreads = 256;
constexpr u32 kCell = 72;  // u64 words per argus_agg_t
constexpr u32 kAggCompactRegions = 400;  // 112 B each: 44.8 KB of shared memory at most (k_agg_iter_windows: 136 KB)
constexpr u32 kIterThreads = 512, kIterWarps = kIterThreads / 32;  // k_agg_iter_windows
constexpr u32 kMaxParts = 16;            // blocks that share a stream in the passes over the records

struct AggArgs {
  const argus_interval_t* intervals;
  const u64* interval_offsets;
  const argus_ambiguity_t* ambig;
  const u64* ambig_offsets;
  u32 num_streams, warps_per_cta, num_ctas, num_sms, num_regions;
  const u32* cta_sm;
  u64* warp_tab;  // [S][R][72] (caller's table or workspace)
  u64* sm_tab;    // nullable
  u64* kernel_tab;  // nullable
  argus_status_t* status;
  // scope selection
  int scoped;
  u32 ctx_lo, ctx_hi;
  u64 warp_mask;
  const u32* sm_mask;
  const u32* region_mask;
  u64* role_tab;  // [W][R][72], nullable
  u64* iter_tab;  // [num_iters][R][72], nullable
  u32 num_iters;
  ulonglong2* ranges; // [S][parts] first and last + 1 interval of the part that is in the iteration window (null: not asked for)
  // overlap selection in the pass over the digests (argus_synthesize)
  ArgusFuseArgs ov;
  u32 parts;          // blocks that share a stream
  u32 slices;         // k_agg_streams_digest: slices of a stream, one per warp of its blocks
  const u64* digest;  // digests of the intervals (k_agg_streams_digest; overwritten with entries where overlap is selected), null = read the records
  u64 interval_limit; // records the interval array holds: a stream whose offsets reach beyond it is reported, not read
};

// The tables that the kernels after the one that calls this add to start empty.
__device__ __forceinline__ void agg_empty_tables(const AggArgs& a) {
  const u64 first = (u64)blockIdx.x * blockDim.x + threadIdx.x, stride = (u64)gridDim.x * blockDim.x, row = (u64)a.num_regions * kCell;
  if (a.sm_tab) for (u64 i = first; i < a.num_sms * row; i += stride) a.sm_tab[i] = (i % kCell == 2) ? ~0ull : 0ull;
  if (a.kernel_tab) for (u64 i = first; i < row; i += stride) a.kernel_tab[i] = (i % kCell == 2) ? ~0ull : 0ull;
  if (a.role_tab) for (u64 i = first; i < a.warps_per_cta * row; i += stride) a.role_tab[i] = (i % kCell == 2) ? ~0ull : 0ull;
  if (a.iter_tab) for (u64 i = first; i < a.num_iters * row; i += stride) a.iter_tab[i] = (i % kCell == 2) ? ~0ull : 0ull;
}

__device__ __forceinline__ bool mask_bit(const u32* mask, u32 i) { return !mask || ((mask[i >> 5] >> (i & 31)) & 1u); }

__device__ __forceinline__ void bad_sm(const AggArgs& a, u32 cta) { argus_report_bad_sm(a.status, a.cta_sm, a.num_sms, a.warps_per_cta, cta); }

// Warp-role and SM tests of a scope: one answer per stream. 2 = bad cta_sm entry.
__device__ __forceinline__ int stream_in_scope(const AggArgs& a, u32 s) {
  if (!a.scoped) return 1;
  const u32 w = s % a.warps_per_cta;
  if (a.warp_mask != ~0ull && (w >= 64 || !((a.warp_mask >> w) & 1ull))) return 0;
  if (a.sm_mask) {
    const u32 m = a.cta_sm[s / a.warps_per_cta];
    if (m >= a.num_sms) return 2;
    if (!mask_bit(a.sm_mask, m)) return 0;
  }
  return 1;
}

// Iteration-window and region tests of a scope: one answer per record.
__device__ __forceinline__ bool record_in_scope(const AggArgs& a, u32 ctx, u32 region) {
  return !a.scoped || (ctx >= a.ctx_lo && ctx <= a.ctx_hi && mask_bit(a.region_mask, region));
}

__device__ __forceinline__ u32 log2_bin(u64 d) { return d ? 63u - (u32)__clzll((long long)d) : 0u; }

__device__ __forceinline__ void agg_add_interval(u64* tab, u32 region, u64 incl, u64 excl, u32 flags) {
  u64* c = tab + (size_t)region * kCell;
  atomicAdd(c + 0, 1ull);
  atomicAdd(c + 1, incl);
  atomicMin(c + 2, incl);
  atomicMax(c + 3, incl);
  atomicAdd(c + 4, excl);
  if (flags) atomicAdd(c + 7, 1ull);
  atomicAdd(c + 8 + log2_bin(incl), 1ull);
}

__global__ void __launch_bounds__(kAggThreads) k_agg_streams(AggArgs a) {
  argus_kernel_begin_long();
  agg_empty_tables(a);
  const u32 R = a.num_regions;
  const u32 cells = R * kCell;
  for (u32 s = blockIdx.x; s < a.num_streams; s += gridDim.x) {
    u64* row = a.warp_tab + (size_t)s * cells;
    for (u32 i = threadIdx.x; i < cells; i += blockDim.x) row[i] = (i % kCell == 2) ? ~0ull : 0ull;
    __threadfence();
    __syncthreads();
    const u64 lo = a.interval_offsets[s], hi = a.interval_offsets[s + 1];
    const int sel = stream_in_scope(a, s);
    if (sel == 2 && threadIdx.x == 0) bad_sm(a, s / a.warps_per_cta);
    if (hi < lo || hi > a.interval_limit) {
      if (threadIdx.x == 0) argus_set_error(a.status, ARGUS_ERR_BAD_OFFSETS, s, 0);
    } else if (sel == 1) {
      for (u64 i = lo + threadIdx.x; i < hi; i += blockDim.x) {
        const uint4* p = reinterpret_cast<const uint4*>(a.intervals + i);
        const uint4 q0 = __ldg(p), q1 = __ldg(p + 1), q2 = __ldg(p + 2);
        const u64 incl = (u64)q0.z | ((u64)q0.w << 32);
        const u64 excl = (u64)q1.x | ((u64)q1.y << 32);
        const u32 region = q1.z;
        if (region >= R) { argus_set_error(a.status, ARGUS_ERR_BAD_REGION, s, i); continue; }
        if (!record_in_scope(a, q1.w, region)) continue;
        agg_add_interval(row, region, incl, excl, q2.w >> 16);
      }
    }
    if (a.ambig && a.ambig_offsets && sel == 1) {
      const u64 alo = a.ambig_offsets[s], ahi = a.ambig_offsets[s + 1];
      for (u64 i = alo + threadIdx.x; i < ahi && ahi >= alo; i += blockDim.x) {
        const u32 region = a.ambig[i].tag >> 1;
        if (region >= R) { argus_set_error(a.status, ARGUS_ERR_BAD_REGION, s, i); continue; }
        if (!record_in_scope(a, a.ambig[i].ctx, region)) continue;
        atomicAdd(row + (size_t)region * kCell + (a.ambig[i].kind == ARGUS_AMBIG_UNMATCHED_END ? 6 : 5), 1ull);
      }
    }
  }
}

__global__ void __launch_bounds__(kAggThreads) k_agg_streams_compact(AggArgs a) {
  argus_kernel_begin_long();
  agg_empty_tables(a);
  extern __shared__ __align__(128) unsigned char sh_raw[];
  __shared__ u64 range[2];
  ArgusAggCell* const ctab = reinterpret_cast<ArgusAggCell*>(sh_raw);
  const u32 R = a.num_regions;
  const u32 cells = R * kCell;
  const u32 s = blockIdx.x / a.parts, part = blockIdx.x % a.parts;
  u64* row = a.warp_tab + (size_t)s * cells;
  // the global row takes bins outside the windows and the ambiguity counters directly
  if (a.parts == 1)  // (else the rows have been initialised: several blocks add to one)
    for (u32 i = threadIdx.x; i < cells; i += blockDim.x) row[i] = (i % kCell == 2) ? ~0ull : 0ull;
  argus_fuse_init(ctab, R, threadIdx.x, blockDim.x);
  if (threadIdx.x == 0) { range[0] = ~0ull; range[1] = 0; }
  __threadfence();
  __syncthreads();
  ArgusFuseCtx fx;
  fx.tab = ctab; fx.row = row;
  u64 lo = a.interval_offsets[s], hi = a.interval_offsets[s + 1];
  const int sel = stream_in_scope(a, s);
  if (sel == 2 && threadIdx.x == 0) bad_sm(a, s / a.warps_per_cta);
  if (hi < lo || hi > a.interval_limit) {
    if (threadIdx.x == 0) argus_set_error(a.status, ARGUS_ERR_BAD_OFFSETS, s, 0);
  } else if (sel == 1) {
    if (a.parts > 1) {
      const u64 per = (hi - lo + a.parts - 1) / a.parts;
      const u64 from = lo + per * part;
      lo = from < hi ? from : hi;
      hi = lo + per < hi ? lo + per : hi;
    }
    u64 first = ~0ull, last = 0;
    for (u64 i = lo + threadIdx.x; i < hi; i += blockDim.x) {
      const uint4* p = reinterpret_cast<const uint4*>(a.intervals + i);
      const uint4 q0 = __ldg(p), q1 = __ldg(p + 1), q2 = __ldg(p + 2);
      const u32 region = q1.z;
      if (region >= R) { argus_set_error(a.status, ARGUS_ERR_BAD_REGION, s, i); continue; }
      if (!record_in_scope(a, q1.w, region)) continue;
      const u64 incl = (u64)q0.z | ((u64)q0.w << 32), excl = (u64)q1.x | ((u64)q1.y << 32);
      argus_fuse_aggregate(fx, region, incl, excl, q2.w >> 16);
      if (first == ~0ull) first = i;
      last = i + 1;
    }
    if (a.ranges && last) { atomicMin(&range[0], first); atomicMax(&range[1], last); }
  }
  if (a.ambig && a.ambig_offsets && sel == 1 && part == 0) {
    const u64 alo = a.ambig_offsets[s], ahi = a.ambig_offsets[s + 1];
    for (u64 i = alo + threadIdx.x; i < ahi && ahi >= alo; i += blockDim.x) {
      const u32 region = a.ambig[i].tag >> 1;
      if (region >= R) { argus_set_error(a.status, ARGUS_ERR_BAD_REGION, s, i); continue; }
      if (!record_in_scope(a, a.ambig[i].ctx, region)) continue;
      atomicAdd(row + (size_t)region * kCell + (a.ambig[i].kind == ARGUS_AMBIG_UNMATCHED_END ? 6 : 5), 1ull);
    }
  }
  __syncthreads();
  if (a.ranges && threadIdx.x == 0) a.ranges[blockIdx.x] = make_ulonglong2(range[0], range[1]);
  argus_fuse_flush(ctab, row, R, threadIdx.x, blockDim.x);
}

// ---- the pass over the intervals' 8-byte digests (what argus_synthesize's pairing wrote beside the records) ----
// One block per stream (or several), no scope. The stream's row is gathered in shared memory in cells of kDgWords = 31 32-bit
// words (an odd size: the cells of 32 different regions start in 32 different banks) that hold all the 23 histogram bins a
// digest can fall into. All words start at zero: the minimum is kept as the maximum of the complement. A few regions usually
// own most intervals of a stream, and 32 lanes adding to one address serialise; so after a count of the regions in the first
// round of every warp the kDigestHot most frequent ones get copies of their cell, lanes apart (consecutive cells: rarely a
// bank conflict), which are folded into the region's cell when the stream ends. meta[region] holds the byte address of the
// cell to add to, whether it is one of the copies, and whether the region appears in an overlap pair. What does not count (past
// the end, a bad region, a digest marked wide) goes to a cell of its own that nobody reads, so that the common case has no
// selects. Every warp walks a slice of the stream, so that overlap candidates stay in order; their entries replace digests that
// the warp has consumed: no list, no atomics. The row is written once, with plain stores; wide intervals (a duration of 2^23
// ticks or more) are added to it afterwards, from their records, by the warps that saw one.
constexpr u32 kDigestHot = 4;
constexpr u32 kDgSumInclLo = 0, kDgSumInclHi = 1, kDgSumExclLo = 2, kDgSumExclHi = 3, kDgNotMin = 4, kDgMax = 5, kDgFlag = 6,
              kDgBins = 7, kDgCount = kDgBins + kDigestBits, kDgWords = kDgCount + 1;
static_assert(kDgWords % 2 == 1, "an odd cell size keeps the cells of different regions in different banks");
constexpr u32 kDgHot = 1u << 31, kDgInPair = 1u << 30, kDgNoRegion = 1u << 29, kDgAddr = (1u << 18) - 1;  // meta
constexpr u64 kDgPad = 0xffffull;              // what a lane past the end looks at: no such region

// cells of the regions, the cell that nobody reads, copies; then meta for each region and for no region
__host__ __device__ constexpr u32 digest_cell_words(u32 R, u32 copies) { return (kDgWords * (R + 1 + kDigestHot * copies) + 3) & ~3u; }
__host__ __device__ constexpr size_t digest_table_bytes(u32 R, u32 copies) { return 4 * ((size_t)digest_cell_words(R, copies) + R + 1 + (R + 31) / 32); }

template <u32 F> __device__ __forceinline__ u32 dg_add(u32 cell, u32 v) {  // returns the old value
  u32 old;
  asm volatile("atom.shared.add.u32 %0, [%1+%3], %2;" : "=r"(old) : "r"(cell), "r"(v), "n"(F * 4) : "memory");
  return old;
}
template <u32 F> __device__ __forceinline__ void dg_inc(u32 cell, u32 v) {
  asm volatile("red.shared.add.u32 [%0+%2], %1;" :: "r"(cell), "r"(v), "n"(F * 4) : "memory");
}
template <u32 F> __device__ __forceinline__ void dg_max(u32 cell, u32 v) {
  asm volatile("red.shared.max.u32 [%0+%2], %1;" :: "r"(cell), "r"(v), "n"(F * 4) : "memory");
}

// A wide interval, from its record, with atomics on the global row.
__device__ __noinline__ void digest_wide(u64* row, u32 R, uint4 q0, uint4 q1, u32 flags) {
  if (q1.z >= R) return;
  u64* const c = row + (size_t)q1.z * kCell;
  const u64 span = (u64)q0.z | ((u64)q0.w << 32);
  atomicAdd(c + 0, 1ull);
  atomicAdd(c + 1, span);
  atomicMin(c + 2, span);
  atomicMax(c + 3, span);
  atomicAdd(c + 4, (u64)q1.x | ((u64)q1.y << 32));
  if (flags) atomicAdd(c + 7, 1ull);
  atomicAdd(c + 8 + log2_bin(span), 1ull);
}

// The regions' cells of a stream into its row, 16 bytes at a time where one block has gathered it (`alone`; else the rows have been
// initialised and several blocks add): a warp takes a region's bins, of which the upper ones are empty, a lane two of them, and then eight
// regions' other fields. (A word at a time, a field for a thread, took 24 warp instructions for 32 words; 36 lanes' worth of a
// region in a row, bins and fields in one warp, more: 71 M digests, 2,368 rows of 202 regions 260 us, 281 and 250 so.)
template <u32 kWords, u32 kBins, u32 kThreads>
__device__ __forceinline__ void row_out(const u32* tab, u64* row, u32 R, bool alone) {
  static_assert(kCell == 72 && kBins <= 32, "eight fields, then 32 pairs of bins");
  const u32 lane = threadIdx.x & 31;
  const bool vectors = alone && !(reinterpret_cast<uintptr_t>(row) & 15);
  for (u32 r = threadIdx.x / 32; r < R; r += kThreads / 32) {
    const u32* const c = tab + r * kWords + kDgBins + 2 * lane;
    const u64 x = 2 * lane < kBins ? c[0] : 0u, y = 2 * lane + 1 < kBins ? c[1] : 0u;
    u64* const p = row + (size_t)r * kCell + 8 + 2 * lane;
    if (vectors) {
      *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(x, y);
    } else if (alone) {
      p[0] = x; p[1] = y;
    } else {
      if (x) atomicAdd(p, x);
      if (y) atomicAdd(p + 1, y);
    }
  }
  for (u32 k = threadIdx.x; k < 4 * R; k += kThreads) {
    const u32 v = k & 3;
    const u32* const c = tab + (k >> 2) * kWords;
    u64 x = 0, y = 0;
    if (v == 0) {
#pragma unroll
      for (u32 j = 0; j < kBins; ++j) x += c[kDgBins + j];
    }
    if (v == 1) { const u32 least = c[kDgNotMin]; x = least ? (u64)(u32)~least : ~0ull; y = c[kDgMax]; }
    if ((v & 1) == 0) {
      const u32 at = v ? kDgSumExclLo : kDgSumInclLo;
      (v ? x : y) = (u64)c[at] | ((u64)c[at + 1] << 32);
    }
    if (v == 3) y = c[kDgFlag];  // (ambiguity records are added later)
    u64* const p = row + (size_t)(k >> 2) * kCell + 2 * v;
    if (vectors) {
      *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(x, y);
    } else if (alone) {
      p[0] = x; p[1] = y;
    } else if (v == 1) {
      if (x != ~0ull) atomicMin(p, x);
      if (y) atomicMax(p + 1, y);
    } else {
      if (x) atomicAdd(p, x);
      if (y) atomicAdd(p + 1, y);
    }
  }
}

// Bound by instruction issue and the atomics' way through the load/store pipe. Bins that need no window, a trash cell instead of
// selects, a row written once instead of emptied, added to and read back, and a loop of two rounds (the digests asked for
// ahead change places without moves): decode trace (307 M intervals) 1,215 -> 903 us = 2.7 TB/s of digests, attention 400 -> 323,
// GEMM 234 -> 188. Unrolled once 1,017, three times 898 (GEMM 191), four times 913. What a stream costs before its first
// interval and after its last one (85 us of the decode trace's 903) decides for short ones: fewer threads for them and eight
// copies instead of 32, so that more streams are on the chip (see argus_aggregate_digest_slices). Whole rounds without a look at the end of the
// slice, one flag for a region that does not exist, and 16 copies instead of 32 in the large blocks: half of the decode trace 487 -> 465,
// attention 321 -> 311, GEMM 186 -> 182.
template <u32 kThreads, u32 kCopies, u32 kBlocks>
__global__ void __launch_bounds__(kThreads, kBlocks) k_agg_streams_digest(AggArgs a) {
  constexpr u32 kMinProbe = 4 * kThreads;    // shorter streams are gathered without copies
  constexpr u32 kSlices = kThreads / 32;   // slices of a stream, one per warp (also the slices of the overlap entries)
  extern __shared__ __align__(128) unsigned char sh_raw[];
  const u32 R = a.num_regions;
  u32* const tab = reinterpret_cast<u32*>(sh_raw);
  u32* const meta = tab + digest_cell_words(R, kCopies);
  u32* const pairbits = meta + R + 1;
  __shared__ u32 hot_region[kDigestHot], often[64], num_often;
  const u32 tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const u32 tab_addr = (u32)__cvta_generic_to_shared(tab);
  const bool has_ov = a.ov.num_pairs != 0;
  const u32 s = blockIdx.x / a.parts, part = blockIdx.x % a.parts;
  for (u32 i = tid; i < digest_cell_words(R, kCopies) / 4; i += kThreads) reinterpret_cast<uint4*>(tab)[i] = make_uint4(0, 0, 0, 0);
  for (u32 i = tid; i < (R + 31) / 32; i += kThreads) pairbits[i] = 0;
  if (tid < kDigestHot) hot_region[tid] = 0xffffffffu;
  if (tid == 0) num_often = 0;
  argus_kernel_begin_long();
  agg_empty_tables(a);
  if (has_ov && blockIdx.x == 0 && tid == 0) *a.ov.ctl = ArgusOvCtl{};
  const u64 lo = a.interval_offsets[s], hi = a.interval_offsets[s + 1];
  u64* const row = a.warp_tab + (size_t)s * R * kCell;
  __syncthreads();
  if (has_ov) {
    for (u32 i = tid; i < 2 * a.ov.num_pairs; i += kThreads) {
      const u32 r = a.ov.pairs[i];
      if (r < R) atomicOr(&pairbits[r >> 5], 1u << (r & 31));
    }
    __syncthreads();
  }
  for (u32 r = tid; r <= R; r += kThreads)
    meta[r] = (tab_addr + r * (kDgWords * 4)) | (r == R ? kDgNoRegion : (pairbits[r >> 5] >> (r & 31)) & 1u ? kDgInPair : 0u);
  if (has_ov && tid == 0) {
    const u32 m = a.cta_sm[s / a.warps_per_cta];
    if (m >= a.num_sms) bad_sm(a, s / a.warps_per_cta);
  }
  const bool good = hi >= lo && hi <= a.interval_limit && !((hi - lo) >> 32);
  if (!good && tid == 0) argus_set_error(a.status, ARGUS_ERR_BAD_OFFSETS, s, 0);
  const u32 n = good ? (u32)(hi - lo) : 0u;
  const u64* const dgs = a.digest + lo;
  const argus_interval_t* const ivs = a.intervals + lo;
  u32 i0, i1;
  argus_ov_slice(n, a.slices, part * kSlices + warp, &i0, &i1);
  u64* const ents = a.ov.entries + lo + i0;
  u64* const starts = a.ov.starts + lo + i0;
  // digests are asked for two rounds ahead (one round is shorter than a loaded DRAM access)
  u32 i = i0 + lane;
  u64 dg_next = i < i1 ? dgs[i] : kDgPad;
  u64 dg_next2 = i + 32 < i1 ? dgs[i + 32] : kDgPad;
  __syncthreads();
  if (n / a.parts >= kMinProbe) {  // the regions that the first round of every warp sees most
    const u32 region = (u32)dg_next & 0xffffu;
    if (region < R) dg_inc<kDgCount>(tab_addr + region * (kDgWords * 4), 1u);
    __syncthreads();
    for (u32 r = tid; r < R; r += kThreads) {
      const u32 cnt = tab[r * kDgWords + kDgCount];
      if (cnt >= kThreads / 64) often[atomicAdd(&num_often, 1u)] = (cnt << 16) | r;  // at most 64 of them
    }
    __syncthreads();
    if (tid < num_often) {
      const u32 key = often[tid], r = key & 0xffffu;
      u32 rank = 0;
      for (u32 k = 0; k < num_often; ++k) rank += often[k] > key;
      if (rank < kDigestHot) {
        hot_region[rank] = r;
        meta[r] = (tab_addr + (R + 1 + rank * kCopies) * (kDgWords * 4)) | kDgHot | (meta[r] & kDgInPair);
      }
    }
    __syncthreads();
  }
  // every lane of a warp runs the same number of rounds, so that entries can be appended a warp at a time
  const u32 own_copy = lane % kCopies * (kDgWords * 4);
  u32 out_count = 0;  // warp-uniform: entries of the warp's slice
  bool wide = false;  // the lane met a wide digest
  bool late = false;  // the lane's candidate of the round before: its begin time may still be on its way
  u64 late_t0 = 0;
  u64* late_start = nullptr;
  auto round = [&](u64 dg, auto FULL) {
    const u32 dlo = (u32)dg, dhi = (u32)(dg >> 32);
    const u32 region = dlo & 0xffffu;
    const u32 m = meta[min(region, R)];
    const u32 incl = __funnelshift_r(dlo, dhi, 18) & ((1u << kDigestBits) - 1), excl = dhi >> (32 - kDigestBits);
    const u32 normal = (m & kDgAddr) + (m >> 31) * own_copy;
    const u32 cell = dlo & kDigestWide ? tab_addr + R * (kDgWords * 4) : normal;
    const u32 old_i = dg_add<kDgSumInclLo>(cell, incl);
    const u32 old_e = dg_add<kDgSumExclLo>(cell, excl);
    dg_max<kDgNotMin>(cell, ~incl);
    dg_max<kDgMax>(cell, incl);
    dg_inc<kDgBins>(cell + (31u - (u32)__clz((int)(incl | 1u))) * 4, 1u);
    bool cand = (m & kDgInPair) && incl;
    // whatever is rare (a carry, a flag, a wide digest, no such region) is settled in one place
    if (old_i > ~incl || old_e > ~excl || ((dlo & (kDigestFlag | kDigestWide)) | (m & kDgNoRegion))) {
      if (m & kDgNoRegion) {
        if (decltype(FULL)::value || i < i1) argus_set_error(a.status, ARGUS_ERR_BAD_REGION, s, lo + i);
      } else if (dlo & kDigestWide) {
        wide = true;
        cand = m & kDgInPair;  // (its inclusive duration is not 0: the exclusive one is never longer)
      } else {
        if (old_i > ~incl) dg_inc<kDgSumInclHi>(cell, 1u);
        if (old_e > ~excl) dg_inc<kDgSumExclHi>(cell, 1u);
        if (dlo & kDigestFlag) dg_inc<kDgFlag>(cell, 1u);
      }
    }
    const u32 bal = __ballot_sync(0xffffffffu, cand);
    if (late) late_start[0] = late_t0;  // asked for a round ago
    late = cand;
    if (bal) {  // (the entries of a slice never reach the digests that are still to be read)
      if (cand) {
        const u32 at = out_count + __popc(bal & ((1u << lane) - 1u));
        ents[at] = argus_entry_pack(dg, i - i0);
        late_start = starts + at;
        late_t0 = __ldg(reinterpret_cast<const u64*>(ivs + i));
      }
      out_count += __popc(bal);
    }
  };
  u32 b = i0;
#pragma unroll 2
  for (; b + 96 <= i1; b += 32, i += 32) {  // whole rounds, and those asked for as well
    const u64 dg = dg_next;
    dg_next = dg_next2;
    dg_next2 = dgs[i + 64];
    round(dg, std::true_type{});
  }
#pragma unroll 1
  for (; b < i1; b += 32, i += 32) {
    const u64 dg = dg_next;
    dg_next = dg_next2;
    dg_next2 = i + 64 < i1 ? dgs[i + 64] : kDgPad;
    round(dg, std::false_type{});
  }
  if (late) late_start[0] = late_t0;
  if (has_ov && lane == 0) {
    ArgusOvPiece e;
    e.pos = lo + (good ? i0 : 0u); e.count = out_count; e.next = kOvNone;
    a.ov.pieces[s * a.slices + part * kSlices + warp] = e;
  }
  __syncthreads();
  // the copies into their region's cell (which nobody added to): a thread per (hot region, field)
  if (tid < kDigestHot * kDgCount) {
    const u32 h = tid / kDgCount, f = tid % kDgCount, r = hot_region[h];
    if (r != 0xffffffffu && f != kDgSumInclHi && f != kDgSumExclHi) {
      const u32* src = tab + (R + 1 + h * kCopies) * kDgWords + f;
      u32* dst = tab + r * kDgWords + f;
      const bool sum = f == kDgSumInclLo || f == kDgSumExclLo, most = f == kDgNotMin || f == kDgMax;
      u64 acc = 0;
#pragma unroll 8
      for (u32 l = 0; l < kCopies; ++l) {
        const u32 v = src[l * kDgWords];
        if (sum) acc += (u64)v | ((u64)src[l * kDgWords + 1] << 32);
        else acc = most ? (v > acc ? v : acc) : acc + v;
      }
      dst[0] = (u32)acc;
      if (sum) dst[1] = (u32)(acc >> 32);
    }
  }
  __syncthreads();
  // the regions' cells into the global row
  row_out<kDgWords, kDigestBits, kThreads>(tab, row, R, a.parts == 1);
  u64 alo = 0, ahi = 0;
  if (a.ambig && a.ambig_offsets && part == 0) { alo = a.ambig_offsets[s]; ahi = a.ambig_offsets[s + 1]; }
  wide = __any_sync(0xffffffffu, wide);
  if (!__syncthreads_or(wide || alo < ahi)) return;
  __threadfence();
  __syncthreads();
  if (wide) {  // (where entries have replaced the digests, the records tell)
    for (u32 k = i0 + lane; k < i1; k += 32) {
      const bool gone = k - i0 < out_count;
      if (!gone && !((u32)dgs[k] & kDigestWide)) continue;
      const uint4* p = reinterpret_cast<const uint4*>(ivs + k);
      const uint4 q0 = __ldg(p), q1 = __ldg(p + 1), q2 = __ldg(p + 2);
      const u32 too_long = ((q0.z | q1.x) >> kDigestBits) | q0.w | q1.y;
      if (too_long) digest_wide(row, R, q0, q1, q2.w >> 16);
    }
  }
  for (u64 k = alo + tid; k < ahi; k += kThreads) {
    const u32 region = a.ambig[k].tag >> 1;
    if (region >= R) { argus_set_error(a.status, ARGUS_ERR_BAD_REGION, s, k); continue; }
    atomicAdd(row + (size_t)region * kCell + (a.ambig[k].kind == ARGUS_AMBIG_UNMATCHED_END ? 6 : 5), 1ull);
  }
}

__global__ void __launch_bounds__(256) k_agg_init(u64* tab, u64 n) {
  argus_kernel_begin();
  for (u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (u64)gridDim.x * blockDim.x)
    tab[i] = (i % kCell == 2) ? ~0ull : 0ull;
}

// One word of the cells of kGroup CTAs: CTA cells = reduction over the warps of each (written if asked for), warp-role cells over
// the CTAs; CTA cells go to the SM-scope cells, their reduction over the group to the kernel-scope cells (atomic add / max
// on integers; empty words add nothing). A minimum is taken as the maximum of complements, so that a word is either added or compared.
// Bound by the one read of the warp-scope table. 275 MB, us without roles / with them, one, two, four and eight CTAs a thread: 60 / 113, 55 /
// 86, 67 / 61 and 77 / 98; with three ways to combine for every word, and for the roles whether asked for or not (40 M warp
// instructions, issued on 60 % of the cycles), eight took 69 / 83. Five regions, 1,776 streams: 9.3 -> 7.0.
__device__ __forceinline__ void cell_add(u64* d, u32 field, u64 v) {  // (v: as roll_in gives it)
  if (v == 0ull) return;  // nothing to add
  if (field == 2) atomicMin(d, ~v); else if (field == 3) atomicMax(d, v); else atomicAdd(d, v);
}
__device__ __forceinline__ u64 roll_in(bool most, u64 flip, u64 v, u64 x) {
  x ^= flip;
  if (most) return x > v ? x : v;
  return v + x;
}
template <u32 kGroup, bool kRoles>
__global__ void __launch_bounds__(256) k_agg_rollup(AggArgs a, u64* cta_out) {
  argus_kernel_begin_long();
  const u64 per_cta = (u64)a.num_regions * kCell, n = (u64)((a.num_ctas + kGroup - 1) / kGroup) * per_cta;
  for (u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (u64)gridDim.x * blockDim.x) {
    const u32 c0 = (u32)(i / per_cta) * kGroup, have = a.num_ctas - c0 < kGroup ? a.num_ctas - c0 : kGroup;
    const u64 rem = i % per_cta;
    const u32 field = (u32)(rem % kCell);
    const bool most = field == 2 || field == 3;
    const u64 flip = field == 2 ? ~0ull : 0ull;
    const u64* src = a.warp_tab + (u64)c0 * a.warps_per_cta * per_cta + rem;
    const u64 cta = a.warps_per_cta * per_cta;
    u64 v[kGroup];
#pragma unroll
    for (u32 q = 0; q < kGroup; ++q) v[q] = 0;
    if (have == kGroup) {
#pragma unroll kGroup <= 2 ? 8 : 2
      for (u32 w = 0; w < a.warps_per_cta; ++w, src += per_cta) {
        u64 x[kGroup];
#pragma unroll
        for (u32 q = 0; q < kGroup; ++q) x[q] = __ldcg(src + q * cta);
#pragma unroll
        for (u32 q = 0; q < kGroup; ++q) v[q] = roll_in(most, flip, v[q], x[q]);
        if (kRoles) {
          u64 all = 0;
#pragma unroll
          for (u32 q = 0; q < kGroup; ++q) all = roll_in(most, flip, all, x[q]);
          cell_add(a.role_tab + w * per_cta + rem, field, all);
        }
      }
    } else {
      for (u32 w = 0; w < a.warps_per_cta; ++w, src += per_cta) {
        u64 all = 0;
#pragma unroll
        for (u32 q = 0; q < kGroup; ++q) {
          if (q >= have) break;
          const u64 x = __ldcg(src + q * cta);
          v[q] = roll_in(most, flip, v[q], x);
          all = roll_in(most, flip, all, x);
        }
        if (kRoles) cell_add(a.role_tab + w * per_cta + rem, field, all);
      }
    }
    u64 all = 0;
#pragma unroll
    for (u32 q = 0; q < kGroup; ++q) {
      if (q >= have) break;
      if (cta_out) cta_out[(u64)(c0 + q) * per_cta + rem] = v[q] ^ flip;
      if (a.sm_tab && v[q] != 0ull) {
        const u32 m = a.cta_sm[c0 + q];
        if (m >= a.num_sms) { bad_sm(a, c0 + q); continue; }
        cell_add(a.sm_tab + (u64)m * per_cta + rem, field, v[q]);
      }
      all = roll_in(most, 0ull, all, v[q]);
    }
    if (a.kernel_tab) cell_add(a.kernel_tab + rem, field, all);
  }
}

constexpr u32 kIterCopies = 8;  // of the cells of the kDigestHot most frequent regions
constexpr u32 kItWords = kDgBins + 32;  // a cell: as in the pass over the digests, but with all bins of 32-bit durations (also an odd size)
static_assert(kItWords % 2 == 1, "an odd cell size keeps the cells of different regions in different banks");
__host__ __device__ constexpr u32 iter_cells(u32 R) { return R + kDigestHot * kIterCopies; }
__host__ __device__ constexpr size_t iter_bytes(u32 R) { return 4 * (2 * (size_t)kItWords * iter_cells(R) + R + 4); }

__device__ __forceinline__ void iter_add(u32 cell, u32 incl, u32 excl, u32 flags) {
  const u32 old_i = dg_add<kDgSumInclLo>(cell, incl), old_e = dg_add<kDgSumExclLo>(cell, excl);
  dg_max<kDgNotMin>(cell, ~incl);
  dg_max<kDgMax>(cell, incl);
  dg_inc<kDgBins>(cell + (31u - (u32)__clz((int)(incl | 1u))) * 4, 1u);
  if (old_i > ~incl) dg_inc<kDgSumInclHi>(cell, 1u);
  if (old_e > ~excl) dg_inc<kDgSumExclHi>(cell, 1u);
  if (flags) dg_inc<kDgFlag>(cell, 1u);
}

// Adds the cells of an iteration to its row of the table, and empties them. A thread a cell.
__device__ __forceinline__ void iter_flush(u32* cells, const u32* hot_region, u64* row, u32 R) {
  for (u32 i = threadIdx.x; i < iter_cells(R); i += kIterThreads) {
    const u32 r = i < R ? i : hot_region[(i - R) / kIterCopies];
    if (r >= R) continue;
    u32* const c = cells + i * kItWords;
    u64* const g = row + (size_t)r * kCell;
    u32 cnt = 0;
#pragma unroll
    for (u32 j = 0; j < 32; ++j) {
      const u32 v = c[kDgBins + j];
      if (v) { atomicAdd(g + 8 + j, (u64)v); c[kDgBins + j] = 0; }
      cnt += v;
    }
    if (!cnt) continue;
    atomicAdd(g + 0, (u64)cnt);
    atomicAdd(g + 1, (u64)c[kDgSumInclLo] | ((u64)c[kDgSumInclHi] << 32));
    atomicMin(g + 2, (u64)~c[kDgNotMin]);
    atomicMax(g + 3, (u64)c[kDgMax]);
    atomicAdd(g + 4, (u64)c[kDgSumExclLo] | ((u64)c[kDgSumExclHi] << 32));
    if (c[kDgFlag]) atomicAdd(g + 7, (u64)c[kDgFlag]);
#pragma unroll
    for (u32 f = 0; f < kDgBins; ++f) c[f] = 0;
  }
}

// ---- the pass over the records (argus_aggregate) ----
// One block per stream (or several), as in the pass over the digests: the stream's row in cells of 32-bit words, with copies of the most
// frequent regions' cells, lanes apart, and the row written once. An interval of 2^32 ticks and more is added to the row
// afterwards, by the lanes that met one. Bound by HBM where streams are long; the records come by bulk copies, because the cells leave
// little L1 for what three loads of a lane have in common. k_agg_streams_compact with its 64-bit cells, of which 32 lanes often want the
// same one, and compare-and-swap loops for minimum and maximum, took (us, then / now): 12.5 M records of 5 regions 162 / 119, 34 M 385 /
// 293, 42 M of 202 regions 700 / 626, 1.7 M 139 / 72, 207,000 18.5 / 17.3; but of a scope that selects a third of 115 M records 931 /
// 1,026, because nothing is added for most records and eight blocks of it fit an SM instead of three.
constexpr u32 kRecCopies = 8;
constexpr u32 kRecStages = 2;
__host__ __device__ constexpr u32 record_tile_bytes(u32 threads) { return threads * (u32)sizeof(argus_interval_t); }  // a record a thread
__host__ __device__ constexpr u32 record_cell_words(u32 R) { return (kItWords * (R + kDigestHot * kRecCopies) + 3) & ~3u; }
__host__ __device__ constexpr size_t record_table_bytes(u32 R, u32 threads) {
  return kRecStages * record_tile_bytes(threads) + 4 * ((size_t)record_cell_words(R) + R);
}

template <u32 kThreads>
__global__ void __launch_bounds__(kThreads) k_agg_streams_records(AggArgs a) {
  constexpr u32 kRecTileBytes = record_tile_bytes(kThreads);
  extern __shared__ __align__(128) unsigned char sh_raw[];
  __shared__ u32 hot_region[kDigestHot], often[64], num_often;
  __shared__ u64 full[kRecStages];
  const u32 R = a.num_regions, tid = threadIdx.x, lane = tid & 31;
  u32 *const tab = reinterpret_cast<u32*>(sh_raw + kRecStages * kRecTileBytes), *const meta = tab + record_cell_words(R);
  const u32 tab_addr = (u32)__cvta_generic_to_shared(tab);
  if (tid == 0) {
#pragma unroll
    for (u32 k = 0; k < kRecStages; ++k) mbar_init(&full[k], 1);
    fence_mbar_init();
    num_often = 0;
  }
  argus_kernel_begin_long();
  const u32 s = blockIdx.x / a.parts, part = blockIdx.x % a.parts;
  u64* const row = a.warp_tab + (size_t)s * R * kCell;
  u64 lo = a.interval_offsets[s], hi = a.interval_offsets[s + 1];
  if (hi < lo || hi > a.interval_limit) {
    if (tid == 0) argus_set_error(a.status, ARGUS_ERR_BAD_OFFSETS, s, 0);
    lo = hi = 0;
  } else if (a.parts > 1) {
    const u64 per = (hi - lo + a.parts - 1) / a.parts;
    const u64 from = lo + per * part;
    lo = from < hi ? from : hi;
    hi = lo + per < hi ? lo + per : hi;
  }
  // a tile of records into its stage (thread 0)
  auto fetch = [&](u64 first_record, u32 stage) {
    const u32 bytes = hi - first_record < kThreads ? (u32)(hi - first_record) * (u32)sizeof(argus_interval_t) : kRecTileBytes;
    mbar_expect_tx(&full[stage], bytes);
    tma_load_1d(sh_raw + stage * kRecTileBytes, a.intervals + first_record, bytes, &full[stage]);
  };
  if (tid == 0) {
#pragma unroll
    for (u32 k = 0; k < kRecStages; ++k) if (lo + k * kThreads < hi) fetch(lo + k * kThreads, k);
  }
  for (u32 i = tid; i < record_cell_words(R) / 4; i += kThreads) reinterpret_cast<uint4*>(tab)[i] = make_uint4(0, 0, 0, 0);
  for (u32 r = tid; r < R; r += kThreads) meta[r] = tab_addr + r * (kItWords * 4);
  if (tid < kDigestHot) hot_region[tid] = 0xffffffffu;
  agg_empty_tables(a);
  __syncthreads();
  const u32 own_copy = lane % kRecCopies * (kItWords * 4);
  bool wide = false, arrived = true, lost = false;  // the lane met a wide interval; the copy has arrived; one has not
  u32 stage = 0, parity = 0;
  for (u64 at = lo; at < hi; at += kThreads) {
    arrived = mbar_wait_bounded(&full[stage], parity);
    const u64 i = at + tid;
    const u32* const p = reinterpret_cast<const u32*>(sh_raw + stage * kRecTileBytes) + tid * (sizeof(argus_interval_t) / 4);
    bool in = arrived && i < hi;
    const u32 region = in ? p[6] : 0u;
    if (region >= R) { argus_set_error(a.status, ARGUS_ERR_BAD_REGION, s, i); in = false; }
    if (at == lo && hi - lo >= 4 * kThreads) {  // the regions that the first tile has most get copies of their cells, lanes apart: 32 adds to one address take turns
      if (in) dg_inc<kDgBins>(tab_addr + region * (kItWords * 4), 1u);
      __syncthreads();
      for (u32 r = tid; r < R; r += kThreads) {
        const u32 cnt = tab[r * kItWords + kDgBins];
        tab[r * kItWords + kDgBins] = 0;
        if (cnt >= kThreads / 64) often[atomicAdd(&num_often, 1u)] = (cnt << 16) | r;  // at most 64 of them
      }
      __syncthreads();
      if (tid < num_often) {
        const u32 key = often[tid], r = key & 0xffffu;
        u32 rank = 0;
        for (u32 k = 0; k < num_often; ++k) rank += often[k] > key;
        if (rank < kDigestHot) { hot_region[rank] = r; meta[r] = (tab_addr + (R + rank * kRecCopies) * (kItWords * 4)) | kDgHot; }
      }
      __syncthreads();
    }
    if (in) {
      const uint2 incl = *reinterpret_cast<const uint2*>(p + 2), excl = *reinterpret_cast<const uint2*>(p + 4);
      if (incl.y | excl.y || incl.x == 0xffffffffu) {
        wide = true;
      } else {
        const u32 m = meta[region];
        iter_add((m & ~kDgHot) + (m >> 31) * own_copy, incl.x, excl.x, p[11] >> 16);
      }
    }
    lost = __syncthreads_or(!arrived);  // everybody has read the stage
    if (lost) break;
    if (tid == 0 && at + kRecStages * kThreads < hi) fetch(at + kRecStages * kThreads, stage);
    if (++stage == kRecStages) { stage = 0; parity ^= 1; }
  }
  if (lost) {  // a copy never arrived: reported, and what else is on its way is waited for (again with a limit)
    if (tid == 0) argus_set_error(a.status, ARGUS_ERR_TIMEOUT, s, 0);
    for (u32 k = 0; k < kRecStages; ++k) mbar_wait_bounded(&full[k], k >= stage ? parity : parity ^ 1u);
    __syncthreads();
  }
  // the copies into their region's cell (which nobody added to): a thread per (hot region, field)
  for (u32 hf = tid; num_often && hf < kDigestHot * kItWords; hf += kThreads) {
    const u32 h = hf / kItWords, f = hf % kItWords, r = hot_region[h];
    if (r != 0xffffffffu && f != kDgSumInclHi && f != kDgSumExclHi) {
      const u32* src = tab + (R + h * kRecCopies) * kItWords + f;
      u32* dst = tab + r * kItWords + f;
      const bool sum = f == kDgSumInclLo || f == kDgSumExclLo, most = f == kDgNotMin || f == kDgMax;
      u64 acc = 0;
#pragma unroll
      for (u32 l = 0; l < kRecCopies; ++l) {
        const u32 v = src[l * kItWords];
        if (sum) acc += (u64)v | ((u64)src[l * kItWords + 1] << 32);
        else acc = most ? (v > acc ? v : acc) : acc + v;
      }
      dst[0] = (u32)acc;
      if (sum) dst[1] = (u32)(acc >> 32);
    }
  }
  __syncthreads();
  // the regions' cells into the global row
  row_out<kItWords, 32, kThreads>(tab, row, R, a.parts == 1);
  u64 alo = 0, ahi = 0;
  if (a.ambig && a.ambig_offsets && part == 0) { alo = a.ambig_offsets[s]; ahi = a.ambig_offsets[s + 1]; }
  if (!__syncthreads_or(wide || alo < ahi)) return;
  __threadfence();
  __syncthreads();
  if (wide) {  // (the lane's records are looked at again)
    for (u64 k = lo + tid; k < hi; k += kThreads) {
      const uint4* p = reinterpret_cast<const uint4*>(a.intervals + k);
      const uint4 q0 = __ldg(p), q1 = __ldg(p + 1), q2 = __ldg(p + 2);
      if (q0.w | q1.y || q0.z == 0xffffffffu) digest_wide(row, R, q0, q1, q2.w >> 16);
    }
  }
  for (u64 k = alo + tid; k < ahi; k += kThreads) {
    const u32 r = a.ambig[k].tag >> 1;
    if (r >= R) { argus_set_error(a.status, ARGUS_ERR_BAD_REGION, s, k); continue; }
    atomicAdd(row + (size_t)r * kCell + (a.ambig[k].kind == ARGUS_AMBIG_UNMATCHED_END ? 6 : 5), 1ull);
  }
}

// iter_tab[ctx - ctx_lo][r] with cells as in the pass over the digests. A block walks a few streams side by side (kIterWarps warps, shared out
// among them) and holds the cells of two neighbouring iterations in shared memory; a warp that comes to a later one waits until
// all have, then the older cells are added to the table. Iterations come in order in a stream, so each is gathered once for
// all of the block's streams; atomics on the table for every interval took 2.0 ms where this took 550 us. An interval of an earlier
// iteration than the two, or of 2^32 ticks and more, is added to the table directly. Only the part of a stream that the pass before
// found to be in the window is read, a round ahead. What decides is how many lanes add to one address: with copies of the most
// frequent regions' cells, and a thread a cell where they are added to the table, the call with all tables goes from 1,616 to 1,508 us
// for 38 M intervals in 16 iterations of 202 regions, from 2,709 to 2,219 for 115 M in 48, and from 10.1 to 4.4 ms for 34 M in 2,000
// iterations of five regions. In the same pass as the rows (cells of one stream and iteration) the first took 2,107. More regions leave
// room for fewer blocks on an SM (136 KB at 400, where two tables of 112-byte cells took 90), which does not turn the gain: 112 M
// intervals of 292 regions, 16 of 32 iterations, 1,964 -> 1,743 us, 115 M of 400 regions, 16 of 24, 2,487 -> 2,390.
__global__ void __launch_bounds__(kIterThreads) k_agg_iter_windows(AggArgs a, u32 streams_per_block) {
  argus_kernel_begin_long();
  extern __shared__ __align__(128) unsigned char sh_raw[];
  __shared__ u32 need;
  const u32 R = a.num_regions, cells = R * kCell, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  u32 *const tab0 = reinterpret_cast<u32*>(sh_raw), *const tab1 = tab0 + kItWords * iter_cells(R), *const meta = tab1 + kItWords * iter_cells(R);
  const u32 addr0 = (u32)__cvta_generic_to_shared(tab0), addr1 = (u32)__cvta_generic_to_shared(tab1);
  __shared__ u32 hot_region[kDigestHot], often[64], num_often;
  constexpr u32 kNone = 0xffffffffu;
  const u32 m = kIterWarps / streams_per_block;  // warps of a stream
  const u32 s = blockIdx.x * streams_per_block + warp / m, mine = warp % m;
  u64 lo = ~0ull, hi = 0;
  if (s < a.num_streams && stream_in_scope(a, s) == 1) {  // (a bad cta_sm entry has been reported)
    for (u32 q = 0; q < a.parts; ++q) {
      const ulonglong2 r = a.ranges[(u64)s * a.parts + q];
      lo = r.x < lo ? r.x : lo;
      hi = r.y > hi ? r.y : hi;
    }
    if (mine == 0 && a.ambig && a.ambig_offsets) {
      const u64 alo = a.ambig_offsets[s], ahi = a.ambig_offsets[s + 1];
      for (u64 i = alo + lane; i < ahi && ahi >= alo; i += 32) {
        const u32 region = a.ambig[i].tag >> 1, ctx = a.ambig[i].ctx;
        if (region >= R || !record_in_scope(a, ctx, region)) continue;
        atomicAdd(a.iter_tab + ((u64)(ctx - a.ctx_lo) * R + region) * kCell + (a.ambig[i].kind == ARGUS_AMBIG_UNMATCHED_END ? 6 : 5), 1ull);
      }
    }
  }
  for (u32 i = threadIdx.x; i < (2 * kItWords * iter_cells(R) + 3) / 4; i += kIterThreads) reinterpret_cast<uint4*>(tab0)[i] = make_uint4(0, 0, 0, 0);
  __syncthreads();  // (the last vector may reach into what follows)
  for (u32 r = threadIdx.x; r < R; r += kIterThreads) meta[r] = r * (kItWords * 4);
  if (threadIdx.x < kDigestHot) hot_region[threadIdx.x] = kNone;
  if (threadIdx.x == 0) { need = kNone; num_often = 0; }
  __syncthreads();
  u64 at = lo < hi ? lo + mine * 32 : ~0ull;
  const u64 end = lo < hi ? hi : 0ull;
  u32 cur = 0;         // the two iterations at hand: cur (in table `odd`) and cur + 1
  u32 odd = 0, want = kNone;
  bool fresh = true;   // the round at `at` has not been taken up
  uint4 q0 = make_uint4(0, 0, 0, 0), q1 = q0, n0 = q0, n1 = q0;  // the record at hand and the one after it, asked for a round ahead
  u32 flags = 0, nflags = 0;
  auto ask = [&](u64 i) {
    if (i >= end) return;
    const uint4* p = reinterpret_cast<const uint4*>(a.intervals + i);
    n0 = __ldg(p); n1 = __ldg(p + 1);
    nflags = __ldg(reinterpret_cast<const u32*>(p + 2) + 3) >> 16;
  };
  if (at < end) ask(at + lane);
  // the regions that the first round sees most get copies of their cells, lanes apart: 32 adds to one address take turns
  if (at < end && at + lane < end && n1.z < R && record_in_scope(a, n1.w, n1.z)) atomicAdd(tab0 + n1.z * kItWords + kDgBins, 1u);
  __syncthreads();
  for (u32 r = threadIdx.x; r < R; r += kIterThreads) {
    const u32 cnt = tab0[r * kItWords + kDgBins];
    tab0[r * kItWords + kDgBins] = 0;
    if (cnt >= kIterThreads / 64) often[atomicAdd(&num_often, 1u)] = (cnt << 16) | r;  // at most 64 of them
  }
  __syncthreads();
  if (threadIdx.x < num_often) {
    const u32 key = often[threadIdx.x], r = key & 0xffffu;
    u32 rank = 0;
    for (u32 k = 0; k < num_often; ++k) rank += often[k] > key;
    if (rank < kDigestHot) { hot_region[rank] = r; meta[r] = ((R + rank * kIterCopies) * (kItWords * 4)) | kDgHot; }
  }
  __syncthreads();
  const u32 own_copy = lane % kIterCopies * (kItWords * 4);
  for (;;) {
    // take what belongs to the two iterations
    while (at < end) {
      if (fresh) {
        const u64 i = at + lane;
        q0 = n0; q1 = n1; flags = nflags;
        want = i < end && q1.z < R && record_in_scope(a, q1.w, q1.z) ? q1.w - a.ctx_lo : kNone;
        ask(i + (u64)m * 32);
        fresh = false;
      }
      if (want != kNone && want <= cur + 1) {
        const u64 incl = (u64)q0.z | ((u64)q0.w << 32), excl = (u64)q1.x | ((u64)q1.y << 32);
        u64* const row = a.iter_tab + (u64)want * cells;
        if (want < cur || (q0.w | q1.y)) {
          agg_add_interval(row, q1.z, incl, excl, flags);
        } else {
          const u32 mt = meta[q1.z];
          iter_add((((want - cur) ^ odd) ? addr1 : addr0) + (mt & ~kDgHot) + (mt >> 31) * own_copy, (u32)incl, (u32)excl, flags);
        }
        want = kNone;
      }
      if (__any_sync(0xffffffffu, want != kNone)) break;
      at += (u64)m * 32;
      fresh = true;
    }
    const u32 least = __reduce_min_sync(0xffffffffu, at < end ? want : kNone);
    if (lane == 0 && least != kNone) atomicMin(&need, least);
    __syncthreads();
    const u32 next = need;
    __syncthreads();
    if (threadIdx.x == 0) need = kNone;
    u32* const older = odd ? tab1 : tab0;
    iter_flush(older, hot_region, a.iter_tab + (u64)cur * cells, R);
    if (next != cur + 2 && cur + 1 < a.num_iters) iter_flush(odd ? tab0 : tab1, hot_region, a.iter_tab + (u64)(cur + 1) * cells, R);
    if (next == kNone) return;
    if (next == cur + 2) { cur += 1; odd ^= 1; } else { cur = next; }
    __syncthreads();
  }
}

// The same for more regions than the compact cells are kept for: every interval straight into the table.
__global__ void __launch_bounds__(kAggThreads) k_agg_iter(AggArgs a) {
  argus_kernel_begin_long();
  const u32 R = a.num_regions;
  for (u32 s = blockIdx.x; s < a.num_streams; s += gridDim.x) {
    if (stream_in_scope(a, s) != 1) continue;  // a bad cta_sm entry is reported by k_agg_streams
    const u64 lo = a.interval_offsets[s], hi = a.interval_offsets[s + 1];
    for (u64 i = lo + threadIdx.x; i < hi && hi >= lo && hi <= a.interval_limit; i += blockDim.x) {
      const uint4* p = reinterpret_cast<const uint4*>(a.intervals + i);
      const uint4 q1 = __ldg(p + 1);
      const u32 region = q1.z, ctx = q1.w;
      if (region >= R || !record_in_scope(a, ctx, region)) continue;
      const uint4 q0 = __ldg(p), q2 = __ldg(p + 2);
      agg_add_interval(a.iter_tab + (u64)(ctx - a.ctx_lo) * R * kCell, region, (u64)q0.z | ((u64)q0.w << 32), (u64)q1.x | ((u64)q1.y << 32), q2.w >> 16);
    }
    if (a.ambig && a.ambig_offsets) {
      const u64 alo = a.ambig_offsets[s], ahi = a.ambig_offsets[s + 1];
      for (u64 i = alo + threadIdx.x; i < ahi && ahi >= alo; i += blockDim.x) {
        const u32 region = a.ambig[i].tag >> 1, ctx = a.ambig[i].ctx;
        if (region >= R || !record_in_scope(a, ctx, region)) continue;
        atomicAdd(a.iter_tab + ((u64)(ctx - a.ctx_lo) * R + region) * kCell + (a.ambig[i].kind == ARGUS_AMBIG_UNMATCHED_END ? 6 : 5), 1ull);
      }
    }
  }
}

struct AggLayout { size_t warp, ranges, total; };

AggLayout agg_layout(uint32_t num_streams, uint32_t num_regions) {
  AggLayout L;
  const size_t row = (size_t)num_regions * sizeof(argus_agg_t);
  L.warp = 0;
  L.ranges = argus_align_up((size_t)num_streams * row, 256);
  L.total = L.ranges + argus_align_up((size_t)num_streams * kMaxParts * sizeof(ulonglong2), 256);
  if (L.total < 2 * L.ranges) L.total = 2 * L.ranges;  // two tables of the warp scope's size have always fitted
  return L;
}

auto record_kernel(u32 threads) { return threads == 256 ? k_agg_streams_records<256> : threads == 192 ? k_agg_streams_records<192> : k_agg_streams_records<128>; }

// Blocks of the pass over the records that an SM holds: what registers and threads let fit and the kernel's static shared memory belong to the
// device and are looked up once, under a lock (two host threads may make their first call at the same time).
struct RecordFit { int sms, plain[3]; size_t sm_bytes, block_bytes[3]; };
constexpr u32 kRecThreads[3] = {256, 192, 128};
int record_fit(RecordFit* fit) {
  constexpr int kMaxDevices = 64;
  static RecordFit of[kMaxDevices];
  static std::mutex mu;
  int dev = 0;
  ARGUS_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return ARGUS_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lk(mu);
  if (!of[dev].sms) {
    RecordFit f;
    int sm = 0, reserved = 0;
    ARGUS_CUDA_TRY(cudaDeviceGetAttribute(&sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev));
    ARGUS_CUDA_TRY(cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev));
    ARGUS_CUDA_TRY(cudaDeviceGetAttribute(&f.sms, cudaDevAttrMultiProcessorCount, dev));
    for (int k = 0; k < 3; ++k) {
      cudaFuncAttributes attr;
      ARGUS_CUDA_TRY(cudaFuncGetAttributes(&attr, record_kernel(kRecThreads[k])));
      ARGUS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&f.plain[k], record_kernel(kRecThreads[k]), (int)kRecThreads[k], 0));
      f.block_bytes[k] = attr.sharedSizeBytes + (size_t)reserved;
    }
    f.sm_bytes = (size_t)sm;
    of[dev] = f;
  }
  *fit = of[dev];
  return ARGUS_OK;
}
u32 record_blocks(const RecordFit& fit, int k, u32 num_regions) {
  const size_t held = fit.sm_bytes / argus_align_up(record_table_bytes(num_regions, kRecThreads[k]) + fit.block_bytes[k], 128);
  return held < (size_t)fit.plain[k] ? (u32)held : (u32)fit.plain[k];
}

// Threads of a block of the pass over the records. A block takes a stream, and how much of the chip the last round of blocks leaves idle
// decides, weighed against smaller blocks' slower reads (1, 0.96 and 0.8). 20 M records, us with 256 / 192 / 128 threads and the share of
// the rounds that is filled: 832 streams of 74 regions 194 / 157 / 164 (0.56, 0.94, 0.80), 960 of 5 181 / 146 / 154 (0.54, 0.72, 0.59), 960 of 74 182 / 200
// / 161 (0.65, 0.54, 0.93), 1,572 of 5 149 / 200 / 159 (0.89, 0.59, 0.97), 2,368 of 146 194 / 202 / 233 (1, 1, 0.8), 736 of 146 199 / 220
// / 172 (0.62, 0.62, 0.99). 1 and 20 M records in 24 to 4,736 streams of 5 to 400 regions (400 shapes): on average 1.2 % above the best of
// the three; 256 threads throughout 3.4 %.
u32 record_threads(const RecordFit& fit, u32 num_regions, u32 blocks) {
  constexpr double weight[3] = {1.0, 0.96, 0.8};
  double most = 0;
  u32 threads = 0;
  for (int k = 0; k < 3; ++k) {
    const u32 slots = (u32)fit.sms * (record_blocks(fit, k, num_regions) ? record_blocks(fit, k, num_regions) : 1), rounds = (blocks + slots - 1) / slots;
    const double share = weight[k] * blocks / ((double)slots * (rounds ? rounds : 1));
    if (share > most || !threads) { most = share; threads = kRecThreads[k]; }
  }
  return threads;
}

}  // namespace

extern "C" int argus_testing_record_blocks(uint32_t num_regions, uint32_t threads, uint32_t* by_rule, uint32_t* by_device) {
  if (num_regions == 0 || num_regions > kAggCompactRegions) return ARGUS_ERR_INVALID_ARG;
  int k = 0;
  while (k < 3 && kRecThreads[k] != threads) ++k;
  if (k == 3) return ARGUS_ERR_INVALID_ARG;
  RecordFit fit;
  { const int rc = record_fit(&fit); if (rc != ARGUS_OK) return rc; }
  const size_t bytes = record_table_bytes(num_regions, threads);
  ARGUS_CUDA_TRY(argus_allow_smem(record_kernel(threads), bytes, record_table_bytes(kAggCompactRegions, threads)));
  int blocks = 0;
  ARGUS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, record_kernel(threads), (int)threads, bytes));
  *by_rule = record_blocks(fit, k, num_regions);
  *by_device = (uint32_t)blocks;
  return ARGUS_OK;
}

extern "C" size_t argus_aggregate_workspace_bytes(uint64_t /*num_intervals*/, uint32_t num_streams, uint32_t num_regions) {
  return agg_layout(num_streams, num_regions).total + 256;
}

int argus_internal_aggregate_scoped(const argus_interval_t* intervals, const uint64_t* interval_offsets,
                                    const argus_ambiguity_t* ambig, const uint64_t* ambig_offsets, uint32_t num_streams,
                                    uint32_t warps_per_cta, const uint32_t* cta_sm, uint32_t num_sms, uint32_t num_regions,
                                    const argus_scope_t* scope, argus_agg_t* warp_tab, argus_agg_t* cta_tab,
                                    argus_agg_t* sm_tab, argus_agg_t* kernel_tab, argus_agg_t* role_tab,
                                    argus_agg_t* iter_tab, argus_status_t* status, void* workspace,
                                    size_t workspace_bytes, void* cuda_stream, bool reset_status,
                                    const ArgusFuseArgs* ov_select, const uint64_t* digest, uint32_t digest_parts, uint32_t digest_slices,
                                    uint64_t interval_limit) {
  if (!interval_offsets || !status || !workspace) return ARGUS_ERR_INVALID_ARG;
  if (ov_select && !digest) return ARGUS_ERR_INVALID_ARG;
  if (warps_per_cta == 0 || num_streams % warps_per_cta != 0) return ARGUS_ERR_INVALID_ARG;
  if (num_regions == 0 || num_regions > ARGUS_MAX_REGIONS) return ARGUS_ERR_INVALID_ARG;
  if ((sm_tab || (scope && scope->sm_mask)) && ((!cta_sm && num_streams) || num_sms == 0)) return ARGUS_ERR_INVALID_ARG;
  if (scope && scope->ctx_hi < scope->ctx_lo) return ARGUS_ERR_INVALID_ARG;
  if (iter_tab && (!scope || scope->ctx_hi - scope->ctx_lo >= ARGUS_MAX_ITER_ROWS)) return ARGUS_ERR_INVALID_ARG;
  if (((uintptr_t)intervals & 15) || ((uintptr_t)workspace & 255) || ((uintptr_t)warp_tab & 7) || ((uintptr_t)cta_tab & 7) ||
      ((uintptr_t)sm_tab & 7) || ((uintptr_t)kernel_tab & 7) || ((uintptr_t)role_tab & 7) || ((uintptr_t)iter_tab & 7))
    return ARGUS_ERR_INVALID_ARG;
  const AggLayout L = agg_layout(num_streams, num_regions);
  if (workspace_bytes < L.total) return ARGUS_ERR_WORKSPACE;
  cudaStream_t stream = (cudaStream_t)cuda_stream;
  if (reset_status) { const int rc = argus_internal_clear(status, nullptr, 0, cuda_stream); if (rc != ARGUS_OK) return rc; }
  const u32 num_iters = iter_tab ? scope->ctx_hi - scope->ctx_lo + 1 : 0;
  if (num_streams == 0) {
    if (kernel_tab) ARGUS_LAUNCH(k_agg_init, 16, 256, 0, stream, (u64*)kernel_tab, (u64)num_regions * kCell);
    if (sm_tab) ARGUS_LAUNCH(k_agg_init, 296, 256, 0, stream, (u64*)sm_tab, (u64)num_sms * num_regions * kCell);
    if (role_tab) { ARGUS_LAUNCH(k_agg_init, 64, 256, 0, stream, (u64*)role_tab, (u64)warps_per_cta * num_regions * kCell); }
    if (iter_tab) { ARGUS_LAUNCH(k_agg_init, 64, 256, 0, stream, (u64*)iter_tab, (u64)num_iters * num_regions * kCell); }
    return ARGUS_OK;
  }
  AggArgs a;
  a.intervals = intervals; a.interval_offsets = (const u64*)interval_offsets; a.ambig = ambig; a.ambig_offsets = (const u64*)ambig_offsets;
  a.num_streams = num_streams; a.warps_per_cta = warps_per_cta; a.num_ctas = num_streams / warps_per_cta;
  a.num_sms = num_sms; a.num_regions = num_regions; a.cta_sm = cta_sm;
  a.warp_tab = warp_tab ? (u64*)warp_tab : (u64*)((char*)workspace + L.warp);
  a.sm_tab = (u64*)sm_tab; a.kernel_tab = (u64*)kernel_tab; a.status = status;
  a.scoped = scope != nullptr;
  a.ctx_lo = scope ? scope->ctx_lo : 0; a.ctx_hi = scope ? scope->ctx_hi : 0xffffffffu;
  a.warp_mask = scope ? scope->warp_mask : ~0ull;
  a.sm_mask = scope ? scope->sm_mask : nullptr; a.region_mask = scope ? scope->region_mask : nullptr;
  a.role_tab = (u64*)role_tab; a.iter_tab = (u64*)iter_tab; a.num_iters = num_iters;
  if (ov_select) { a.ov = *ov_select; } else { a.ov = ArgusFuseArgs(); }
  a.digest = !scope && !role_tab && !iter_tab && num_regions <= kAggCompactRegions ? (const u64*)digest : nullptr;
  a.parts = digest_parts; a.slices = digest_slices; a.interval_limit = interval_limit;
  const bool windows = iter_tab && num_regions <= kAggCompactRegions;
  a.ranges = windows ? (ulonglong2*)((char*)workspace + L.ranges) : nullptr;
  if (!a.digest) {  // few streams: several blocks share one (how many intervals there are is not known here)
    const u32 room = 888 / num_streams;
    a.parts = num_regions > kAggCompactRegions || room < 1 ? 1 : room < kMaxParts ? room : kMaxParts;
  }
  if (num_regions <= kAggCompactRegions && a.parts > 1)
    ARGUS_LAUNCH(k_agg_init, 592, 256, 0, stream, a.warp_tab, (u64)num_streams * num_regions * kCell);
  argus_prof_mark(ARGUS_PROF_AGGREGATE, stream, 0);
  if (num_regions <= kAggCompactRegions) {
    if (a.digest) {
      const u32 warps = a.slices / a.parts;
      const u32 copies = warps == 16 ? 16 : 8;
      const size_t dg = digest_table_bytes(num_regions, copies);
      const auto kernel = warps == 16 ? k_agg_streams_digest<512, 16, 3> : warps == 8 ? k_agg_streams_digest<256, 8, 6> : k_agg_streams_digest<128, 8, 12>;
      ARGUS_CUDA_TRY(argus_allow_smem(kernel, dg, digest_table_bytes(kAggCompactRegions, copies)));
      ARGUS_LAUNCH(kernel, num_streams * a.parts, warps * 32, dg, stream, a);
    } else {
      const size_t compact = (size_t)num_regions * sizeof(ArgusAggCell);
      static_assert(kAggCompactRegions * sizeof(ArgusAggCell) <= 48 * 1024, "no more shared memory than every kernel gets");
      if (scope) {
        ARGUS_LAUNCH(k_agg_streams_compact, num_streams * a.parts, kAggThreads, compact, stream, a);
      } else {
        RecordFit fit;
        { const int rc = record_fit(&fit); if (rc != ARGUS_OK) return rc; }
        const u32 threads = record_threads(fit, num_regions, num_streams * a.parts);
        const size_t bytes = record_table_bytes(num_regions, threads);
        const auto kernel = record_kernel(threads);
        ARGUS_CUDA_TRY(argus_allow_smem(kernel, bytes, record_table_bytes(kAggCompactRegions, threads)));
        ARGUS_LAUNCH(kernel, num_streams * a.parts, threads, bytes, stream, a);
      }
    }
  } else {
    ARGUS_LAUNCH(k_agg_streams, num_streams, kAggThreads, 0, stream, a);
  }
  argus_prof_mark(ARGUS_PROF_AGGREGATE, stream, 1);
  if (iter_tab && windows) {
    u32 per = kIterWarps;  // streams of a block: at least two blocks for every SM where the streams allow it
    while (per > 1 && num_streams / per < 296) per >>= 1;
    ARGUS_CUDA_TRY(argus_allow_smem(k_agg_iter_windows, iter_bytes(num_regions), iter_bytes(kAggCompactRegions)));
    ARGUS_LAUNCH(k_agg_iter_windows, (num_streams + per - 1) / per, kIterThreads, iter_bytes(num_regions), stream, a, per);
  } else if (iter_tab) {
    ARGUS_LAUNCH(k_agg_iter, num_streams < 1184u ? num_streams : 1184u, kAggThreads, 0, stream, a);
  }
  if (cta_tab || sm_tab || kernel_tab || role_tab) {
    // groups of CTAs where that leaves enough threads to fill the chip (148 x 2,048); larger ones save adds to the tables of roles
    const u64 words = (u64)num_regions * kCell, of = role_tab ? 4 : 2, groups = ((u64)a.num_ctas + of - 1) / of;
    const bool grouped = groups * words >= 148 * 1024;
    const u64 blocks = ((grouped ? groups : a.num_ctas) * words + 255) / 256;
    const auto kernel = grouped ? (role_tab ? k_agg_rollup<4, true> : k_agg_rollup<2, false>) : role_tab ? k_agg_rollup<1, true> : k_agg_rollup<1, false>;
    ARGUS_LAUNCH(kernel, (unsigned)(blocks < 4736 ? blocks : 4736), 256, 0, stream, a, (u64*)cta_tab);
  }
  return ARGUS_OK;
}

int argus_internal_aggregate(const argus_interval_t* intervals, const uint64_t* interval_offsets,
                             const argus_ambiguity_t* ambig, const uint64_t* ambig_offsets, uint32_t num_streams,
                             uint32_t warps_per_cta, const uint32_t* cta_sm, uint32_t num_sms, uint32_t num_regions,
                             argus_agg_t* warp_tab, argus_agg_t* cta_tab, argus_agg_t* sm_tab, argus_agg_t* kernel_tab,
                             argus_status_t* status, void* workspace, size_t workspace_bytes, void* cuda_stream,
                             bool reset_status, uint64_t interval_limit) {
  return argus_internal_aggregate_scoped(intervals, interval_offsets, ambig, ambig_offsets, num_streams, warps_per_cta, cta_sm,
                                         num_sms, num_regions, nullptr, warp_tab, cta_tab, sm_tab, kernel_tab, nullptr,
                                         nullptr, status, workspace, workspace_bytes, cuda_stream, reset_status, nullptr,
                                         nullptr, 1, 0, interval_limit);
}

bool argus_aggregate_can_read_digests(uint32_t num_regions) { return num_regions <= kAggCompactRegions; }
// Few streams: several blocks share one, six for every SM in all, as long as each has 8,192 intervals to look at.
// (96 streams of 259,328 intervals: 104 us; 352 us with a block each.)
uint32_t argus_aggregate_digest_parts(uint32_t num_streams, uint64_t num_events) {
  if (num_streams == 0) return 1;
  const uint64_t room = 888 / num_streams, work = num_events / 2 / num_streams / 8192, parts = room < work ? room : work;
  return (uint32_t)(parts < 1 ? 1 : parts);
}
// A warp for each slice. By the streams' average length: 128 threads below 1,024 intervals, 256 below 8,192, else 512. Measured
// with 4 / 8 / 16 warps (148 CTAs, us): 350 intervals a stream 20 / 22 / 31, 870: 27 / 39 / 43, 1,700: 41 / 41 / 60, 3,500:
// 66 / 61 / 69, 6,100: 120 / 99 / 115 (202 regions), 130,000: 2,065 / 1,175 / 1,002.
uint32_t argus_aggregate_digest_slices(uint32_t num_streams, uint64_t num_events) {
  const uint32_t parts = argus_aggregate_digest_parts(num_streams, num_events);
  const uint64_t length = num_streams ? num_events / 2 / num_streams : 0;
  return parts * (length < 1024 ? 4 : length < 8192 ? 8 : 16);
}

extern "C" int argus_aggregate(const argus_interval_t* intervals, const uint64_t* interval_offsets,
                               const argus_ambiguity_t* ambig, const uint64_t* ambig_offsets, uint32_t num_streams,
                               uint32_t warps_per_cta, const uint32_t* cta_sm, uint32_t num_sms, uint32_t num_regions,
                               argus_agg_t* warp_tab, argus_agg_t* cta_tab, argus_agg_t* sm_tab, argus_agg_t* kernel_tab,
                               argus_status_t* status, void* workspace, size_t workspace_bytes, void* cuda_stream) {
  return argus_internal_aggregate(intervals, interval_offsets, ambig, ambig_offsets, num_streams, warps_per_cta, cta_sm,
                                  num_sms, num_regions, warp_tab, cta_tab, sm_tab, kernel_tab, status, workspace,
                                  workspace_bytes, cuda_stream, true);
}

extern "C" int argus_aggregate_scoped(const argus_interval_t* intervals, const uint64_t* interval_offsets,
                                      const argus_ambiguity_t* ambig, const uint64_t* ambig_offsets, uint32_t num_streams,
                                      uint32_t warps_per_cta, const uint32_t* cta_sm, uint32_t num_sms, uint32_t num_regions,
                                      const argus_scope_t* scope, argus_agg_t* warp_tab, argus_agg_t* cta_tab,
                                      argus_agg_t* sm_tab, argus_agg_t* kernel_tab, argus_agg_t* role_tab,
                                      argus_agg_t* iter_tab, argus_status_t* status, void* workspace,
                                      size_t workspace_bytes, void* cuda_stream) {
  return argus_internal_aggregate_scoped(intervals, interval_offsets, ambig, ambig_offsets, num_streams, warps_per_cta, cta_sm,
                                         num_sms, num_regions, scope, warp_tab, cta_tab, sm_tab, kernel_tab, role_tab, iter_tab,
                                         status, workspace, workspace_bytes, cuda_stream, true, nullptr);
}
