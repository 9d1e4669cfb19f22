// argus_aggregate.cu — argus_aggregate: intervals (+ ambiguity records) -> per-(scope, region) tables.
//
//   k_agg_streams_digest : argus_synthesize's pass: one CTA per stream reads the 8-byte digests the pairing
//                   kernel wrote beside the interval records (not the records) and gathers the stream's row
//                   in 100-byte shared-memory cells, with per-lane copies of the most frequent regions' cells;
//   k_agg_streams_compact : the same over the 48-byte records, with an optional scope: that stream's row in
//                   a compact shared-memory form (112 B per region: sums, min, max, a 16-bin window, so
//                   several CTAs fit an SM), for up to kAggCompactRegions regions;
//   k_agg_streams : the same with a full 576 B-per-region copy in shared memory when that fits, else on
//                   the global row itself. Integer atomics only: the result does not depend on thread order.
//   k_agg_rollup  : CTA-scope and warp-role cells = reductions over the warps of each CTA and over the CTAs; SM-scope and
//                   kernel-scope cells by atomic add/min/max of CTA cells.
//   k_agg_iter_windows, k_agg_iter : per-iteration cells (key = ctx - ctx_lo) of the intervals of a scope.
// A scope (iteration window, warp mask, SM mask, region mask) filters what the kernels over intervals
// take in; without one everything is selected.
#include "argus_internal.cuh"

namespace {

constexpr int kAggThreads = 256;
constexpr u32 kCell = 72;  // u64 words per argus_agg_t
constexpr size_t kAggSmemLimit = 200 * 1024;
constexpr u32 kAggCompactRegions = 400;  // 112 B each: 44.8 KB of shared memory at most
constexpr u32 kIterThreads = 512, kIterWarps = kIterThreads / 32;  // k_agg_iter_windows
constexpr u32 kMaxParts = 16;            // blocks that share a stream in k_agg_streams_compact

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
  int use_smem;
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
  u32 parts;          // k_agg_streams_digest, k_agg_streams_compact: blocks that share a stream
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
  extern __shared__ __align__(16) u64 sh_tab[];
  const u32 R = a.num_regions;
  const u32 cells = R * kCell;
  for (u32 s = blockIdx.x; s < a.num_streams; s += gridDim.x) {
    u64* row = a.warp_tab + (size_t)s * cells;
    u64* tab = a.use_smem ? sh_tab : row;
    for (u32 i = threadIdx.x; i < cells; i += blockDim.x) tab[i] = (i % kCell == 2) ? ~0ull : 0ull;
    if (!a.use_smem) __threadfence();
    __syncthreads();
    const u64 lo = a.interval_offsets[s], hi = a.interval_offsets[s + 1];
    const int sel = stream_in_scope(a, s);
    if (sel == 2 && threadIdx.x == 0) argus_set_error(a.status, ARGUS_ERR_INVALID_ARG, s, a.cta_sm[s / a.warps_per_cta]);
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
        agg_add_interval(tab, region, incl, excl, q2.w >> 16);
      }
    }
    if (a.ambig && a.ambig_offsets && sel == 1) {
      const u64 alo = a.ambig_offsets[s], ahi = a.ambig_offsets[s + 1];
      for (u64 i = alo + threadIdx.x; i < ahi && ahi >= alo; i += blockDim.x) {
        const u32 region = a.ambig[i].tag >> 1;
        if (region >= R) { argus_set_error(a.status, ARGUS_ERR_BAD_REGION, s, i); continue; }
        if (!record_in_scope(a, a.ambig[i].ctx, region)) continue;
        atomicAdd(tab + (size_t)region * kCell + (a.ambig[i].kind == ARGUS_AMBIG_UNMATCHED_END ? 6 : 5), 1ull);
      }
    }
    __syncthreads();
    if (a.use_smem) {
      for (u32 i = threadIdx.x; i < cells; i += blockDim.x) row[i] = sh_tab[i];
      __syncthreads();
    }
  }
}

__global__ void __launch_bounds__(kAggThreads) k_agg_streams_compact(AggArgs a) {
  argus_kernel_begin_long();
  agg_empty_tables(a);
  extern __shared__ __align__(16) unsigned char sh_raw[];
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
  if (sel == 2 && threadIdx.x == 0) argus_set_error(a.status, ARGUS_ERR_INVALID_ARG, s, a.cta_sm[s / a.warps_per_cta]);
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
// One CTA per stream, no scope. The stream's row is gathered in shared memory in cells of kDgWords = 25 32-bit
// words (an odd size: the cells of 32 different regions start in 32 different banks). A few regions usually own
// most intervals of a stream, and 32 lanes adding to one address serialise; so after a probe of the stream's
// first intervals the kDigestHot most frequent regions get 32 copies of their cell, one per lane (consecutive
// cells: never a bank conflict), which are folded into the region's cell when the stream ends. The last word of
// a region's cell (meta) holds what a lane needs to know about its region: histogram window base, copy slot,
// whether the region appears in an overlap pair. A digest marked wide (a duration of 2^23 ticks or more) sends
// its lane to the record and to 64-bit atomics on the global row. Every warp walks a slice of the stream, so that overlap
// candidates stay in order; their entries replace digests that the warp has consumed: no list, no atomics. The table is
// addressed with 32-bit shared-memory addresses and the fields by constant offsets.
constexpr u32 kDigestHot = 4;
constexpr u32 kDgSumInclLo = 0, kDgSumInclHi = 1, kDgSumExclLo = 2, kDgSumExclHi = 3, kDgMin = 4, kDgMax = 5, kDgFlag = 6,
              kDgCountOut = 7, kDgBins = 8, kDgMeta = kDgBins + kAggWindow, kDgWords = kDgMeta + 1;
static_assert(kDgWords % 2 == 1, "an odd cell size keeps the cells of different regions in different banks");
constexpr u32 kDgNone = 0xffu;                 // meta: bits 0-7 window base, 8-15 copy slot (kDgNone = unset), bit 16 in a pair
constexpr u32 kDigestProbe = 512;              // intervals looked at before the hot regions are chosen
constexpr u32 kDigestMinStream = 2048;         // shorter streams are gathered without copies

__host__ __device__ constexpr size_t digest_table_words(u32 R) { return (size_t)kDgWords * (R + kDigestHot * 32); }

template <u32 F> __device__ __forceinline__ u32 dg_add(u32 cell, u32 v) {  // returns the old value
  u32 old;
  asm volatile("atom.shared.add.u32 %0, [%1+%3], %2;" : "=r"(old) : "r"(cell), "r"(v), "n"(F * 4) : "memory");
  return old;
}
template <u32 F> __device__ __forceinline__ void dg_inc(u32 cell, u32 v) {
  asm volatile("red.shared.add.u32 [%0+%2], %1;" :: "r"(cell), "r"(v), "n"(F * 4) : "memory");
}
template <u32 F> __device__ __forceinline__ void dg_min(u32 cell, u32 v) {
  asm volatile("red.shared.min.u32 [%0+%2], %1;" :: "r"(cell), "r"(v), "n"(F * 4) : "memory");
}
template <u32 F> __device__ __forceinline__ void dg_max(u32 cell, u32 v) {
  asm volatile("red.shared.max.u32 [%0+%2], %1;" :: "r"(cell), "r"(v), "n"(F * 4) : "memory");
}

// The histogram bin of an interval whose bin is not inside the region's window as the lane saw it: the window
// may not be chosen yet (then this lane tries to), or the bin really lies outside (then it is counted here).
// Returns the bin's place in the window, or kAggWindow and beyond when it has been dealt with.
__device__ __noinline__ u32 digest_bin_rare(u32* meta_word, u32 bin, u32 cell, u64* row_bins) {
  const u32 m = *reinterpret_cast<volatile u32*>(meta_word);
  u32 hb = m & 0xffu;
  if (hb == kDgNone) {
    const u32 want = bin > 6u ? bin - 6u : 0u;   // bin <= 22: the window never passes bin 63
    const u32 prev = atomicCAS(meta_word, m, (m & ~0xffu) | want);  // only the window base changes while intervals are added
    hb = (prev & 0xffu) == kDgNone ? want : (prev & 0xffu);
  }
  const u32 rel = bin - hb;
  if (rel < kAggWindow) return rel;
  dg_inc<kDgCountOut>(cell, 1u);
  atomicAdd(row_bins + bin, 1ull);
  return 0xffffffffu;
}

// (512 threads, three blocks per SM: the same 48 warps as six blocks of 256, but a stream's set-up, the choice of its hot
// regions and the write-back of its row are shared by twice the threads; measured 2.33 ms against 2.45 ms on trace 3)
constexpr int kDgThreads = 512;
constexpr u32 kDgSlices = kDgThreads / 32;     // slices of a stream, one per warp (also the slices of the overlap entries)
__global__ void __launch_bounds__(kDgThreads, 3) k_agg_streams_digest(AggArgs a) {
  argus_kernel_begin_long();
  agg_empty_tables(a);
  if (a.ov.num_pairs && blockIdx.x == 0 && threadIdx.x == 0) *a.ov.ctl = ArgusOvCtl{};
  extern __shared__ __align__(16) unsigned char sh_raw[];
  u32* const tab = reinterpret_cast<u32*>(sh_raw);
  const u32 R = a.num_regions;
  const u32 num_cells = R + kDigestHot * 32;
  u32* const pairbits = tab + (size_t)kDgWords * num_cells;
  __shared__ u32 hot_region[kDigestHot];
  const u32 tab_addr = (u32)__cvta_generic_to_shared(tab);
  const u32 cells = R * kCell;
  const u32 lane = threadIdx.x & 31;
  const u32 warp = threadIdx.x >> 5;
  const bool has_ov = a.ov.num_pairs != 0;
  for (u32 i = threadIdx.x; i < (R + 31) / 32; i += blockDim.x) pairbits[i] = 0;
  __syncthreads();
  if (has_ov) {
    for (u32 i = threadIdx.x; i < 2 * a.ov.num_pairs; i += blockDim.x) {
      const u32 r = a.ov.pairs[i];
      if (r < R) atomicOr(&pairbits[r >> 5], 1u << (r & 31));
    }
    __syncthreads();
  }
  {
    const u32 s = blockIdx.x / a.parts, part = blockIdx.x % a.parts, slices = a.parts * kDgSlices;
    u64* row = a.warp_tab + (size_t)s * cells;
    if (a.parts == 1)  // (else the rows have been initialised: several blocks add to one)
      for (u32 i = threadIdx.x; i < cells; i += blockDim.x) row[i] = (i % kCell == 2) ? ~0ull : 0ull;
    for (u32 i = threadIdx.x; i < kDgWords * num_cells; i += blockDim.x) {
      const u32 f = i % kDgWords, c = i / kDgWords;
      u32 v = f == kDgMin ? 0xffffffffu : 0u;
      if (f == kDgMeta && c < R) v = kDgNone | (kDgNone << 8) | (((pairbits[c >> 5] >> (c & 31)) & 1u) << 16);
      tab[i] = v;
    }
    if (threadIdx.x < kDigestHot) hot_region[threadIdx.x] = 0xffffffffu;
    __threadfence();
    __syncthreads();
    const u64 lo = a.interval_offsets[s], hi = a.interval_offsets[s + 1];
    if (has_ov && threadIdx.x == 0) {
      const u32 m = a.cta_sm[s / a.warps_per_cta];
      if (m >= a.num_sms) argus_set_error(a.status, ARGUS_ERR_INVALID_ARG, s, m);
    }
    u32 out_count = 0, out_first = 0;  // warp-uniform: entries of the warp's slice, where they start in the stream
    if (hi < lo || hi > a.interval_limit || ((hi - lo) >> 32)) {
      if (threadIdx.x == 0) argus_set_error(a.status, ARGUS_ERR_BAD_OFFSETS, s, 0);
    } else {
      const u32 n = (u32)(hi - lo);
      const u64* const dgs = a.digest + lo;
      const argus_interval_t* const ivs = a.intervals + lo;
      u32 i0, i1;
      argus_ov_slice(n, slices, part * kDgSlices + warp, &i0, &i1);
      out_first = i0;
      u64* const ents = a.ov.entries + lo + i0;
      u64* const starts = a.ov.starts + lo + i0;
      // two legs: the probe (the first intervals of every slice, each into its region's cell), then, hot regions chosen, the rest
      const bool probe = n / a.parts >= kDigestMinStream;
      const u32 probe_end = probe ? (i0 + 32 < i1 ? i0 + 32 : i1) : i1;
      for (int leg = 0; leg < 2; ++leg) {
        const u32 leg_lo = leg ? probe_end : i0, leg_hi = leg ? i1 : probe_end;
        if (leg && probe) {
          // warp 0 ranks the regions by their counts so far; kDigestHot rounds of a warp-wide maximum
          if (threadIdx.x < 32) {
            for (u32 h = 0; h < kDigestHot; ++h) {
              u32 best = 0;
              for (u32 r = lane; r < R; r += 32) {
                const u32* c = tab + r * kDgWords;
                if (((c[kDgMeta] >> 8) & 0xffu) != kDgNone) continue;
                u32 cnt = c[kDgCountOut];
#pragma unroll
                for (u32 j = 0; j < kAggWindow; ++j) cnt += c[kDgBins + j];
                const u32 key = ((cnt > 0xffffu ? 0xffffu : cnt) << 16) | r;
                best = key > best ? key : best;
              }
              const u32 top = __reduce_max_sync(0xffffffffu, best);
              if ((top >> 16) < kDigestProbe / 64) break;  // not worth a set of copies
              if (lane == 0) { atomicAnd(&tab[(top & 0xffffu) * kDgWords + kDgMeta], ~0xff00u | (h << 8)); hot_region[h] = top & 0xffffu; }
              __syncwarp();
            }
          }
          __syncthreads();
        }
        // every lane of a warp runs the same number of rounds, so that entries can be appended a warp at a time
        u32 b = leg_lo;
        bool late = false;  // the lane's candidate of the round before: its begin time may still be on its way
        u64 late_t0 = 0;
        u64* late_start = nullptr;
        // digests are asked for two rounds ahead (one round is shorter than a loaded DRAM access)
        u64 dg_next = b + lane < leg_hi ? dgs[b + lane] : 0ull;
        u64 dg_next2 = b + lane + 32 < leg_hi ? dgs[b + lane + 32] : 0ull;
        for (; b < leg_hi; b += 32) {
          const u32 i = b + lane;
          const u64 dg = dg_next;
          dg_next = dg_next2;
          dg_next2 = i + 64 < leg_hi ? dgs[i + 64] : 0ull;
          const u32 dlo = (u32)dg, dhi = (u32)(dg >> 32);
          const bool in = i < leg_hi;
          const u32 region = dlo & 0xffffu;
          const bool ok = in && region < R;
          const u32 rsafe = ok ? region : 0u;
          const u32 incl = (dlo >> 18) | ((dhi & 0x1ffu) << 14), excl = dhi >> 9;
          const u32 meta = tab[rsafe * kDgWords + kDgMeta];
          const u32 slot = (meta >> 8) & 0xffu;
          const u32 cell = tab_addr + (slot != kDgNone ? R + slot * 32 + lane : rsafe) * (kDgWords * 4);
          // the common case without a branch: a lane that does not take part (past the end, wide, bad region)
          // adds nothing; whatever is rare (a carry, a flag, a bin outside the window, ...) is settled in one place
          const bool take = ok && !(dlo & (1u << 17));
          const u32 vi = take ? incl : 0u, ve = take ? excl : 0u;
          const u32 old_i = dg_add<kDgSumInclLo>(cell, vi);
          const u32 old_e = dg_add<kDgSumExclLo>(cell, ve);
          dg_min<kDgMin>(cell, take ? incl : 0xffffffffu);
          dg_max<kDgMax>(cell, vi);
          const u32 bin = 31u - (u32)__clz((int)(incl | 1u));
          const u32 rel = bin - (meta & 0xffu);
          const bool in_win = take && rel < kAggWindow;
          dg_inc<kDgBins>(cell + (in_win ? rel : 0u) * 4, in_win ? 1u : 0u);
          u64 span = vi;
          const bool rare = in && ((dlo & (3u << 16)) || !ok || old_i + vi < old_i || old_e + ve < old_e || !in_win);
          if (rare) {
            if (!ok) {
              argus_set_error(a.status, ARGUS_ERR_BAD_REGION, s, lo + i);
            } else if (!take) {
              u64* const row_cell = row + (size_t)region * kCell;
              const uint4* p = reinterpret_cast<const uint4*>(ivs + i);
              const uint4 q0 = __ldg(p), q1 = __ldg(p + 1);
              span = (u64)q0.z | ((u64)q0.w << 32);
              atomicAdd(row_cell + 0, 1ull);
              atomicAdd(row_cell + 1, span);
              atomicMin(row_cell + 2, span);
              atomicMax(row_cell + 3, span);
              atomicAdd(row_cell + 4, (u64)q1.x | ((u64)q1.y << 32));
              if (dlo & (1u << 16)) atomicAdd(row_cell + 7, 1ull);
              atomicAdd(row_cell + 8 + log2_bin(span), 1ull);
            } else {
              if (old_i + vi < old_i) dg_inc<kDgSumInclHi>(cell, 1u);
              if (old_e + ve < old_e) dg_inc<kDgSumExclHi>(cell, 1u);
              if (dlo & (1u << 16)) dg_inc<kDgFlag>(cell, 1u);
              if (!in_win) {
                const u32 r2 = digest_bin_rare(tab + region * kDgWords + kDgMeta, bin, cell, row + (size_t)region * kCell + 8);
                if (r2 < kAggWindow) dg_inc<kDgBins>(cell + r2 * 4, 1u);
              }
            }
          }
          const bool cand = ok && ((meta >> 16) & 1u) && span;
          const u32 bal = __ballot_sync(0xffffffffu, cand);
          if (late) late_start[0] = late_t0;  // asked for a round ago
          late = cand;
          if (bal) {  // (the entries of a slice never reach the digests that are still to be read)
            const u32 at = out_count + __popc(bal & ((1u << lane) - 1u));
            if (cand) {
              ents[at] = argus_entry_pack(dg, i - i0);
              late_start = starts + at;
              late_t0 = __ldg(reinterpret_cast<const u64*>(ivs + i));
            }
            out_count += __popc(bal);
          }
        }
        if (late) late_start[0] = late_t0;
        __syncthreads();
      }
    }
    if (has_ov && lane == 0) {
      ArgusOvPiece e;
      e.pos = lo + out_first; e.count = out_count; e.next = kOvNone;
      a.ov.pieces[s * slices + part * kDgSlices + warp] = e;
    }
    if (a.ambig && a.ambig_offsets && part == 0) {
      const u64 alo = a.ambig_offsets[s], ahi = a.ambig_offsets[s + 1];
      for (u64 i = alo + threadIdx.x; i < ahi && ahi >= alo; i += blockDim.x) {
        const u32 region = a.ambig[i].tag >> 1;
        if (region >= R) { argus_set_error(a.status, ARGUS_ERR_BAD_REGION, s, i); continue; }
        atomicAdd(row + (size_t)region * kCell + (a.ambig[i].kind == ARGUS_AMBIG_UNMATCHED_END ? 6 : 5), 1ull);
      }
    }
    __syncthreads();
    // fold the lanes' copies into their region's cell: one thread per (hot region, field)
    if (threadIdx.x < kDigestHot * kDgMeta) {
      const u32 h = threadIdx.x / kDgMeta, f = threadIdx.x % kDgMeta;
      const u32 r = hot_region[h];
      if (r != 0xffffffffu && f != kDgSumInclHi && f != kDgSumExclHi) {
        const u32* src = tab + (R + h * 32) * kDgWords + f;
        u32* dst = tab + r * kDgWords + f;
        if (f == kDgSumInclLo || f == kDgSumExclLo) {
          u64 sum = (u64)dst[0] | ((u64)dst[1] << 32);
          for (u32 l = 0; l < 32; ++l) sum += (u64)src[l * kDgWords] | ((u64)src[l * kDgWords + 1] << 32);
          dst[0] = (u32)sum;
          dst[1] = (u32)(sum >> 32);
        } else {
          u32 acc = dst[0];
          for (u32 l = 0; l < 32; ++l) {
            const u32 v = src[l * kDgWords];
            acc = f == kDgMin ? (v < acc ? v : acc) : f == kDgMax ? (v > acc ? v : acc) : acc + v;
          }
          dst[0] = acc;
        }
      }
    }
    __syncthreads();
    // the regions' cells into the global row, which already holds the wide intervals, the bins outside the
    // windows and the ambiguity counters: everything is combined, nothing overwritten
    constexpr u32 kItems = 6 + kAggWindow;
    for (u32 i = threadIdx.x; i < R * kItems; i += blockDim.x) {
      const u32 r = i % R, f = i / R;
      const u32* c = tab + r * kDgWords;
      u64* cell = row + (size_t)r * kCell;
      switch (f) {
        case 0: {
          u64 cnt = c[kDgCountOut];
#pragma unroll
          for (u32 j = 0; j < kAggWindow; ++j) cnt += c[kDgBins + j];
          if (cnt) atomicAdd(cell + 0, cnt);
          break;
        }
        case 1: { const u64 v = (u64)c[kDgSumInclLo] | ((u64)c[kDgSumInclHi] << 32); if (v) atomicAdd(cell + 1, v); break; }
        case 2: { const u32 v = c[kDgMin]; if (v != 0xffffffffu) atomicMin(cell + 2, (u64)v); break; }
        case 3: { const u32 v = c[kDgMax]; if (v) atomicMax(cell + 3, (u64)v); break; }
        case 4: { const u64 v = (u64)c[kDgSumExclLo] | ((u64)c[kDgSumExclHi] << 32); if (v) atomicAdd(cell + 4, v); break; }
        case 5: { const u32 v = c[kDgFlag]; if (v) atomicAdd(cell + 7, (u64)v); break; }
        default: {
          const u32 j = f - 6;
          const u32 v = c[kDgBins + j];
          if (v) atomicAdd(cell + 8 + (c[kDgMeta] & 0xffu) + j, (u64)v);
        }
      }
    }
    __syncthreads();
  }
}

__device__ __forceinline__ u64 combine(u32 field, u64 x, u64 y) {
  return field == 2 ? (x < y ? x : y) : field == 3 ? (x > y ? x : y) : x + y;
}

__global__ void __launch_bounds__(256) k_agg_init(u64* tab, u64 n) {
  argus_kernel_begin();
  for (u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (u64)gridDim.x * blockDim.x)
    tab[i] = (i % kCell == 2) ? ~0ull : 0ull;
}

// One word of the cells of kGroup CTAs: CTA cells = reduction over the warps of each (written if asked for), warp-role cells over
// the CTAs; CTA cells go to the SM-scope cells, their reduction over the group to the kernel-scope cells (atomic add / min / max
// on integers; empty words add nothing). Bound by the one read of the warp-scope table, of which a thread has kGroup words in
// flight: 64 us for 275 MB; 77 us a CTA a thread, and 288 us more for the roles by themselves.
__device__ __forceinline__ void cell_add(u64* d, u32 field, u64 v) {
  if (field == 2 ? v == ~0ull : v == 0ull) return;  // identity element: nothing to add
  if (field == 2) atomicMin(d, v); else if (field == 3) atomicMax(d, v); else atomicAdd(d, v);
}
template <u32 kGroup>
__global__ void __launch_bounds__(256) k_agg_rollup(AggArgs a, u64* cta_out) {
  argus_kernel_begin_long();
  const u64 per_cta = (u64)a.num_regions * kCell, n = (u64)((a.num_ctas + kGroup - 1) / kGroup) * per_cta;
  for (u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (u64)gridDim.x * blockDim.x) {
    const u32 c0 = (u32)(i / per_cta) * kGroup, have = a.num_ctas - c0 < kGroup ? a.num_ctas - c0 : kGroup;
    const u64 rem = i % per_cta;
    const u32 field = (u32)(rem % kCell);
    const u64 none = field == 2 ? ~0ull : 0ull;
    const u64* src = a.warp_tab + (u64)c0 * a.warps_per_cta * per_cta + rem;
    u64 v[kGroup];
#pragma unroll
    for (u32 q = 0; q < kGroup; ++q) v[q] = none;
#pragma unroll kGroup == 1 ? 8 : 2
    for (u32 w = 0; w < a.warps_per_cta; ++w) {
      u64 x[kGroup];
#pragma unroll
      for (u32 q = 0; q < kGroup; ++q) x[q] = q < have ? src[((u64)q * a.warps_per_cta + w) * per_cta] : none;
      u64 all = none;
#pragma unroll
      for (u32 q = 0; q < kGroup; ++q) { v[q] = combine(field, v[q], x[q]); all = combine(field, all, x[q]); }
      if (a.role_tab) cell_add(a.role_tab + w * per_cta + rem, field, all);
    }
    u64 all = none;
#pragma unroll
    for (u32 q = 0; q < kGroup; ++q) {
      if (q >= have) break;
      if (cta_out) cta_out[(u64)(c0 + q) * per_cta + rem] = v[q];
      if (a.sm_tab && v[q] != none) {
        const u32 m = a.cta_sm[c0 + q];
        if (m >= a.num_sms) { argus_set_error(a.status, ARGUS_ERR_INVALID_ARG, c0 + q, m); continue; }
        cell_add(a.sm_tab + (u64)m * per_cta + rem, field, v[q]);
      }
      all = combine(field, all, v[q]);
    }
    if (a.kernel_tab) cell_add(a.kernel_tab + rem, field, all);
  }
}

// iter_tab[ctx - ctx_lo][r] with the compact cells. A block walks a few streams side by side (kIterWarps warps, shared out
// among them) and holds the cells of two neighbouring iterations in shared memory; a warp that comes to a later one waits until
// all have, then the older cells are added to the table. Iterations come in order in a stream, so each is gathered once for
// all of the block's streams: 551 us for 38 M intervals in 16 iterations of 202 regions, where atomics on the table for every
// interval took 2.0 ms. An interval of an earlier iteration than the two is added to the table directly. Only the part of a
// stream that the pass before found to be in the window is read.
__global__ void __launch_bounds__(kIterThreads) k_agg_iter_windows(AggArgs a, u32 streams_per_block) {
  argus_kernel_begin_long();
  extern __shared__ __align__(16) unsigned char sh_raw[];
  __shared__ u32 need;
  const u32 R = a.num_regions, cells = R * kCell, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  ArgusAggCell* const tab0 = reinterpret_cast<ArgusAggCell*>(sh_raw);
  ArgusAggCell* const tab1 = tab0 + R;
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
  argus_fuse_init(tab0, 2 * R, threadIdx.x, kIterThreads);
  if (threadIdx.x == 0) need = kNone;
  __syncthreads();
  u64 at = lo < hi ? lo + mine * 32 : ~0ull;
  const u64 end = lo < hi ? hi : 0ull;
  u32 cur = 0;         // the two iterations at hand: cur (in table `odd`) and cur + 1
  u32 odd = 0, want = kNone;
  bool fresh = true;   // the round at `at` has not been loaded
  uint4 q0 = make_uint4(0, 0, 0, 0), q1 = q0;
  u32 flags = 0;
  for (;;) {
    // take what belongs to the two iterations
    while (at < end) {
      if (fresh) {
        const u64 i = at + lane;
        want = kNone;
        if (i < end) {
          const uint4* p = reinterpret_cast<const uint4*>(a.intervals + i);
          q0 = __ldg(p); q1 = __ldg(p + 1);
          flags = __ldg(reinterpret_cast<const u32*>(p + 2) + 3) >> 16;
          if (q1.z < R && record_in_scope(a, q1.w, q1.z)) want = q1.w - a.ctx_lo;
        }
        fresh = false;
      }
      if (want != kNone && want <= cur + 1) {
        const u64 incl = (u64)q0.z | ((u64)q0.w << 32), excl = (u64)q1.x | ((u64)q1.y << 32);
        u64* const row = a.iter_tab + (u64)want * cells;
        if (want < cur) {
          agg_add_interval(row, q1.z, incl, excl, flags);
        } else {
          ArgusFuseCtx fx;
          fx.tab = ((want - cur) ^ odd) ? tab1 : tab0;
          fx.row = row;
          argus_fuse_aggregate(fx, q1.z, incl, excl, flags);
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
    ArgusAggCell* const older = odd ? tab1 : tab0;
    argus_fuse_flush(older, a.iter_tab + (u64)cur * cells, R, threadIdx.x, kIterThreads);
    if (next != cur + 2 && cur + 1 < a.num_iters) argus_fuse_flush(odd ? tab0 : tab1, a.iter_tab + (u64)(cur + 1) * cells, R, threadIdx.x, kIterThreads);
    if (next == kNone) return;
    __syncthreads();
    argus_fuse_init(older, R, threadIdx.x, kIterThreads);
    if (next != cur + 2) argus_fuse_init(odd ? tab0 : tab1, R, threadIdx.x, kIterThreads);
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

}  // namespace

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
                                    const ArgusFuseArgs* ov_select, const uint64_t* digest, uint32_t digest_parts,
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
  a.parts = digest_parts; a.interval_limit = interval_limit;
  const size_t smem = (size_t)num_regions * sizeof(argus_agg_t);
  a.use_smem = smem <= kAggSmemLimit;
  const size_t need = a.use_smem ? smem : 0;
  if (need > 48 * 1024)
    ARGUS_CUDA_TRY(cudaFuncSetAttribute(k_agg_streams, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)need));
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
    const size_t compact = (size_t)num_regions * sizeof(ArgusAggCell);
    if (compact > 48 * 1024)
      ARGUS_CUDA_TRY(cudaFuncSetAttribute(k_agg_streams_compact, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)compact));
    if (a.digest) {
      const size_t dg = digest_table_words(num_regions) * 4 + ((num_regions + 31) / 32) * 4;
      if (dg > 48 * 1024)
        ARGUS_CUDA_TRY(cudaFuncSetAttribute(k_agg_streams_digest, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dg));
      ARGUS_LAUNCH(k_agg_streams_digest, num_streams * a.parts, kDgThreads, dg, stream, a);
    } else {
      ARGUS_LAUNCH(k_agg_streams_compact, num_streams * a.parts, kAggThreads, compact, stream, a);
    }
  } else {
    ARGUS_LAUNCH(k_agg_streams, num_streams, kAggThreads, need, stream, a);
  }
  argus_prof_mark(ARGUS_PROF_AGGREGATE, stream, 1);
  if (iter_tab && windows) {
    u32 per = kIterWarps;  // streams of a block: at least two blocks for every SM where the streams allow it
    while (per > 1 && num_streams / per < 296) per >>= 1;
    const size_t two = 2 * (size_t)num_regions * sizeof(ArgusAggCell);
    if (two > 48 * 1024)
      ARGUS_CUDA_TRY(cudaFuncSetAttribute(k_agg_iter_windows, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)two));
    ARGUS_LAUNCH(k_agg_iter_windows, (num_streams + per - 1) / per, kIterThreads, two, stream, a, per);
  } else if (iter_tab) {
    ARGUS_LAUNCH(k_agg_iter, num_streams < 1184u ? num_streams : 1184u, kAggThreads, 0, stream, a);
  }
  if (cta_tab || sm_tab || kernel_tab || role_tab) {
    // groups of CTAs where that leaves enough threads to fill the chip (148 x 2,048)
    const u64 words = (u64)num_regions * kCell, groups = ((u64)a.num_ctas + 7) / 8;
    if (groups * words >= 148 * 1024)
      ARGUS_LAUNCH(k_agg_rollup<8>, (unsigned)((groups * words + 255) / 256 < 4736 ? (groups * words + 255) / 256 : 4736), 256, 0, stream, a, (u64*)cta_tab);
    else
      ARGUS_LAUNCH(k_agg_rollup<1>, (unsigned)((a.num_ctas * words + 255) / 256 < 4736 ? (a.num_ctas * words + 255) / 256 : 4736), 256, 0, stream, a, (u64*)cta_tab);
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
                                         nullptr, 1, interval_limit);
}

bool argus_aggregate_can_read_digests(uint32_t num_regions) { return num_regions <= kAggCompactRegions; }
// Few streams: several blocks share one, six for every SM in all, as long as each has 8,192 intervals to look at.
// (96 streams of 259,328 intervals: 142 us; 352 us with a block each.)
uint32_t argus_aggregate_digest_parts(uint32_t num_streams, uint64_t num_events) {
  if (num_streams == 0) return 1;
  const uint64_t room = 888 / num_streams, work = num_events / 2 / num_streams / 8192, parts = room < work ? room : work;
  return (uint32_t)(parts < 1 ? 1 : parts);
}
uint32_t argus_aggregate_digest_slices(uint32_t parts) { return parts * kDgSlices; }

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
