// argus_fuse.cuh — what the pairing kernels and the aggregation passes share: the compact shared-memory
// form of a stream's row of the warp-scope table, the 8-byte digest of an interval, and the form in which
// intervals are handed to the overlap kernel.
//
// Compact row: per region the sums, min, max, counts and a 16-bin window of the 64-bin log2 histogram
// (bins outside the window go straight to the global row); the CTA that aggregates a stream keeps the row
// in shared memory and writes it to the global row when the stream ends. All updates are integer atomics,
// so thread order is irrelevant.
#ifndef ARGUS_FUSE_CUH_
#define ARGUS_FUSE_CUH_

#include "argus_common.cuh"

constexpr u32 kAggWindow = 16;          // histogram bins kept in shared memory per region
constexpr u32 kAggUnset = 0xffffffffu;  // window base not chosen yet
constexpr u32 kAggCellWords = 72;       // u64 words of one argus_agg_t

struct ArgusAggCell {  // 112 bytes
  u64 sum_incl, sum_excl, min_incl, max_incl;
  u32 count_out, nflag, hbase, pad;  // count_out: intervals whose bin fell outside the window
  u32 h[kAggWindow];                 // the interval count of the region is count_out + the sum of these
};

// Overlap selection. The intervals whose region appears in a pair are handed to the overlap kernel as 8-byte entries, slice
// by slice of a stream and in order. A slice is a run of consecutive intervals that one warp looks at; its entries lie in
// one piece or in a chain of pieces. Entries from digests: the digest with the interval's place in its slice instead of the
// exclusive duration, or, when it is wide or the place does not fit, region, wide bit and place; the piece lies where the
// slice's digests did, so position + place is the record's index. Entries from records: index within the stream (low word),
// region (high word).
constexpr u32 kOvNone = 0xffffffffu;
struct ArgusOvPiece {  // 16 bytes; piece [stream * slices + slice] is the slice's first
  u64 pos;             // first entry
  u32 count, next;     // entries; the slice's next piece or kOvNone
};
struct ArgusOvCtl {    // zeroed before the selection
  u64 num_entries;     // entries appended (selection that appends; may exceed the room)
  u64 num_spans;       // room asked for by the blocks of the overlap kernel (may exceed the capacity)
  u32 num_pieces;      // later pieces taken from the pool
  u32 asked;           // blocks that have asked for room
};
// Intervals [*i0, *i1) of a stream of n are slice `slice` of `slices`: whole warps' worth, equal but for the last ones.
__device__ __forceinline__ void argus_ov_slice(u32 n, u32 slices, u32 slice, u32* i0, u32* i1) {
  const u64 per = (((u64)n + slices - 1) / slices + 31) & ~31ull;
  const u64 a = per * slice, b = a + per;
  *i0 = a < n ? (u32)a : n;
  *i1 = b < n ? (u32)b : n;
}

struct ArgusFuseArgs {    // selection inside the pass over the digests
  const u32* pairs;       // [K][2]
  u32 num_pairs;          // 0 = no selection
  u64* entries;           // the digest array: a warp writes the entries of its slice over the digests it has consumed
  u64* starts;            // begin times of the entries' intervals, same positions
  ArgusOvPiece* pieces;   // [S][slices]
  ArgusOvCtl* ctl;        // cleared by the pass
};

struct ArgusFuseCtx {     // per CTA, for the stream it is aggregating
  ArgusAggCell* tab;      // shared memory [R]
  u64* row;               // global row of this stream in the warp-scope table
};

// Digest of an interval (8 bytes): all that aggregation needs of it. argus_synthesize lets the pairing kernels
// write one per interval record, at the same position, so that the aggregation pass reads 8 bytes per interval
// instead of 48. Bits 0-15 region, 16 any flag set, 17 wide (a duration does not fit: take both from the
// record; the duration bits then mean nothing), 18-40 inclusive, 41-63 exclusive duration.
constexpr u32 kDigestBits = 23;
constexpr u32 kDigestFlag = 1u << 16, kDigestWide = 1u << 17;
constexpr u32 kEntryIndexShift = 18 + kDigestBits;        // an entry's place in its slice
__device__ __forceinline__ u64 argus_digest_pack(u32 region, u64 incl, u64 excl, u32 flags) {
  const u32 il = (u32)incl, el = (u32)excl;
  const bool wide = (((il | el) >> kDigestBits) | (u32)(incl >> 32) | (u32)(excl >> 32)) != 0;
  const u32 lo = region | (flags ? 1u << 16 : 0u) | (wide ? 1u << 17 : 0u) | (il << 18);
  const u32 hi = ((il >> 14) & 0x1ffu) | (el << 9);
  return (u64)lo | ((u64)hi << 32);
}

// The same for durations that fit 32 bits, excl <= incl.
__device__ __forceinline__ u64 argus_digest_pack32(u32 region, u32 incl, u32 excl, u32 flags) {
  const u32 lo = region | (flags ? 1u << 16 : 0u) | (incl >> kDigestBits ? 1u << 17 : 0u) | (incl << 18);
  return (u64)lo | ((u64)(((incl >> 14) & 0x1ffu) | (excl << 9)) << 32);
}

__device__ __forceinline__ u64 argus_entry_pack(u64 digest, u32 place) {
  if (((u32)digest & kDigestWide) || place >> (64 - kEntryIndexShift)) return ((u64)place << 18) | kDigestWide | ((u32)digest & 0xffffu);
  return (digest & ((1ull << kEntryIndexShift) - 1ull)) | ((u64)place << kEntryIndexShift);
}

__device__ __forceinline__ u32 argus_log2_bin(u64 d) { return d ? 63u - (u32)__clzll((long long)d) : 0u; }

// 64-bit add as native 32-bit atomics; each carry is propagated exactly once
__device__ __forceinline__ void argus_atomic_add64_split(u64* p64, u64 v) {
  u32* p = reinterpret_cast<u32*>(p64);
  const u32 lo = (u32)v, hi = (u32)(v >> 32);
  if (lo) {
    const u32 old = atomicAdd(p, lo);
    if (old + lo < old) atomicAdd(p + 1, 1u);
  }
  if (hi) atomicAdd(p + 1, hi);
}

__device__ __forceinline__ void argus_fuse_init(ArgusAggCell* tab, u32 num_regions, u32 tid, u32 nthreads) {
  u32* w = reinterpret_cast<u32*>(tab);
  constexpr u32 kWords = sizeof(ArgusAggCell) / 4;
  for (u32 i = tid; i < num_regions * kWords; i += nthreads) {
    const u32 f = i % kWords;
    w[i] = (f == 4 || f == 5 || f == 10) ? 0xffffffffu : 0u;  // min_incl = all ones, hbase = unset
  }
}

// sums of one cell
__device__ __forceinline__ void argus_fuse_agg_sums(ArgusAggCell& c, u64 sum_incl, u64 sum_excl) {
  argus_atomic_add64_split(&c.sum_incl, sum_incl);
  argus_atomic_add64_split(&c.sum_excl, sum_excl);
}

// min, max, flag count and histogram bin of one interval; the bin also counts the interval
__device__ __forceinline__ void argus_fuse_agg_rest(ArgusAggCell& c, u64* row, u32 region, u64 incl, u32 flags) {
  if (incl < *reinterpret_cast<volatile u64*>(&c.min_incl)) atomicMin(&c.min_incl, incl);
  if (incl > *reinterpret_cast<volatile u64*>(&c.max_incl)) atomicMax(&c.max_incl, incl);
  if (flags) atomicAdd(&c.nflag, 1u);
  const u32 bin = argus_log2_bin(incl);
  u32 hb = *reinterpret_cast<volatile u32*>(&c.hbase);
  if (hb == kAggUnset) {
    const u32 want = bin > 6u ? (bin - 6u > 64u - kAggWindow ? 64u - kAggWindow : bin - 6u) : 0u;
    const u32 old = atomicCAS(&c.hbase, kAggUnset, want);
    hb = old == kAggUnset ? want : old;
  }
  const u32 rel = bin - hb;
  if (rel < kAggWindow) {
    atomicAdd(&c.h[rel], 1u);
  } else {
    atomicAdd(&c.count_out, 1u);
    atomicAdd(row + (size_t)region * kAggCellWords + 8 + bin, 1ull);
  }
}

__device__ __forceinline__ void argus_fuse_aggregate(const ArgusFuseCtx& fx, u32 region, u64 incl, u64 excl, u32 flags) {
  ArgusAggCell& c = fx.tab[region];
  argus_fuse_agg_sums(c, incl, excl);
  argus_fuse_agg_rest(c, fx.row, region, incl, flags);
}

// Adds the cells to a global row, which may hold something already (bins outside the windows, ambiguity counters, what other
// blocks have added).
__device__ __forceinline__ void argus_fuse_flush(const ArgusAggCell* tab, u64* row, u32 num_regions, u32 tid, u32 nthreads) {
  constexpr u32 kItems = 6 + kAggWindow;
  for (u32 i = tid; i < num_regions * kItems; i += nthreads) {
    const u32 r = i / kItems, f = i % kItems;
    const ArgusAggCell& c = tab[r];
    if (c.hbase == kAggUnset) continue;  // the first interval of a region chooses its window
    u64* cell = row + (size_t)r * kAggCellWords;
    switch (f) {
      case 0: {
        u64 n = c.count_out;
#pragma unroll
        for (u32 j = 0; j < kAggWindow; ++j) n += c.h[j];
        atomicAdd(cell + 0, n);
        break;
      }
      case 1: atomicAdd(cell + 1, c.sum_incl); break;
      case 2: atomicMin(cell + 2, c.min_incl); break;
      case 3: atomicMax(cell + 3, c.max_incl); break;
      case 4: atomicAdd(cell + 4, c.sum_excl); break;
      case 5: if (c.nflag) atomicAdd(cell + 7, (u64)c.nflag); break;
      default: {
        const u32 j = f - 6;
        if (c.h[j]) atomicAdd(cell + 8 + c.hbase + j, (u64)c.h[j]);
      }
    }
  }
}

#endif  // ARGUS_FUSE_CUH_
