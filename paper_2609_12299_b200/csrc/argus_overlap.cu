// argus_overlap.cu — argus_overlap: per-SM overlap time of producer/consumer region pairs.
//
//   k_ov_select : one pass over the intervals: those whose region appears in a pair are appended, slice by slice of a
//                 stream and in order, as entries {index within the stream, region} (argus_synthesize gets the same
//                 entries from the aggregation pass, which writes them over the digests that it has consumed)
//   k_ov_pair   : one block per (pair k, SM m): gathers the spans of the producer and of the consumer region from the
//                 entries of the SM's streams, in stream and slice order; sorts a role by start time if it is not in order
//                 already and cuts it into the disjoint pieces of its union if its spans overlap one another; then walks
//                 the merged sequence of both roles, where every piece meets the last piece of the other role:
//                 |U_P ∩ U_C| in one pass, |U_P| and |U_C| being sums of lengths.
//
// A region that is not nested in itself leaves its spans of one stream disjoint and in time order. The entries are kept in
// order, so a role that sits in one warp of a CTA needs no sort, and spans of several warps are runs that need few merges.
#include "argus_internal.cuh"

#include <atomic>

namespace {

constexpr int kSelThreads = 256;
constexpr u32 kSelWarps = kSelThreads / 32;
constexpr u32 kSelStage = 128;    // entries a warp collects before it appends them
constexpr u32 kSelFilter = 4096;  // bits of the region filter
constexpr unsigned kSelGrid = 148 * 8;

struct OvSelectArgs {
  const argus_interval_t* intervals;
  const u64* interval_offsets;
  u64 max_intervals;  // records the interval array holds
  u32 num_streams, warps_per_cta, num_sms, num_pairs;
  const u32* cta_sm;
  const u32* pairs;
  argus_status_t* status;
  u64* entries;
  u64 entry_capacity;
  ArgusOvPiece* pieces;  // [num_streams * slices] first pieces, then the pool of later ones
  u32 slices;            // per stream, a multiple of kSelWarps
  u32 piece_capacity;
  int direct;            // the entry array has a place for every interval: a slice's entries start at its first interval's
  ArgusOvCtl* ctl;
  // scope selection (argus_overlap_scoped): iteration window, warp mask, SM mask, region mask
  int scoped;
  u32 ctx_lo, ctx_hi;
  u64 warp_mask;
  const u32* sm_mask;
  const u32* region_mask;
};

__device__ __forceinline__ bool ov_mask_bit(const u32* mask, u32 i) { return !mask || ((mask[i >> 5] >> (i & 31)) & 1u); }

// Bound by HBM: the 32-byte sectors of a record that hold its duration, region and ctx. A warp walks one slice of a stream.
// Where the workspace has a place for every interval the entries go straight to their slice's; else the warp collects them
// and appends about 100 at a time, exactly as many places as it needs, as pieces of a chain.
__global__ void __launch_bounds__(kSelThreads) k_ov_select(OvSelectArgs a) {
  argus_kernel_begin_long();
  __shared__ u32 filter[kSelFilter / 32];
  __shared__ u32 sh_pairs[2 * ARGUS_MAX_PAIRS];
  __shared__ u64 stage[kSelWarps][kSelStage];
  for (u32 i = threadIdx.x; i < kSelFilter / 32; i += blockDim.x) filter[i] = 0;
  __syncthreads();
  for (u32 i = threadIdx.x; i < 2 * a.num_pairs; i += blockDim.x) {
    const u32 r = a.pairs[i];
    sh_pairs[i] = r;
    atomicOr(&filter[(r & (kSelFilter - 1)) >> 5], 1u << (r & 31));
  }
  __syncthreads();
  const u32 lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const u32 parts = a.slices / kSelWarps, heads = a.num_streams * a.slices;
  u64* const mine = stage[warp];
  for (u64 item = blockIdx.x; item < (u64)a.num_streams * parts; item += gridDim.x) {
    const u32 s = (u32)(item / parts), slice = (u32)(item % parts) * kSelWarps + warp;
    const u32 head = s * a.slices + slice;
    const u32 m = a.cta_sm[s / a.warps_per_cta];
    const u64 lo = a.interval_offsets[s], hi = a.interval_offsets[s + 1];
    bool take = true;
    if (m >= a.num_sms || hi < lo || hi > a.max_intervals || ((hi - lo) >> 32)) {  // offsets beyond the interval array are reported, not read
      if (threadIdx.x == 0 && m >= a.num_sms) argus_report_bad_sm(a.status, a.cta_sm, a.num_sms, a.warps_per_cta, s / a.warps_per_cta);
      else if (threadIdx.x == 0) argus_set_error(a.status, ARGUS_ERR_BAD_OFFSETS, s, m);
      take = false;
    } else if (a.scoped) {  // warp-role and SM tests: one answer per stream
      const u32 w = s % a.warps_per_cta;
      if (a.warp_mask != ~0ull && (w >= 64 || !((a.warp_mask >> w) & 1ull))) take = false;
      if (!ov_mask_bit(a.sm_mask, m)) take = false;
    }
    const u32 n = take ? (u32)(hi - lo) : 0u;
    u32 i0, i1;
    argus_ov_slice(n, a.slices, slice, &i0, &i1);
    const argus_interval_t* const ivs = a.intervals + lo;
    u64* const to = a.direct ? a.entries + lo + i0 : mine;
    u32 held = 0, last = head, total_pieces = 0;
    if (lane == 0) { ArgusOvPiece e; e.pos = 0; e.count = 0; e.next = kOvNone; a.pieces[head] = e; }
    for (u32 base = i0; base < i1 || (held && !a.direct); base += 32) {
      const bool end = base >= i1;
      u32 bal = 0, region = 0;
      bool cand = false;
      if (!end) {
        const u32 i = base + lane;
        if (i < i1) {
          const uint4* p = reinterpret_cast<const uint4*>(ivs + i);
          const u64 incl = __ldg(reinterpret_cast<const u64*>(p) + 1);
          const uint2 rc = __ldg(reinterpret_cast<const uint2*>(p + 1) + 1);
          region = rc.x;
          cand = incl != 0 && ((filter[(region & (kSelFilter - 1)) >> 5] >> (region & 31)) & 1u);
          // iteration-window and region tests: one answer per interval
          if (cand && a.scoped) cand = rc.y >= a.ctx_lo && rc.y <= a.ctx_hi && ov_mask_bit(a.region_mask, region);
        }
        bal = __ballot_sync(0xffffffffu, cand);
        if (bal) {  // the filter lets a few other regions through
          if (cand) {
            bool hit = false;
            for (u32 k = 0; k < 2 * a.num_pairs && !hit; ++k) hit = sh_pairs[k] == region;
            cand = hit;
          }
          bal = __ballot_sync(0xffffffffu, cand);
        }
        if (cand) to[held + __popc(bal & ((1u << lane) - 1u))] = (u64)i | ((u64)region << 32);
        held += __popc(bal);
        __syncwarp();
      }
      if (!a.direct && (held > kSelStage - 32 || end)) {
        u64 pos = 0;
        u32 piece = head;
        if (lane == 0) {
          pos = atomicAdd(&a.ctl->num_entries, (u64)held);
          if (total_pieces) piece = heads + atomicAdd(&a.ctl->num_pieces, 1u);
        }
        pos = __shfl_sync(0xffffffffu, pos, 0);
        piece = __shfl_sync(0xffffffffu, piece, 0);
        if (pos + held <= a.entry_capacity && piece < a.piece_capacity) {  // else the counter tells that they did not fit
          for (u32 t = lane; t < held; t += 32) a.entries[pos + t] = mine[t];
          if (lane == 0) {
            ArgusOvPiece e; e.pos = pos; e.count = held; e.next = kOvNone;
            a.pieces[piece] = e;
            if (total_pieces) a.pieces[last].next = piece;
          }
          last = piece;
          ++total_pieces;
        }
        held = 0;
        __syncwarp();
        if (end) break;
      }
    }
    if (a.direct && lane == 0) { ArgusOvPiece e; e.pos = lo + i0; e.count = held; e.next = kOvNone; a.pieces[head] = e; }
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------------------------------------------------
constexpr u32 kVT = 9;                                 // spans a thread merges at a time (odd: lanes that far apart hit different banks)
__host__ __device__ constexpr u32 bucket_word(u32 b) { return b + (b >> 5); }  // padded: threads sum up runs of counters without bank conflicts
constexpr u32 kSorted = 9216;                          // spans of both roles that are sorted at once, whatever the block's size: 144 KB
constexpr u32 kBucketBits = 13;                        // 2^kBucketBits buckets of a role at most
constexpr size_t kPairSmem = (size_t)kSorted * sizeof(ulonglong2);
static_assert(kSorted <= 1u << 14, "places fit 14 bits");
static_assert((2u << kBucketBits) >= kSorted && (size_t)kSorted * 8 + bucket_word(2u << kBucketBits) * 4 <= kPairSmem, "a bucket a span, in the tile's room");
template <u32 NT>
struct PairSizes {                                     // of a block of NT threads
  static constexpr u32 kWarps = NT / 32;
  static constexpr u32 kTile = NT * kVT;               // spans that are merged at a time
  static constexpr u32 kBatch = NT;                    // slices whose spans are placed at a time
  static_assert(kTile <= kSorted, "a tile fits shared memory");
};

struct OvPairArgs {
  const argus_interval_t* intervals;
  const u64* interval_offsets;
  const u64* starts;    // begin times, at the entries' positions (entries from digests)
  const u64* entries;
  const ArgusOvPiece* pieces;
  u32 slices, num_streams, warps_per_cta, num_sms, num_pairs, blocks;
  const u32* cta_sm;
  const u32* pairs;
  argus_overlap_t* out;
  argus_status_t* status;
  ulonglong2* spans;    // [capacity] (start, end) of the producer role, from the block's base on; what it leaves, the other side of a merge
  ulonglong2* scratch;  // [capacity] the same for the consumer role
  u64 capacity, entry_capacity;
  ArgusOvCtl* ctl;
};

__device__ __forceinline__ bool before_or_at(const ulonglong2& x, const ulonglong2& y) { return x.x <= y.x; }

// Number of the first `diag` elements of the merge of A and B that come from A (elements of A first on ties).
__device__ __forceinline__ u32 merge_split(const ulonglong2* A, u32 na, const ulonglong2* B, u32 nb, u32 diag) {
  u32 lo = diag > nb ? diag - nb : 0u, hi = diag < na ? diag : na;
  while (lo < hi) {
    const u32 mid = (lo + hi) >> 1;
    if (before_or_at(A[mid], B[diag - 1 - mid])) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// The same by one warp, 32 probes a round (for arrays in global memory, where a probe is a round trip to the L2).
__device__ __forceinline__ u64 merge_split_warp(const ulonglong2* A, u64 na, const ulonglong2* B, u64 nb, u64 diag, u32 lane) {
  u64 lo = diag > nb ? diag - nb : 0ull, hi = diag < na ? diag : na;
  while (lo < hi) {
    const u64 step = (hi - lo + 31) >> 5, mid = lo + lane * step;
    const bool yes = mid < hi && __ldcg(&A[mid].x) <= __ldcg(&B[diag - 1 - mid].x);
    const u32 c = __popc(__ballot_sync(0xffffffffu, yes));  // the probes that say yes come first
    if (c == 0) break;
    const u64 nlo = lo + (c - 1) * step + 1, nhi = lo + c * step;
    lo = nlo;
    if (nhi < hi) hi = nhi;
  }
  return lo;
}

// One thread's share of a merge in shared memory: kVT elements from A[a..na) and B[b..nb) into registers; elements past the
// end of both are left alone.
__device__ __forceinline__ void merge_serial(const ulonglong2* A, u32 a, u32 na, const ulonglong2* B, u32 b, u32 nb, ulonglong2 (&v)[kVT]) {
#pragma unroll
  for (u32 j = 0; j < kVT; ++j) {
    if (a < na || b < nb) {
      const ulonglong2 x = A[a < na ? a : 0], y = B[b < nb ? b : 0];
      const bool take_a = b >= nb || (a < na && before_or_at(x, y));
      v[j] = take_a ? x : y;
      if (take_a) ++a; else ++b;
    }
  }
}

// Sorts t[0..cnt) in shared memory by start time: kVT elements a thread in registers, then merges of doubling width.
template <u32 NT>
__device__ __noinline__ void sort_tile(ulonglong2* t, u32 cnt) {
  const u32 at = threadIdx.x * kVT;
  ulonglong2 v[kVT];
  if (at < cnt) {
#pragma unroll
    for (u32 j = 0; j < kVT; ++j) v[j] = at + j < cnt ? t[at + j] : make_ulonglong2(~0ull, ~0ull);
#pragma unroll
    for (u32 r = 0; r < kVT; ++r)  // odd-even transposition
#pragma unroll
      for (u32 j = r & 1u; j + 1 < kVT; j += 2)
        if (v[j + 1].x < v[j].x) { const ulonglong2 x = v[j]; v[j] = v[j + 1]; v[j + 1] = x; }
    // (padding has the largest key; equal keys keep their order, so padding stays last)
#pragma unroll
    for (u32 j = 0; j < kVT; ++j) if (at + j < cnt) t[at + j] = v[j];
  }
  __syncthreads();
  for (u32 width = kVT; width < cnt; width <<= 1) {
    const u32 a0 = at / (2 * width) * (2 * width), b0 = a0 + width < cnt ? a0 + width : cnt, e0 = a0 + 2 * width < cnt ? a0 + 2 * width : cnt;
    const bool work = at < cnt && b0 < e0 && t[b0].x < t[b0 - 1].x;  // runs that follow one another need no merge
    if (work) {
      const u32 na = b0 - a0, nb = e0 - b0, diag = at - a0;
      const u32 a = merge_split(t + a0, na, t + b0, nb, diag);
      merge_serial(t + a0, a, na, t + b0, diag - a, nb, v);
    }
    __syncthreads();
    if (work) {
#pragma unroll
      for (u32 j = 0; j < kVT; ++j) if (at + j < cnt) t[at + j] = v[j];
    }
    __syncthreads();
  }
}

// Sorts d[0..n) in global memory by start time; `scratch` has as much room. Returns where the sorted spans lie.
template <u32 NT>
__device__ __noinline__ ulonglong2* sort_spans(ulonglong2* d, ulonglong2* scratch, u64 n, ulonglong2* t, u64* sh) {
  constexpr u32 kTile = PairSizes<NT>::kTile;
  for (u64 t0 = 0; t0 < n; t0 += kTile) {
    const u32 cnt = (u32)(n - t0 < kTile ? n - t0 : kTile);
    for (u32 i = threadIdx.x; i < cnt; i += NT) t[i] = d[t0 + i];
    __syncthreads();
    sort_tile<NT>(t, cnt);
    for (u32 i = threadIdx.x; i < cnt; i += NT) d[t0 + i] = t[i];
    __syncthreads();
  }
  const u32 lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (u64 width = kTile; width < n; width <<= 1) {
    for (u64 t0 = 0; t0 < n; t0 += kTile) {  // every tile of the output lies inside one merge (widths are multiples of a tile)
      const u64 a0 = t0 / (2 * width) * (2 * width), b0 = a0 + width < n ? a0 + width : n, e0 = a0 + 2 * width < n ? a0 + 2 * width : n;
      const u64 d0 = t0 - a0, d1 = (t0 + kTile < e0 ? t0 + kTile : e0) - a0;
      if (warp < 2) {
        const u64 sp = merge_split_warp(d + a0, b0 - a0, d + b0, e0 - b0, warp ? d1 : d0, lane);
        if (lane == 0) sh[warp] = sp;
      }
      __syncthreads();
      const u64 aA = sh[0], aB = sh[1];
      const u32 na = (u32)(aB - aA), cnt = (u32)(d1 - d0), nb = cnt - na;
      for (u32 i = threadIdx.x; i < cnt; i += NT) t[i] = i < na ? d[a0 + aA + i] : d[b0 + (d0 - aA) + (i - na)];
      __syncthreads();
      const u32 at = threadIdx.x * kVT;
      ulonglong2 v[kVT];
      if (at < cnt) {
        const u32 a = merge_split(t, na, t + na, nb, at);
        merge_serial(t, a, na, t + na, at - a, nb, v);
      }
      __syncthreads();
#pragma unroll
      for (u32 j = 0; j < kVT; ++j) if (at + j < cnt) t[at + j] = v[j];
      __syncthreads();
      for (u32 i = threadIdx.x; i < cnt; i += NT) scratch[t0 + i] = t[i];
      __syncthreads();
    }
    ulonglong2* const x = d; d = scratch; scratch = x;
  }
  return d;
}

// Sort of both roles together, up to kSorted spans (in0[0..n0), in1[0..n1); a role that is in order already comes with n = 0),
// into out0 and out1: spans are spread over buckets of equal width in start time, about one for a span, and a span's place is
// the number of earlier ones in its bucket. Elements are 8 bytes, start time relative to the role's earliest (50 bits) and place (14
// bits); the spans follow once (4,096 spans a role: 20 us; merging runs pairwise took 50 us). Returns false, the same for
// all threads and with nothing written, when a bucket would hold
// more than kBucketMost (starts that crowd) or a role's starts spread over 2^50 ticks: the caller then merges.
constexpr u32 kBucketMost = 32;
template <u32 NT>
__device__ __noinline__ bool sort_buckets(const ulonglong2* in0, const ulonglong2* in1, u32 n0, u32 n1, ulonglong2* out0, ulonglong2* out1,
                                          ulonglong2* room, u64 (*red)[NT / 32 + 1], u32 (&scan)[33]) {
  constexpr u32 kWarps = NT / 32;
  u64* const t = reinterpret_cast<u64*>(room);
  u32* const cnt = reinterpret_cast<u32*>(t + kSorted);  // a role's counters after the other's; then where a bucket ends
  const u32 n = n0 + n1, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  u32 bits = 5;  // 2^bits buckets a role
  while (bits < kBucketBits && (2u << bits) < n) ++bits;
  const u32 nb = 2u << bits;
  for (u32 b = threadIdx.x; b < nb; b += NT) cnt[bucket_word(b)] = 0;
  u64 low0 = ~0ull, low1 = ~0ull, high0 = 0, high1 = 0;
#pragma unroll 1
  for (u32 i = threadIdx.x; i < n; i += NT) {
    const u64 x = i < n0 ? in0[i].x : in1[i - n0].x;
    if (i < n0) { low0 = x < low0 ? x : low0; high0 = x > high0 ? x : high0; }
    else { low1 = x < low1 ? x : low1; high1 = x > high1 ? x : high1; }
  }
  u32 shift0 = 0, shift1 = 0;
#pragma unroll 1
  for (int role = 0; role < 2; ++role) {
    u64 mn = role ? low1 : low0, mx = role ? high1 : high0;
#pragma unroll 1
    for (int step = 0; step < 2; ++step) {
#pragma unroll
      for (int dd = 16; dd > 0; dd >>= 1) {
        const u64 a = __shfl_xor_sync(0xffffffffu, mn, dd), b = __shfl_xor_sync(0xffffffffu, mx, dd);
        mn = a < mn ? a : mn; mx = b > mx ? b : mx;
      }
      if (step) break;
      if (lane == 0) { red[0][warp] = mn; red[1][warp] = mx; }
      __syncthreads();
      mn = lane < kWarps ? red[0][lane] : ~0ull; mx = lane < kWarps ? red[1][lane] : 0ull;
      __syncthreads();
    }
    const u64 range = mx > mn ? mx - mn : 0ull;
    if (range >> 50) return false;
    const u32 have = 64u - (u32)__clzll((long long)range), sh = have > bits ? have - bits : 0u;  // range < 2^have
    if (role) { low1 = mn; shift1 = sh; } else { low0 = mn; shift0 = sh; }
  }
#pragma unroll 1
  for (u32 i = threadIdx.x; i < n; i += NT) {
    const bool role = i >= n0;
    const u64 x = role ? in1[i - n0].x - low1 : in0[i].x - low0;
    atomicAdd(&cnt[bucket_word((role ? 1u << bits : 0u) + (u32)(x >> (role ? shift1 : shift0)))], 1u);
  }
  __syncthreads();
  const u32 per = (nb + NT - 1) / NT, c0 = threadIdx.x * per;  // counters a thread sums up: consecutive ones
  u32 mine = 0, most = 0;
  for (u32 b = c0; b < c0 + per && b < nb; ++b) { const u32 c = cnt[bucket_word(b)]; mine += c; most = c > most ? c : most; }
  if (__syncthreads_or(most > kBucketMost)) return false;
  u32 total;
  u32 at = argus_block_exclusive_scan<u32>(mine, scan, &total);
  for (u32 b = c0; b < c0 + per && b < nb; ++b) { const u32 c = cnt[bucket_word(b)]; cnt[bucket_word(b)] = at; at += c; }
  __syncthreads();
#pragma unroll 1
  for (u32 i = threadIdx.x; i < n; i += NT) {
    const bool role = i >= n0;
    const u64 x = role ? in1[i - n0].x - low1 : in0[i].x - low0;
    t[atomicAdd(&cnt[bucket_word((role ? 1u << bits : 0u) + (u32)(x >> (role ? shift1 : shift0)))], 1u)] = (x << 14) | i;
  }
  __syncthreads();
#pragma unroll 1
  for (u32 i = threadIdx.x; i < n; i += NT) {  // the counter of a bucket is now where it ends
    const bool role = i >= n0;  // (the first n0 elements are role 0's)
    const u64 v = t[i];
    const u32 b = (role ? 1u << bits : 0u) + (u32)((v >> 14) >> (role ? shift1 : shift0)), from = (u32)v & 0x3fffu;
    const u32 b0 = b ? cnt[bucket_word(b - 1)] : 0u, b1 = cnt[bucket_word(b)];
    u32 to = b0;
    for (u32 k = b0; k < b1; ++k) to += t[k] < v;
    if (role) out1[to - n0] = in1[from - n0]; else out0[to] = in0[from];
  }
  __syncthreads();
  return true;
}

// d[0..n) in start order -> the disjoint pieces of their union: piece i = [max(start_i, E), max(end_i, that)) with E the largest
// end of the spans before i (pieces may be empty). Returns this thread's share of the sum of their lengths.
template <u32 NT>
__device__ __noinline__ u64 cut_pieces(ulonglong2* d, u64 n, u64* red) {
  const u32 lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  u64 carry = 0, len = 0;
#pragma unroll 1
  for (u64 i0 = 0; i0 < n; i0 += NT) {
    const u64 at = i0 + threadIdx.x;
    const ulonglong2 s = at < n ? d[at] : make_ulonglong2(0, 0);
    u64 e = s.y;
#pragma unroll
    for (int dd = 1; dd < 32; dd <<= 1) {
      const u64 o = __shfl_up_sync(0xffffffffu, e, dd);
      if (lane >= (u32)dd && o > e) e = o;
    }
    if (lane == 31) red[warp] = e;
    __syncthreads();
    u64 w = lane < NT / 32 ? red[lane] : 0ull;
#pragma unroll
    for (int dd = 1; dd < 32; dd <<= 1) {
      const u64 o = __shfl_up_sync(0xffffffffu, w, dd);
      if (lane >= (u32)dd && o > w) w = o;
    }
    u64 before = __shfl_up_sync(0xffffffffu, e, 1);
    if (lane == 0) before = 0;
    const u64 warps_before = warp ? __shfl_sync(0xffffffffu, w, warp - 1) : 0ull, all = __shfl_sync(0xffffffffu, w, 31);
    before = before > warps_before ? before : warps_before;
    before = before > carry ? before : carry;
    if (at < n) {
      const u64 a = s.x > before ? s.x : before, b = s.y > a ? s.y : a;
      d[at] = make_ulonglong2(a, b);
      len += b - a;
    }
    carry = all > carry ? all : carry;
    __syncthreads();
  }
  return len;
}

// Latency decides (one block per SM and pair). The entries of up to kBatch slices are taken as one flat sequence, so that
// every thread has kGather entries and then as many begin times (or pieces of records) in flight, whatever the slices hold.
// 148 SMs, two roles of 16,000 spans each: 109 us (five kernels before it: 393 us), about 6.5 a group of 4,096 entries and 10 a tile of
// the walk; a few hundred spans: 25 with 1,024 threads, 21 with 512, most of it fixed steps one after the other.
// DIGEST: entries as the pass over the digests leaves them (argus_fuse.cuh); else {index in the stream, region}.
template <bool DIGEST, u32 NT, u32 kGather>
__global__ void __launch_bounds__(NT, 1) k_ov_pair(OvPairArgs a) {
  using Z = PairSizes<NT>;
  constexpr u32 kPairThreads = NT, kPairWarps = Z::kWarps, kTile = Z::kTile, kBatch = Z::kBatch;
  argus_kernel_begin_long();
  extern __shared__ __align__(16) unsigned char pair_raw[];
  ulonglong2* const tile = reinterpret_cast<ulonglong2*>(pair_raw);
  __shared__ u32 sh_hit[kPairThreads];             // CTAs of this SM among the ones just looked at
  __shared__ u32 sh_ex[kBatch + 1];                // entries of the batch before slice i
  __shared__ u64 sh_pos[kBatch], sh_iv[kBatch];    // where a slice's entries and its stream's intervals start
  __shared__ u32 sh_scan[33];
  __shared__ u64 sh_scan64[33];
  __shared__ u64 sh64[4];
  __shared__ u64 red[2][kPairWarps + 1];
  __shared__ u32 sh_cnt[kGather * kPairWarps];
  __shared__ u32 sh_u;
  const u32 tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const u32 k = blockIdx.x / a.num_sms, m = blockIdx.x % a.num_sms;
  const u32 P = a.pairs[2 * k], C = a.pairs[2 * k + 1];
  const u32 num_ctas = a.num_streams / a.warps_per_cta, per_cta = a.warps_per_cta * a.slices;
  if (tid == 0) {
    sh_u = __ldcg(&a.status->code);
    if (a.ctl->num_entries > a.entry_capacity) {  // the selection ran out of room
      sh_u = ARGUS_ERR_CAPACITY;
      if (blockIdx.x == 0) {
        argus_set_error(a.status, ARGUS_ERR_CAPACITY, 0, a.ctl->num_entries);
        a.status->intervals_required = a.ctl->num_entries;
      }
    }
  }
  __syncthreads();
  // (a capacity error that another block of this launch reports is not waited for: such a block has no room itself or is done)
  if (sh_u != 0) {  // nothing measured: zeros
    if (tid == 0) a.out[blockIdx.x] = argus_overlap_t{};
    return;
  }

  // ---- gather: round 0 counts, round 1 places, in stream and slice order ----
  // With one pair every entry is in a role of it, and round 0 only adds up the pieces.
  u64 nP = 0, nC = 0, base = 0;
  bool suspect[2] = {false, false};  // this thread has seen a span of the role that starts before the end of the one before it
  u64 len[2] = {0, 0};               // this thread's share of |U_P| and |U_C|
  u64 carry_p = 0, carry_c = 0;      // end of the last span of a role
  ArgusOvPiece held; held.pos = 0; held.count = 0; held.next = kOvNone;
  bool hold = false;                 // one batch holds everything: its CTAs and first pieces are kept from round 0
  u32 hits = 0;
  for (int round = 0; round < 2; ++round) {
    u64 my_all = 0, my_p = 0, my_c = 0;  // round 0, per thread
    for (u32 c0 = 0; c0 < num_ctas; c0 += kPairThreads) {
      if (!hold) {
        const bool hit = c0 + tid < num_ctas && a.cta_sm[c0 + tid] == m;
        const u32 ex = argus_block_exclusive_scan<u32>(hit ? 1u : 0u, sh_scan, &hits);
        if (hit) sh_hit[ex] = c0 + tid;
        __syncthreads();
      }
      const u64 heads = (u64)hits * per_cta;
      hold = num_ctas <= kPairThreads && heads <= kBatch;
      for (u64 h0 = 0; h0 < heads; h0 += kBatch) {
        u32 piece = kOvNone;
        u64 iv0 = 0;
        if (h0 + tid < heads) {
          const u32 cta = sh_hit[(h0 + tid) / per_cta], rest = (u32)((h0 + tid) % per_cta);
          piece = cta * per_cta + rest;
          if (!DIGEST) iv0 = a.interval_offsets[cta * a.warps_per_cta + rest / a.slices];
        }
        // (chains of pieces are taken one link at a time: the spans are then no longer in slice order, and get sorted)
        do {
          ArgusOvPiece pc; pc.pos = 0; pc.count = 0; pc.next = kOvNone;
          if (piece != kOvNone) {
            const bool first = piece < num_ctas * per_cta;
            pc = round == 1 && hold && first ? held : a.pieces[piece];
            if (hold && first) held = pc;
          }
          piece = pc.next;
          if (round == 0 && a.num_pairs == 1) { my_all += pc.count; continue; }
          // slices that hold something, one after the other: where each starts in the flat sequence
          u64 all;
          const u64 ex = argus_block_exclusive_scan<u64>((u64)pc.count | (pc.count ? 1ull << 32 : 0ull), sh_scan64, &all);
          const u32 total = (u32)all, slices = (u32)(all >> 32);
          if (pc.count) {
            const u32 at = (u32)(ex >> 32);
            sh_ex[at] = (u32)ex;
            sh_pos[at] = pc.pos;
            if (!DIGEST) sh_iv[at] = iv0;
          }
          for (u32 i = slices + tid; i <= kBatch; i += kPairThreads) sh_ex[i] = total;
          __syncthreads();
          for (u32 e0 = 0; e0 < total; e0 += kPairThreads * kGather) {
            u64 ent[kGather];
            u32 at[kGather];
            u32 is_p = 0, is_c = 0;
#pragma unroll
            for (u32 j = 0; j < kGather; ++j) {
              at[j] = 0; ent[j] = 0;
              if (e0 + j * kPairThreads >= total) continue;
              const u32 f = e0 + j * kPairThreads + tid, f0 = f - lane;
              // the slice of the warp's first entry: the last one that starts at or before it, 32 probes at a time
              u32 lo = 32u * ((u32)__popc(__ballot_sync(0xffffffffu, lane < kBatch / 32 && sh_ex[32 * lane % kBatch] <= f0)) - 1u);
              lo += (u32)__popc(__ballot_sync(0xffffffffu, sh_ex[lo + lane] <= f0)) - 1u;
              if (f < total) while (f >= sh_ex[lo + 1]) ++lo;
              at[j] = lo;
              if (f < total) ent[j] = __ldcg(a.entries + sh_pos[lo] + (f - sh_ex[lo]));
            }
#pragma unroll
            for (u32 j = 0; j < kGather; ++j) {
              const bool in = e0 + j * kPairThreads + tid < total;
              const u32 region = DIGEST ? (u32)ent[j] & 0xffffu : (u32)(ent[j] >> 32);
              if (in && region == P) is_p |= 1u << j;
              if (in && region == C) is_c |= 1u << j;
            }
            if (round == 0) { my_p += __popc(is_p); my_c += __popc(is_c); continue; }
            ulonglong2 q[kGather];  // begin time and duration
#pragma unroll
            for (u32 j = 0; j < kGather; ++j) {
              if (!(((is_p | is_c) >> j) & 1u)) continue;
              if (DIGEST) {
                if ((u32)ent[j] & kDigestWide) {
                  q[j] = __ldg(reinterpret_cast<const ulonglong2*>(a.intervals + sh_pos[at[j]] + (ent[j] >> 18)));
                } else {
                  q[j].x = __ldcg(a.starts + sh_pos[at[j]] + (e0 + j * kPairThreads + tid - sh_ex[at[j]]));
                  q[j].y = (ent[j] >> 18) & ((1u << kDigestBits) - 1u);
                }
              } else {
                q[j] = __ldg(reinterpret_cast<const ulonglong2*>(a.intervals + sh_iv[at[j]] + (u32)ent[j]));
              }
            }
            // places: entries of a role before (j, warp, lane)
            u32 bp[kGather], bc[kGather];
#pragma unroll
            for (u32 j = 0; j < kGather; ++j) {
              bp[j] = __ballot_sync(0xffffffffu, (is_p >> j) & 1u);
              bc[j] = __ballot_sync(0xffffffffu, (is_c >> j) & 1u);
              if (lane == 0) sh_cnt[j * kPairWarps + warp] = (u32)__popc(bp[j]) | ((u32)__popc(bc[j]) << 16);
            }
            __syncthreads();
            if (warp == 0) {
              u32 c[kGather], sum = 0;
#pragma unroll
              for (u32 j = 0; j < kGather; ++j) { c[j] = lane < kPairWarps ? sh_cnt[lane * kGather + j] : 0u; sum += c[j]; }
              u32 incl = sum;
#pragma unroll
              for (int dd = 1; dd < 32; dd <<= 1) { const u32 o = __shfl_up_sync(0xffffffffu, incl, dd); if (lane >= (u32)dd) incl += o; }
              u32 ex = incl - sum;
#pragma unroll
              for (u32 j = 0; j < kGather; ++j) { if (lane < kPairWarps) sh_cnt[lane * kGather + j] = ex; ex += c[j]; }
              if (lane == 31) sh_u = incl;
            }
            __syncthreads();
            const u32 tot = sh_u, tot_p = tot & 0xffffu, tot_c = tot >> 16, lt = (1u << lane) - 1u;
            u64* const ends_p = reinterpret_cast<u64*>(tile);      // ends_p[i]: end of the role's span before place i of the group
            u64* const ends_c = ends_p + kPairThreads * kGather + 1;
            if (tid == 0) { ends_p[0] = carry_p; ends_c[0] = carry_c; }
#pragma unroll
            for (u32 j = 0; j < kGather; ++j) {
              const ulonglong2 span = make_ulonglong2(q[j].x, q[j].x + q[j].y);
              const u32 before = sh_cnt[j * kPairWarps + warp];
              if ((is_p >> j) & 1u) {
                const u32 r = (before & 0xffffu) + (u32)__popc(bp[j] & lt);
                a.spans[base + nP + r] = span;
                ends_p[r + 1] = span.y;
                len[0] += span.y - span.x;
              }
              if ((is_c >> j) & 1u) {
                const u32 r = (before >> 16) + (u32)__popc(bc[j] & lt);
                a.scratch[base + nC + r] = span;
                ends_c[r + 1] = span.y;
                len[1] += span.y - span.x;
              }
            }
            __syncthreads();
#pragma unroll
            for (u32 j = 0; j < kGather; ++j) {  // in order and disjoint so far?
              const u64 e = q[j].x + q[j].y;
              const u32 before = sh_cnt[j * kPairWarps + warp];
              if ((is_p >> j) & 1u) suspect[0] |= q[j].x < ends_p[(before & 0xffffu) + (u32)__popc(bp[j] & lt)] || e < q[j].x;
              if ((is_c >> j) & 1u) suspect[1] |= q[j].x < ends_c[(before >> 16) + (u32)__popc(bc[j] & lt)] || e < q[j].x;
            }
            carry_p = ends_p[tot_p];
            carry_c = ends_c[tot_c];
            nP += tot_p;
            nC += tot_c;
            __syncthreads();
          }
          __syncthreads();  // sh_ex and sh_pos are overwritten next
        } while (__syncthreads_or(piece != kOvNone));
      }
      __syncthreads();  // sh_hit is overwritten next
    }
    if (round == 0) {
      u64 mine = a.num_pairs == 1 ? (P == C ? 2 * my_all : my_all) : my_p + my_c;
#pragma unroll
      for (int dd = 16; dd > 0; dd >>= 1) mine += __shfl_down_sync(0xffffffffu, mine, dd);
      if (lane == 0) red[0][warp] = mine;
      __syncthreads();
      if (tid == 0) {  // room for this block's spans; the last block to ask knows whether everybody's fitted
        u64 all = 0;
        for (u32 w = 0; w < kPairWarps; ++w) all += red[0][w];
        sh64[0] = all ? atomicAdd(&a.ctl->num_spans, all) : 0ull;
        sh64[1] = all;
      }
      __syncthreads();
      if (tid == 0) {
        __threadfence();
        if (atomicAdd(&a.ctl->asked, 1u) == a.blocks - 1) {
          const u64 total = *reinterpret_cast<volatile u64*>(&a.ctl->num_spans);
          if (total > a.capacity) {
            argus_set_error(a.status, ARGUS_ERR_CAPACITY, 0, total);
            a.status->intervals_required = total;
          }
        }
      }
      base = sh64[0];
      if (base + sh64[1] > a.capacity) {
        if (tid == 0) a.out[blockIdx.x] = argus_overlap_t{};
        return;
      }
      if (sh64[1] == 0) break;
    }
  }

  // ---- sorted, disjoint pieces of both roles ----
  const u64 total = nP + nC;
  ulonglong2 *A = a.spans + base, *B = a.scratch + base;
  {
    const bool cut_a = __syncthreads_or(suspect[0]), cut_b = __syncthreads_or(suspect[1]);
    ulonglong2 *const free_a = a.scratch + base + nC, *const free_b = a.spans + base + nP;  // as much room again for either role
    if (cut_a || cut_b) {
      if ((cut_a ? nP : 0ull) + (cut_b ? nC : 0ull) <= kSorted &&
          sort_buckets<NT>(A, B, cut_a ? (u32)nP : 0u, cut_b ? (u32)nC : 0u, free_a, free_b, tile, red, sh_scan)) {
        if (cut_a) A = free_a;
        if (cut_b) B = free_b;
      } else {
        if (cut_a) A = sort_spans<NT>(A, free_a, nP, tile, sh64);
        if (cut_b) B = sort_spans<NT>(B, free_b, nC, tile, sh64);
      }
      if (cut_a) len[0] = cut_pieces<NT>(A, nP, red[0]);
      if (cut_b) len[1] = cut_pieces<NT>(B, nC, red[1]);
    }
  }
  __syncthreads();

  // ---- walk of the merged sequence ----
  // a piece that starts inside the last piece of the other role overlaps it, and no other
  u64 both = 0;
  u64 a0 = 0;  // producer pieces taken so far
  for (u64 t0 = 0; nP && nC && t0 < total; t0 += kTile) {
    const u32 cnt = (u32)(total - t0 < kTile ? total - t0 : kTile), step = (u32)((t0 / kTile) % kPairWarps);
    if (step == 0) {  // where the next tiles end, one warp each
      const u64 to = t0 + (u64)(warp + 1) * kTile;
      const u64 s1 = to >= total ? nP : merge_split_warp(A, nP, B, nC, to, lane);
      if (lane == 0) red[0][warp] = s1;
      __syncthreads();
    }
    const u64 a1 = red[0][step], b0 = t0 - a0;
    const u32 na = (u32)(a1 - a0), nb = cnt - na;
    const u64 last_a = a0 ? A[a0 - 1].y : 0ull, last_b = b0 ? B[b0 - 1].y : 0ull;
#pragma unroll
    for (u32 j = 0; j < kVT; ++j) {
      const u32 i = j * kPairThreads + tid;
      if (i < cnt) tile[i] = i < na ? A[a0 + i] : B[b0 + (i - na)];
    }
    __syncthreads();
    const u32 at = tid * kVT;
    if (at < cnt) {
      u32 x = merge_split(tile, na, tile + na, nb, at), y = at - x;
      u64 end_a = x ? tile[x - 1].y : last_a, end_b = y ? tile[na + y - 1].y : last_b;
      ulonglong2 va = x < na ? tile[x] : make_ulonglong2(~0ull, ~0ull), vb = y < nb ? tile[na + y] : make_ulonglong2(~0ull, ~0ull);
#pragma unroll
      for (u32 j = 0; j < kVT; ++j) {
        if (at + j < cnt) {
          const bool take_a = y >= nb || (x < na && va.x <= vb.x);
          const u64 s = take_a ? va.x : vb.x, e = take_a ? va.y : vb.y, other = take_a ? end_b : end_a;
          const u64 upto = e < other ? e : other;
          if (upto > s) both += upto - s;
          if (take_a) { end_a = e; ++x; if (x < na) va = tile[x]; }
          else { end_b = e; ++y; if (y < nb) vb = tile[na + y]; }
        }
      }
    }
    a0 = a1;
    __syncthreads();
  }
#pragma unroll
  for (int dd = 16; dd > 0; dd >>= 1) {
    len[0] += __shfl_down_sync(0xffffffffu, len[0], dd);
    len[1] += __shfl_down_sync(0xffffffffu, len[1], dd);
    both += __shfl_down_sync(0xffffffffu, both, dd);
  }
  __syncthreads();
  if (tid < 3) sh64[tid] = 0;
  __syncthreads();
  if (lane == 0) {
    if (len[0]) atomicAdd(&sh64[0], len[0]);
    if (len[1]) atomicAdd(&sh64[1], len[1]);
    if (both) atomicAdd(&sh64[2], both);
  }
  __syncthreads();
  if (tid == 0) {
    argus_overlap_t o;
    o.producer_ns = sh64[0]; o.consumer_ns = sh64[1]; o.overlap_ns = sh64[2];
    o.either_ns = o.producer_ns + o.consumer_ns - o.overlap_ns;
    a.out[blockIdx.x] = o;
  }
}

// What the list path needs per span besides its fixed part: two places for the span, an entry, its share of a piece.
constexpr size_t kBytesPerSpan = 16 + 16 + 8 + 1;

u32 select_slices(u32 num_streams) {
  u32 parts = num_streams ? kSelGrid / num_streams : 1u;  // few streams: several blocks walk one
  parts = parts < 1 ? 1 : parts > 8 ? 8 : parts;
  return parts * kSelWarps;
}

size_t ov_fixed_bytes(u32 num_streams) {
  return argus_align_up(sizeof(ArgusOvCtl), 256) + argus_align_up((size_t)num_streams * select_slices(num_streams) * sizeof(ArgusOvPiece), 256) + 1024;
}

template <bool DIGEST, u32 NT, u32 kGather>
int launch_pair_as(const OvPairArgs& a, cudaStream_t stream) {
  static std::atomic<bool> opted_in[64];  // the shared-memory opt-in belongs to a device
  int dev = 0;
  ARGUS_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return ARGUS_ERR_INVALID_ARG;
  if (!opted_in[dev].load(std::memory_order_acquire)) {
    ARGUS_CUDA_TRY(argus_allow_smem(k_ov_pair<DIGEST, NT, kGather>, kPairSmem, kPairSmem));
    opted_in[dev].store(true, std::memory_order_release);
  }
  argus_prof_mark(ARGUS_PROF_OVERLAP, stream, 0);
  ARGUS_LAUNCH((k_ov_pair<DIGEST, NT, kGather>), a.blocks, NT, kPairSmem, stream, a);
  argus_prof_mark(ARGUS_PROF_OVERLAP, stream, 1);
  return ARGUS_OK;
}

// Threads of a block, and entries that a thread asks for at a time, by how many intervals an SM has on average: a block that has little
// to do waits at its barriers for the warps it has, one that has much to sort and walk needs them. How many intervals are spans
// of a pair, and whether they come in order, is not known here. us with 1,024 threads and two entries / 512 and four, intervals an SM:
// spans in order (one pair; 148 SMs): 2,300 18.5 / 16.2, 4,600 18.5 / 16.6, 11,600 21.0 / 18.5, 23,600 22.7 / 20.5, 34,800 35.6 / 35.7, 94,000
// 43.2 / 43.1; to be sorted (three pairs): 800 27.0 / 22.1, 2,500 30.8 / 24.7, 5,600 36.9 / 33.0, 16,000 57.4 / 57.3; (one pair, 16 CTAs
// an SM, whole call) 18,600 38.6 / 37.0, 37,000 55.9 / 58.6, 56,000 66.9 / 76.0, 111,000 177 / 195. From 2^17 on four entries with
// 1,024 threads: 232,000 113.5 / 108.8 (two / four). 256 threads were 1 us less than 512 for spans in order below 6,000 intervals
// an SM, but 40.3 where 5,600 had to be sorted, and twice the time where a call's CTAs lie on a few of the SMs that it names (37,000 on
// each of six of 148: 55.9, 58.6 with 512, 114.7 with 256).
template <bool DIGEST>
int launch_pair(const OvPairArgs& a, uint64_t num_intervals, cudaStream_t stream) {
  const u32 ctas = a.num_streams / a.warps_per_cta;  // each is on one SM
  const u64 sms = ctas < a.num_sms ? (ctas ? ctas : 1u) : a.num_sms, each = num_intervals / sms;
  return each < 1u << 15 ? launch_pair_as<DIGEST, 512, 4>(a, stream) : each < 1u << 17 ? launch_pair_as<DIGEST, 1024, 2>(a, stream) : launch_pair_as<DIGEST, 1024, 4>(a, stream);
}

}  // namespace

extern "C" size_t argus_overlap_workspace_bytes(uint64_t max_intervals, uint32_t num_streams, uint32_t num_pairs,
                                                uint32_t /*num_sms*/) {
  // worst case: every interval selected in both roles of every pair
  return ov_fixed_bytes(num_streams) + argus_align_up(((size_t)max_intervals * 2 * num_pairs + 64) * kBytesPerSpan, 256);
}

size_t argus_internal_overlap_bytes(uint64_t max_spans, uint32_t num_streams) {
  return ov_fixed_bytes(num_streams) + argus_align_up(((size_t)max_spans + 64) * kBytesPerSpan, 256);
}

static OvPairArgs pair_args(const argus_interval_t* intervals, const uint64_t* interval_offsets, const uint64_t* entries, uint64_t entry_capacity,
                            const ArgusOvPiece* pieces, uint32_t slices, uint32_t num_streams, uint32_t warps_per_cta, const uint32_t* cta_sm,
                            uint32_t num_sms, const uint32_t* pairs, uint32_t num_pairs, argus_overlap_t* out, argus_status_t* status,
                            ArgusOvCtl* ctl, void* spans, uint64_t max_spans) {
  OvPairArgs a;
  a.intervals = intervals; a.interval_offsets = (const u64*)interval_offsets; a.starts = nullptr; a.entries = (const u64*)entries; a.pieces = pieces;
  a.slices = slices; a.num_streams = num_streams; a.warps_per_cta = warps_per_cta; a.num_sms = num_sms; a.num_pairs = num_pairs;
  a.blocks = num_pairs * num_sms; a.cta_sm = cta_sm; a.pairs = pairs; a.out = out; a.status = status;
  a.spans = (ulonglong2*)spans; a.scratch = a.spans + max_spans; a.capacity = max_spans; a.entry_capacity = entry_capacity; a.ctl = ctl;
  return a;
}

// Overlap from what the pass over the digests selected: span area and scratch in `spans`.
int argus_internal_overlap_from_digests(const argus_interval_t* intervals, const uint64_t* starts, const uint64_t* entries, const ArgusOvPiece* pieces,
                                        uint32_t slices, uint32_t num_streams, uint32_t warps_per_cta, const uint32_t* cta_sm,
                                        uint32_t num_sms, const uint32_t* pairs, uint32_t num_pairs, argus_overlap_t* out,
                                        argus_status_t* status, ArgusOvCtl* ctl, void* spans, uint64_t max_spans, uint64_t num_intervals,
                                        void* cuda_stream) {
  OvPairArgs a = pair_args(intervals, nullptr, entries, ~0ull, pieces, slices, num_streams, warps_per_cta, cta_sm, num_sms, pairs, num_pairs,
                           out, status, ctl, spans, max_spans);
  a.starts = (const u64*)starts;
  return launch_pair<true>(a, num_intervals, (cudaStream_t)cuda_stream);
}

static int overlap_scoped(const argus_interval_t* intervals, uint64_t max_intervals, const uint64_t* interval_offsets,
                          uint32_t num_streams, uint32_t warps_per_cta, const uint32_t* cta_sm, uint32_t num_sms,
                          const uint32_t* pairs, uint32_t num_pairs, const argus_scope_t* scope, argus_overlap_t* out,
                          argus_status_t* status, void* workspace, size_t workspace_bytes, void* cuda_stream,
                          bool reset_status) {
  if (!interval_offsets || (!cta_sm && num_streams) || !status || !workspace) return ARGUS_ERR_INVALID_ARG;
  if (scope && scope->ctx_hi < scope->ctx_lo) return ARGUS_ERR_INVALID_ARG;
  if (warps_per_cta == 0 || num_streams % warps_per_cta != 0 || num_sms == 0) return ARGUS_ERR_INVALID_ARG;
  if (num_pairs > ARGUS_MAX_PAIRS || (num_pairs && (!pairs || !out))) return ARGUS_ERR_INVALID_ARG;
  if ((max_intervals && !intervals) || ((uintptr_t)intervals & 15) || ((uintptr_t)workspace & 255) || ((uintptr_t)out & 7))
    return ARGUS_ERR_INVALID_ARG;
  if ((uint64_t)num_pairs * num_sms * 2 > 0x7fffffffull) return ARGUS_ERR_INVALID_ARG;
  cudaStream_t stream = (cudaStream_t)cuda_stream;
  const size_t fixed = ov_fixed_bytes(num_streams);
  if (num_pairs && workspace_bytes < fixed) return ARGUS_ERR_WORKSPACE;
  if (reset_status || num_pairs) {
    const int rc = argus_internal_clear(reset_status ? status : nullptr, num_pairs ? workspace : nullptr, sizeof(ArgusOvCtl), cuda_stream);
    if (rc != ARGUS_OK) return rc;
  }
  if (num_pairs == 0) return ARGUS_OK;
  const u64 cap = (workspace_bytes - fixed) / kBytesPerSpan;
  const u32 slices = select_slices(num_streams), heads = num_streams * slices;
  // control block, spans, scratch, entries, pieces
  char* w = (char*)workspace;
  ArgusOvCtl* const ctl = (ArgusOvCtl*)w;
  w += argus_align_up(sizeof(ArgusOvCtl), 256);
  void* const spans = w;
  w += (size_t)cap * 32;
  uint64_t* const entries = (uint64_t*)w;
  w += argus_align_up((size_t)cap * 8, 16);
  ArgusOvPiece* const pieces = (ArgusOvPiece*)w;
  if (num_streams) {
    OvSelectArgs o;
    o.intervals = intervals; o.interval_offsets = (const u64*)interval_offsets; o.max_intervals = max_intervals;
    o.num_streams = num_streams; o.warps_per_cta = warps_per_cta; o.num_sms = num_sms; o.num_pairs = num_pairs;
    o.cta_sm = cta_sm; o.pairs = pairs; o.status = status; o.entries = (u64*)entries; o.entry_capacity = cap; o.pieces = pieces;
    // a piece beyond a slice's first one holds more than kSelStage - 32 entries or is the slice's last, so one for every 96
    // entries and one for every slice would do; the first ones are counted in the fixed part
    o.slices = slices; o.piece_capacity = heads + (u32)(cap / 16 < 0x7fffffffu ? cap / 16 : 0x7fffffffu); o.ctl = ctl;
    o.direct = max_intervals <= cap;
    o.scoped = scope != nullptr;
    o.ctx_lo = scope ? scope->ctx_lo : 0; o.ctx_hi = scope ? scope->ctx_hi : 0xffffffffu; o.warp_mask = scope ? scope->warp_mask : ~0ull;
    o.sm_mask = scope ? scope->sm_mask : nullptr; o.region_mask = scope ? scope->region_mask : nullptr;
    const u64 items = (u64)num_streams * (slices / kSelWarps);
    ARGUS_LAUNCH(k_ov_select, (unsigned)(items < kSelGrid ? items : kSelGrid), kSelThreads, 0, stream, o);
  }
  return launch_pair<false>(pair_args(intervals, interval_offsets, entries, cap, pieces, slices, num_streams, warps_per_cta, cta_sm, num_sms, pairs,
                                      num_pairs, out, status, ctl, spans, cap), max_intervals, stream);
}

int argus_internal_overlap(const argus_interval_t* intervals, uint64_t max_intervals, const uint64_t* interval_offsets,
                           uint32_t num_streams, uint32_t warps_per_cta, const uint32_t* cta_sm, uint32_t num_sms,
                           const uint32_t* pairs, uint32_t num_pairs, argus_overlap_t* out, argus_status_t* status,
                           void* workspace, size_t workspace_bytes, void* cuda_stream, bool reset_status) {
  return overlap_scoped(intervals, max_intervals, interval_offsets, num_streams, warps_per_cta, cta_sm, num_sms, pairs,
                        num_pairs, nullptr, out, status, workspace, workspace_bytes, cuda_stream, reset_status);
}

extern "C" int argus_overlap_scoped(const argus_interval_t* intervals, uint64_t max_intervals,
                                    const uint64_t* interval_offsets, uint32_t num_streams, uint32_t warps_per_cta,
                                    const uint32_t* cta_sm, uint32_t num_sms, const uint32_t* pairs, uint32_t num_pairs,
                                    const argus_scope_t* scope, argus_overlap_t* out, argus_status_t* status,
                                    void* workspace, size_t workspace_bytes, void* cuda_stream) {
  return overlap_scoped(intervals, max_intervals, interval_offsets, num_streams, warps_per_cta, cta_sm, num_sms, pairs,
                        num_pairs, scope, out, status, workspace, workspace_bytes, cuda_stream, true);
}

extern "C" int argus_overlap(const argus_interval_t* intervals, uint64_t max_intervals, const uint64_t* interval_offsets,
                             uint32_t num_streams, uint32_t warps_per_cta, const uint32_t* cta_sm, uint32_t num_sms,
                             const uint32_t* pairs, uint32_t num_pairs, argus_overlap_t* out, argus_status_t* status,
                             void* workspace, size_t workspace_bytes, void* cuda_stream) {
  return argus_internal_overlap(intervals, max_intervals, interval_offsets, num_streams, warps_per_cta, cta_sm, num_sms,
                                pairs, num_pairs, out, status, workspace, workspace_bytes, cuda_stream, true);
}
