// argus_pair.cu — argus_pair_intervals: marker events -> nested intervals + ambiguity records.
//
// Pipeline enqueued on the caller's stream (no host synchronisation):
//   init, order   : control block and event bitmap cleared; the count of every stream foretold, from its ends or, in a malformed
//                   trace, from all its markers, and from their sum the provisional base of its intervals; the order in which
//                   streams start
//   pair pass 1   : intervals written at the provisional bases; per-stream counts; ambiguity notes + bitmap bits
//   offsets       : scan of counts -> interval_offsets; sets `redo` when a count came out other than foretold;
//                   popcount prefix over the bitmap if there are notes
//   pair pass 2   : only does work when `redo` is set: rewrites the intervals of the streams behind at the final bases
//   ambiguity     : rank of every note in the bitmap -> ordered records, offsets
#include "argus_internal.cuh"
#include "argus_pair_common.cuh"

#include <string.h>

#include <atomic>

namespace {

constexpr int kScanThreads = 1024;
// Streams a thread of the one-block scans over all streams takes at a time: four where there are many (10^6 streams: 1,690 -> 1,325 us
// and 1,640 -> 860), one where a block holds them all (16 streams: a call of 45 us is 1 to 2 us longer with four).
constexpr u32 kScanRun = 4;
constexpr u32 kGroupWords = 8;                              // bitmap words of a prefix: 256 events, a sector, a thread's share
constexpr u32 kWordsPerBlock = kScanThreads * kGroupWords;  // and of a prefix block
std::atomic<u32> g_poll_limit{1u << 19};  // see argus_testing_set_poll_limit
std::atomic<u32> g_hand_on{0};            // see argus_testing_set_hand_overs

// ---------------------------------------------------------------------------------------------
// Reference-order kernel: one thread walks one stream with its stack in local memory.
// Exact for any input; used for small traces and as the arbiter the tiled kernel falls back to.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(128) k_pair_thread_per_stream(ArgusPairArgs a) {
  argus_kernel_begin_long();
  const u32 s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= a.num_streams) return;
  if (a.redo && !__ldcg(&a.ctl->redo)) return;
  const u64 off0 = a.stream_offsets[0];
  const u64 lo = a.stream_offsets[s], hi = a.stream_offsets[s + 1];
  if (hi < lo || hi > a.num_events || lo < off0 || (hi - lo) >> 32) {
    argus_set_error(a.status, ARGUS_ERR_BAD_OFFSETS, s, 0);
    if (!a.redo) a.counts[s] = 0;
    return;
  }
  const u64 base = a.redo ? a.interval_offsets[s] : a.bases[s];
  if (a.redo && s < __ldcg(&a.ctl->redo_from)) return;  // second pass: these intervals already lie where they belong
  ArgusFrame stk[ARGUS_MAX_DEPTH];
  ArgusSeqState st;
  st.h = 0; st.n_int = 0; st.n_ctx = st.n_rev = st.n_clamp = 0; st.failed = false;
  const u32 n = (u32)(hi - lo);
  const uint4* ev = reinterpret_cast<const uint4*>(a.events + lo);
  bool ok = true;
  for (u32 i = 0; i < n && ok; ++i) {
    const uint4 e = __ldg(ev + i);
    ok = argus_seq_step(a, stk, st, s, lo - off0, base, i, (u64)e.x | ((u64)e.y << 32), e.z, e.w);
  }
  if (ok) argus_seq_finish(a, stk, st, lo - off0);
  argus_flush_flag_counters(a, st);
  if (!a.redo) a.counts[s] = st.n_int;
}

// ---------------------------------------------------------------------------------------------
// Foretelling a stream's interval count. Intervals are written before anybody knows how many the streams before theirs
// hold, and a wrong guess costs the second pass. A stream whose markers nest has (events - unmatched ends - unmatched
// begins) / 2 intervals; unmatched ends lie at its front (a ring slot that has wrapped) and unmatched begins at its back (a
// stream that was cut short), so a look at both ends tells them. A stream that starts with begin(r) and stops with end(r) is
// taken to be whole. Otherwise, if its last marker is an end(b), b is taken to be an outermost region and the front is read
// until an unmatched end(b), which tells that the back is whole; if its first marker is a begin(a), the back is read until an
// unmatched begin(a), which tells that the front is whole; kGuessEvents at most. Both may be asked for: a stream whose ends are
// unclear is read from the back first, where a cut shows soon, others from the front.
// Unclear are begin(a) ... end(b): cut, or whole with several outermost regions. Where more than a quarter of the streams look
// like that they are taken to be whole but for a 32nd of their length at either end, and short ones are not read.
// (Pairing of traces cut at either end: 24 M events 551 -> 289 us, 142 M in a ring 2,700 -> 1,374 us; 262 and 1,215 with the
// pairing kernel of today. Streams of five outermost regions, one after the other: 8,000 of 4,000 events 775 us with a block for
// each stream and both ends of each read, 342 us, 402 without foretelling; 10^6 of 24 events 14,449, 6,110 and 6,473.)
// ---------------------------------------------------------------------------------------------
constexpr int kInitThreads = 256;
constexpr u32 kGuessEvents = 8192;

// Unmatched closing markers from one end of a stream on (FRONT: ends, from the first event; else begins, from the last
// backwards), up to and including the first one of region `outer` (*met: there is one), among `limit` events. One warp; a cut is
// usually near, so the first batch is small.
template <bool FRONT>
__device__ __noinline__ u32 guess_unmatched(const ArgusPairArgs& a, const uint4* src, u32 ring_first, u32 n, u32 outer, u32 limit, bool* met) {
  const u32 lane = threadIdx.x & 31;
  int height = 0, lowest = 0;  // uniform
  for (u32 i0 = 0, rows = 8; i0 < limit; i0 += rows * 32, rows = 32) {
    u32 opens = 0, closes = 0, outers = 0;  // bit j of lane l: event i0 + 32 l + j
#pragma unroll 16
    for (u32 r = 0; r < rows; ++r) {
      const u32 i = i0 + r * 32 + lane;
      const bool in = i < limit;
      u32 at = FRONT ? i : n - 1 - i;
      if (a.ring_written) { const u32 room = a.ring_capacity - ring_first; at = at >= room ? at - room : ring_first + at; }
      const u32 tag = in ? __ldg(reinterpret_cast<const u32*>(src + at) + 2) : 0u;
      const bool close = in && ((tag & 1u) != 0) == FRONT;
      const u32 c = __ballot_sync(0xffffffffu, close), o = __ballot_sync(0xffffffffu, close && (tag >> 1) == outer), have = __ballot_sync(0xffffffffu, in);
      if (lane == r) { closes = c; outers = o; opens = have & ~c; }
    }
    const int mine = __popc(opens) - __popc(closes);
    int upto = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) { const int o = __shfl_up_sync(0xffffffffu, upto, d); if (lane >= (u32)d) upto += o; }
    const int start = height + upto - mine;
    int h = start, low = start;  // the lowest height after any event of the lane
    for (u32 j = 0; j < 32; ++j) {
      h += (int)((opens >> j) & 1u) - (int)((closes >> j) & 1u);
      low = h < low ? h : low;
    }
    int before = low;  // and of the lanes before it
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) { const int o = __shfl_up_sync(0xffffffffu, before, d); if (lane >= (u32)d && o < before) before = o; }
    const int all = __shfl_sync(0xffffffffu, before, 31);
    before = __shfl_up_sync(0xffffffffu, before, 1);
    if (lane == 0 || before > lowest) before = lowest;
    u32 stop = 0xffffffffu;
    if (outers && low < before) {  // an unmatched one of `outer` may be here: the first event that goes below everything before it
      h = start;
      for (u32 j = 0; j < 32; ++j) {
        h += (int)((opens >> j) & 1u) - (int)((closes >> j) & 1u);
        if (h < before) {
          before = h;
          if ((outers >> j) & 1u) { stop = (u32)-h; break; }
        }
      }
    }
    stop = __reduce_min_sync(0xffffffffu, stop);  // (unmatched markers are counted one by one: the earliest stop is the one with the least depth)
    if (stop != 0xffffffffu) { *met = true; return stop; }
    lowest = all < lowest ? all : lowest;
    height += __shfl_sync(0xffffffffu, upto, 31);
  }
  *met = false;
  return (u32)-lowest;
}

// Clears the workspace's zeroed part and the status block.
__device__ __forceinline__ void pair_clear(const ArgusPairArgs& a, uint4* zeroed, u64 zeroed_words, int clear_status, u64 first, u64 stride) {
  for (u64 i = first; i < zeroed_words; i += stride) zeroed[i] = make_uint4(0, 0, 0, 0);
  if (clear_status && first < 8) reinterpret_cast<u64*>(a.status)[first] = 0;
}

__device__ __forceinline__ u32 stream_length(const ArgusPairArgs& a, u64 off0, u32 s) {
  const u64 lo = a.stream_offsets[s], hi = a.stream_offsets[s + 1];
  return hi < lo || hi > a.num_events || lo < off0 || ((hi - lo) >> 32) ? 0u : (u32)(hi - lo);  // (bad offsets are reported by the pairing kernel)
}

// First and last marker's tag of a stream; false when it is empty.
__device__ __forceinline__ bool stream_ends(const ArgusPairArgs& a, u32 s, u32 n, u32* first, u32* last) {
  if (!n) return false;
  const u32 head = a.ring_written ? argus_ring_first(a, s) : 0u;
  const uint4* src = reinterpret_cast<const uint4*>(a.events) + (a.ring_written ? (u64)s * a.ring_capacity : a.stream_offsets[s]);
  u32 end = n - 1;
  if (a.ring_written) { const u32 room = a.ring_capacity - head; end = end >= room ? end - room : head + end; }
  *first = __ldg(reinterpret_cast<const u32*>(src + head) + 2);
  *last = __ldg(reinterpret_cast<const u32*>(src + end) + 2);
  return true;
}
// begin(a) ... end(b), and not a ring slot that has wrapped
__device__ __forceinline__ bool ends_unclear(const ArgusPairArgs& a, u32 s, u32 first, u32 last) {
  return !(first & 1u) && (last & 1u) && (first >> 1) != (last >> 1) && !(a.ring_written && a.ring_written[s] > a.ring_capacity);
}

// A lost or doubled marker inside a stream shows at neither end. Windows of 128 markers all over the trace are looked at: where an
// end meets, 32 markers at a time, a begin of another region one below it in height, its stream is malformed, and the counts of all
// streams may be taken from all their markers (recount) instead of from their ends. Seven defects in 10,000 markers show in
// dozens of the 1,024 windows; a window of a sound trace never tells one. (GEMM trace with that many, 68 M events: 2,263 -> 1,512 us a
// call, 944 us of a second pass for 208 us of counting.) The look costs a sound trace about 2 us. Smaller calls do not look, because
// sound ones would be longer by more than a thirtieth: pairing of 1.06, 2.1 and 4.1 M sound events takes 33, 43 and 62 us (with seven
// lost ends in 10,000 markers, and so a second pass, 124, 148 and 246).
// Counting goes by heights, which lost ends and doubled begins raise for good, and lost begins and doubled ends lower; of either
// alone it is exact. A marker of which the region has changed leaves the heights as they are but takes its interval away, and of both kinds
// together one hides the other: counts are then wrong and the second pass comes all the same (68.7 M events, seven in 10,000 ends changed:
// 2,598 us; counting would add its 205). So a window also tells what kind it has met.
constexpr u32 kSamples = 1024;  // as many as k_pair_order has threads
constexpr u32 kSampleRows = 4;
constexpr u64 kSampledEvents = 1ull << 22;
enum : u32 { kNoDefect = 0, kUnclear = 1, kChanged = 2, kLowered = 3, kRaised = 4 };
__device__ __forceinline__ u32 sample_stream(const ArgusPairArgs& a, u32 w) { return (u32)(((u64)w * a.num_streams) / kSamples); }
// What kind of defect a row of 32 markers holds, given which of its ends (`bad`) meet the begin of another region. One warp.
__device__ __noinline__ u32 sample_kind(u32 bad, u32 ends, u32 tag, u32 begin, int level) {
  u32 kind = kUnclear, passed = 0xffffffffu;  // region of the last begin that was met by another region's end
  const u32 region = tag >> 1;
  for (; bad; bad &= bad - 1) {
    const int i = __ffs((int)bad) - 1;
    const u32 closing = __shfl_sync(0xffffffffu, region, i), met = __shfl_sync(0xffffffffu, begin >> 1, i);
    const u32 around = __ballot_sync(0xffffffffu, level == __shfl_sync(0xffffffffu, level, i) - 1);
    const u32 earlier = around & ((1u << i) - 1u), later = around & ends & ~((2u << i) - 1u);
    // the begin of the frame around, and the end that closes it
    const u32 outer = __shfl_sync(0xffffffffu, region, earlier ? 31 - __clz((int)earlier) : 0), next = __shfl_sync(0xffffffffu, region, later ? __ffs((int)later) - 1 : 0);
    const u32 k = closing == passed ? kLowered                    // the frame that the last such end has passed over
                  : earlier && closing == outer ? kRaised         // the frame met here is closed along with the one around it
                  : later && next == met ? kLowered
                  : earlier && later && next == outer ? kChanged  // as if this end were the right one
                                                      : kUnclear;
    kind = k > kind ? k : kind;
    passed = met;
  }
  return kind;
}
// The tags of window `w`; false where its stream is too short. One warp.
__device__ __forceinline__ bool sample_load(const ArgusPairArgs& a, u64 off0, u32 w, u32 (&tags)[kSampleRows]) {
  const u32 lane = threadIdx.x & 31, s = sample_stream(a, w), n = stream_length(a, off0, s);
  if (n < 32 * kSampleRows) return false;
  const u32 head = a.ring_written ? argus_ring_first(a, s) : 0u, at0 = __umulhi(w * 0x9E3779B1u, n - 32 * kSampleRows + 1);
  const uint4* const src = reinterpret_cast<const uint4*>(a.events) + (a.ring_written ? (u64)s * a.ring_capacity : a.stream_offsets[s]);
#pragma unroll
  for (u32 r = 0; r < kSampleRows; ++r) {
    u32 at = at0 + 32 * r + lane;
    if (a.ring_written) { const u32 room = a.ring_capacity - head; at = at >= room ? at - room : head + at; }
    tags[r] = __ldg(reinterpret_cast<const u32*>(src + at) + 2);
  }
  return true;
}
// What they tell. One warp.
__device__ __forceinline__ u32 sample_tell(const u32 (&tags)[kSampleRows]) {
  const u32 lane = threadIdx.x & 31, lower = (1u << lane) - 1u;
  u32 kind = kNoDefect;
#pragma unroll
  for (u32 r = 0; r < kSampleRows; ++r) {
    const bool is_end = tags[r] & 1u;
    const u32 ends = __ballot_sync(0xffffffffu, is_end);
    const int level = (int)lane - 2 * __popc(ends & lower) - (int)is_end;  // of the frame it opens or closes
    const u32 before = __match_any_sync(0xffffffffu, level) & lower;         // (the last of them opened the frame that an end closes)
    const u32 begin = __shfl_sync(0xffffffffu, tags[r], before ? 31 - __clz((int)before) : 0);
    const u32 bad = __ballot_sync(0xffffffffu, is_end && before && (begin ^ tags[r]) != 1u);
    if (bad) {
      const u32 k = sample_kind(bad, ends, tags[r], begin, level);
      kind = k > kind ? k : kind;
    }
  }
  return kind;
}

// A warp takes `per` streams at a time: their first and last markers, a lane each, then a look at those that are not whole.
// `samples` (nullable): what the windows tell.
__global__ void __launch_bounds__(kInitThreads) k_pair_init(ArgusPairArgs a, uint4* zeroed, u64 zeroed_words, int clear_status, u32 per, u32* samples) {
  argus_kernel_begin();
  pair_clear(a, zeroed, zeroed_words, clear_status, (u64)blockIdx.x * blockDim.x + threadIdx.x, (u64)gridDim.x * blockDim.x);
  const u32 lane = threadIdx.x & 31;
  const u64 off0 = a.num_streams ? a.stream_offsets[0] : 0, warps = (u64)gridDim.x * (kInitThreads / 32);
  // the tags of the warp's first window are on their way while it takes its streams (there are mostly no more windows than warps)
  u32 window = samples && a.num_streams ? blockIdx.x * (kInitThreads / 32) + (threadIdx.x >> 5) : kSamples, tags[kSampleRows];
  bool looked = window < kSamples && sample_load(a, off0, window, tags);
  int many = -1;  // whether more than a quarter of the streams have unclear ends (a sample of 32 tells, when it is asked for)
  for (u64 s0 = ((u64)blockIdx.x * (kInitThreads / 32) + (threadIdx.x >> 5)) * per; s0 < a.num_streams; s0 += warps * per) {
    u32 n = 0, f = 0, l = 1;
    if (lane < per && s0 + lane < a.num_streams) {
      const u32 sm = (u32)(s0 + lane);
      n = stream_length(a, off0, sm);
      a.bases[sm] = n >> 1;
      stream_ends(a, sm, n, &f, &l);
    }
    for (u32 todo = __ballot_sync(0xffffffffu, n && ((f & 1u) || !(l & 1u) || (f >> 1) != (l >> 1))); todo; todo &= todo - 1) {
      const int k = __ffs((int)todo) - 1;
      const u32 s = (u32)s0 + k, nk = __shfl_sync(0xffffffffu, n, k), fk = __shfl_sync(0xffffffffu, f, k), lk = __shfl_sync(0xffffffffu, l, k);
      u32 limit = nk < kGuessEvents ? nk : kGuessEvents;
      const bool unclear = ends_unclear(a, s, fk, lk);
      if (unclear) {
        if (many < 0) {
          const u32 si = (u32)((u64)lane * a.num_streams / 32);
          u32 fi = 0, li = 0;
          many = __popc(__ballot_sync(0xffffffffu, stream_ends(a, si, stream_length(a, off0, si), &fi, &li) && ends_unclear(a, si, fi, li))) > 8;
        }
        if (many && nk / 32 < limit) limit = nk / 32;
        if (many && limit < 32) continue;
      }
      const u32 head = a.ring_written ? argus_ring_first(a, s) : 0u;
      const uint4* src = reinterpret_cast<const uint4*>(a.events) + (a.ring_written ? (u64)s * a.ring_capacity : a.stream_offsets[s]);
      bool met = false;
      u32 unmatched = 0;
      if (unclear) {
        unmatched = guess_unmatched<false>(a, src, head, nk, fk >> 1, limit, &met);
        if (!met) unmatched += guess_unmatched<true>(a, src, head, nk, lk >> 1, limit, &met);
      } else {
        if (lk & 1u) unmatched = guess_unmatched<true>(a, src, head, nk, lk >> 1, limit, &met);
        if (!met && !(fk & 1u)) unmatched += guess_unmatched<false>(a, src, head, nk, fk >> 1, limit, &met);
      }
      if (lane == 0) a.bases[s] = (nk - (unmatched < nk ? unmatched : nk)) >> 1;
    }
  }
  while (window < kSamples) {
    const u32 told = looked ? sample_tell(tags) : kNoDefect;
    if (lane == 0) samples[window] = told;
    window += (u32)warps;
    looked = window < kSamples && sample_load(a, off0, window, tags);
  }
}

// ---------------------------------------------------------------------------------------------
// order: provisional bases (exclusive sum of the foretold counts), and the streams sorted by length class
// (an eighth of an octave), longest first. A stream is a chain of tiles that one CTA at a time walks, so when lengths differ
// (producer and consumer warps of one kernel) the long chains must start first or they end last, alone. Counting sort in one
// block; the order inside a class does not matter. Small calls have no init kernel before this one (`alone`).
// ---------------------------------------------------------------------------------------------
constexpr u32 kClasses = 256;
__device__ __forceinline__ u32 length_class(u32 n) {  // 8 floor(log2(n)) and three more bits of n
  if (!n) return 0;
  const u32 e = 31 - (u32)__clz((int)n);
  return e * 8 + (e >= 3 ? (n >> (e - 3)) & 7u : (n << (3 - e)) & 7u);
}
// Returns the sum of the foretold counts; *longest: events of the longest stream of this thread.
template <u32 RUN>
__device__ __forceinline__ u64 order_bases(const ArgusPairArgs& a, u64 off0, int alone, u32* cnt, u64 (&sh)[33], u32* longest) {
  u64 carry = 0;
  for (u64 s0 = 0; s0 < a.num_streams; s0 += kScanThreads * RUN) {
    const u64 s = s0 + threadIdx.x * RUN;
    u64 c[RUN], sum = 0, total;
#pragma unroll
    for (u32 j = 0; j < RUN; ++j) {
      u32 cls = kClasses;
      c[j] = 0;
      if (s + j < a.num_streams) {
        const u32 n = stream_length(a, off0, (u32)s + j);
        c[j] = alone ? n >> 1 : __ldcg(a.bases + s + j);
        cls = length_class(n);
        *longest = n > *longest ? n : *longest;
        if (RUN == 1) atomicAdd(&cnt[cls], 1u);
      }
      sum += c[j];
      if (RUN > 1) {
        const u32 same = __match_any_sync(0xffffffffu, cls);  // a warp's streams are mostly of one class
        if (cls < kClasses && !(same & ((1u << (threadIdx.x & 31)) - 1u))) atomicAdd(&cnt[cls], (u32)__popc(same));
      }
    }
    u64 at = carry + argus_block_exclusive_scan<u64>(sum, sh, &total);
#pragma unroll
    for (u32 j = 0; j < RUN; ++j) {
      if (s + j < a.num_streams) a.bases[s + j] = at;
      at += c[j];
    }
    carry += total;
  }
  return carry;
}

// The intervals of stream s as far as its markers' heights tell: ends less those that come below every height before them. One block.
__device__ __forceinline__ u32 recount_stream(const ArgusPairArgs& a, u64 off0, u32 s, int (&shi)[33], u32* shu) {
  static_assert(kRecountStep == kScanThreads * 32, "32 markers in a row a thread");
  const u32 tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n = stream_length(a, off0, s);
  const u32 head = a.ring_written ? argus_ring_first(a, s) : 0u, room = a.ring_capacity - head;
  const uint4* const src = reinterpret_cast<const uint4*>(a.events) + (a.ring_written ? (u64)s * a.ring_capacity : a.stream_offsets[s]);
  long long height = 0, lowest = 0;
  u32 all_ends = 0;
  for (u32 round = 0, rounds = argus_recount_rounds(n); round < rounds; ++round) {  // rows of 32 are read by a warp, 32 at a time
    const u32 have = argus_recount_markers(n, round), i0 = round * kRecountStep;
    u32 ends = 0;
#pragma unroll 16
    for (u32 r = 0; r < 32; ++r) {
      const u32 j = warp * 1024 + r * 32 + lane;
      u32 at = i0 + j;
      if (a.ring_written) at = at >= room ? at - room : head + at;
      const u32 tag = j < have ? __ldg(reinterpret_cast<const u32*>(src + at) + 2) : 0u;
      const u32 b = __ballot_sync(0xffffffffu, tag & 1u);
      if (lane == r) ends = b;
    }
    const u32 mine = tid * 32 >= have ? 0u : have - tid * 32 < 32 ? have - tid * 32 : 32u;
    const u32 begins = mine ? ~ends & (0xffffffffu >> (32 - mine)) : 0u;
    int total;
    int h = argus_block_exclusive_scan<int>(__popc(begins) - __popc(ends), shi, &total), low = 0;  // (from the round's first marker on)
#pragma unroll
    for (u32 r = 0; r < 32; ++r) {
      h += (int)((begins >> r) & 1u) - (int)((ends >> r) & 1u);
      low = h < low ? h : low;
    }
    lowest = height + low < lowest ? height + low : lowest;
    all_ends += __popc(ends);
    height += total;
  }
  const u32 below = __reduce_max_sync(0xffffffffu, (u32)-lowest);
  all_ends = __reduce_add_sync(0xffffffffu, all_ends);
  if (tid < 2) shu[tid] = 0;
  __syncthreads();
  if (lane == 0) { atomicMax(&shu[0], below); atomicAdd(&shu[1], all_ends); }
  __syncthreads();
  const u32 count = shu[1] - shu[0];
  __syncthreads();
  return count;
}

// Whether counting all markers pays: what it costs against a second pass over the streams behind `first_bad`, the first one that
// is known to be malformed. Both go at the chip's rate (68.6 M events of 1,776 streams: 205 us of counting, 940 of a second pass) or
// at a block's over the longest stream (96 streams of 405,000: 137 us, 2,150). Lost ends in the last half, fifth and tenth of the
// streams of the former: 1,428 -> 956 us, 1,343 -> 961 and, not counted, 1,201 -> 1,209; in all of the latter 4,648 -> 2,478. One block.
__device__ __forceinline__ bool recount_pays(const ArgusPairArgs& a, u32 first_bad, u32* longest /* [2] */) {
  const u64 off0 = a.stream_offsets[0];
  u32 all = 0, behind = 0;
  for (u32 s = threadIdx.x; s < a.num_streams; s += kScanThreads) {
    const u32 n = stream_length(a, off0, s);
    all = n > all ? n : all;
    if (s > first_bad) behind = n > behind ? n : behind;
  }
  if (threadIdx.x < 2) longest[threadIdx.x] = 0;
  __syncthreads();
  atomicMax(&longest[0], all);
  atomicMax(&longest[1], behind);
  __syncthreads();
  const u64 end = a.stream_offsets[a.num_streams], total = end - off0, left = end - a.stream_offsets[first_bad + 1];
  const u64 count = total * 3 > longest[0] * 340ull ? total * 3 : longest[0] * 340ull;      // ps, by 3 an event or 340 of the longest
  const u64 again = left * 14 > longest[1] * 4050ull ? left * 14 : longest[1] * 4050ull;  // by 14, or 4,050
  return count < again;
}

// `samples` (nullable): what the windows that k_pair_init has looked at tell. One block orders; where the trace is malformed in a way
// that counting its markers tells how many intervals it has (windows of one kind, and more than one: a single defect that a window
// happens to meet is no reason to read everything; 1.2 G markers with one corrupted end at the front 24.5 ms counted, 21.6 not), and
// counting costs less than the second pass, the whole grid counts before the last block orders.
template <u32 RUN>
__global__ void __launch_bounds__(kScanThreads, 1) k_pair_order(ArgusPairArgs a, u32* order, uint4* zeroed, u64 zeroed_words,
                                                            int clear_status, int alone, int ask_split, const u32* samples) {
  argus_kernel_begin_long();  // the pairing kernel's blocks spread evenly only over SMs that are free when they come
  __shared__ u32 cnt[kClasses], cur[kClasses];
  __shared__ u64 sh[33];
  __shared__ u32 one_class, longest_of, first_bad;
  u32 told = kNoDefect;
  if (samples) {
    static_assert(kSamples == kScanThreads, "a window a thread");
    told = samples[threadIdx.x];
    if (blockIdx.x == 0 && threadIdx.x * RUN < a.num_streams) {  // (what comes next, asked for at the same time)
      asm volatile("prefetch.global.L1 [%0];" ::"l"(a.stream_offsets + threadIdx.x * RUN));
      asm volatile("prefetch.global.L2 [%0];" ::"l"(a.bases + threadIdx.x * RUN));
    }
    bool counted = __syncthreads_count(told != kNoDefect) > 1;
    if (counted) {
      const int raised = __syncthreads_count(told == kRaised), lowered = __syncthreads_count(told == kLowered);
      if (threadIdx.x == 0) first_bad = 0xffffffffu;
      counted = __syncthreads_or(told == kChanged) == 0 && (raised == 0 || lowered == 0) && raised + lowered > 1;
      if (counted) {
        if (told) atomicMin(&first_bad, sample_stream(a, threadIdx.x));
        __syncthreads();
        counted = recount_pays(a, first_bad, cur);
      }
    }
    if (counted) {
      __shared__ int shi[33];
      __shared__ u32 next;
      const u64 off = a.stream_offsets[0];
      for (;;) {
        if (threadIdx.x == 0) next = atomicAdd(&a.ctl->recount_head, 1u);
        __syncthreads();
        const u32 s = next;
        __syncthreads();
        if (s >= a.num_streams) break;
        const u32 count = recount_stream(a, off, s, shi, cnt);
        if (threadIdx.x == 0) a.bases[s] = count;
      }
      if (threadIdx.x == 0) {
        __threadfence();
        next = atomicAdd(&a.ctl->recount_done, 1u);
      }
      __syncthreads();
      if (next != gridDim.x - 1) return;
      __threadfence();
    } else if (blockIdx.x) {
      return;
    }
  }
  if (threadIdx.x == 0) longest_of = 0;
  if (alone) pair_clear(a, zeroed, zeroed_words, clear_status, threadIdx.x, blockDim.x);
  if (threadIdx.x < kClasses) { cnt[threadIdx.x] = 0; cur[threadIdx.x] = 0; }
  if (threadIdx.x == 0) one_class = 0;
  __syncthreads();
  const u64 off0 = a.num_streams ? a.stream_offsets[0] : 0;
  u32 longest = 0;
  const u64 carry = order_bases<RUN>(a, off0, alone, cnt, sh, &longest);
  if (ask_split) {
    longest = __reduce_max_sync(0xffffffffu, longest);
    if ((threadIdx.x & 31) == 0) atomicMax(&longest_of, longest);
  }
  __syncthreads();
  // a malformed stream that the split pass would give up together with all others
  const bool in_vain = ask_split && __syncthreads_or(told && !argus_split_pays(longest_of - stream_length(a, off0, sample_stream(a, threadIdx.x)), a.num_events, a.num_streams));
  if (threadIdx.x == 0) {
    a.bases[a.num_streams] = carry;
    if (ask_split) { a.ctl->split = !in_vain && argus_split_pays(longest_of, a.num_events, a.num_streams); a.ctl->longest = longest_of; }
  }
  if (threadIdx.x < 32) {  // first places, classes in descending order
    u32 k[kClasses / 32], sum = 0;
#pragma unroll
    for (u32 j = 0; j < kClasses / 32; ++j) {
      k[j] = cnt[kClasses - 1 - (threadIdx.x * (kClasses / 32) + j)];
      sum += k[j];
      if (k[j] == a.num_streams) one_class = 1;
    }
    u32 place = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) { const u32 o = __shfl_up_sync(0xffffffffu, place, d); if (threadIdx.x >= (u32)d) place += o; }
    place -= sum;
#pragma unroll
    for (u32 j = 0; j < kClasses / 32; ++j) { cnt[kClasses - 1 - (threadIdx.x * (kClasses / 32) + j)] = place; place += k[j]; }
  }
  __syncthreads();
  if (one_class) {  // streams of one length class start in index order, as without this kernel
    for (u32 s = threadIdx.x; s < a.num_streams; s += blockDim.x) order[s] = s;
    return;
  }
  for (u32 s = threadIdx.x; s < a.num_streams; s += blockDim.x) {
    const u32 c = length_class(stream_length(a, off0, s));
    order[cnt[c] + atomicAdd(&cur[c], 1u)] = s;
  }
}

// ---------------------------------------------------------------------------------------------
// ambiguity ordering
// ---------------------------------------------------------------------------------------------
struct AmbigArgs {
  ArgusPairArgs p;
  u64 num_words;     // bitmap words covering [0, span) event positions
  u64 span;          // stream_offsets[S] - stream_offsets[0] is <= num_events; bitmap covers num_events
  u32* group_prefix; // per group of words: set bits before it within its block
  u64* block_prefix; // per block: set bits before it (after the scan); [num_blocks + 1]
  u64 num_blocks;
  argus_ambiguity_t* ambig;
  u64 ambig_capacity;
  u64* ambig_offsets;
};

// interval_offsets; returns the sum of the counts. *bad: first stream that does not lie right, *used: last one that has any.
template <u32 RUN>
__device__ __forceinline__ u64 final_offsets(const ArgusPairArgs& a, u64 (&sh)[33], u32* bad, u32* used) {
  u64 carry = 0;
  for (u64 s0 = 0; s0 < a.num_streams; s0 += kScanThreads * RUN) {
    const u64 s = s0 + threadIdx.x * RUN;
    u64 c[RUN], sum = 0, total;
#pragma unroll
    for (u32 j = 0; j < RUN; ++j) { c[j] = s + j < a.num_streams ? a.counts[s + j] : 0; sum += c[j]; }
    u64 fin = carry + argus_block_exclusive_scan<u64>(sum, sh, &total);
    u64 base = s < a.num_streams ? a.bases[s] : 0;
#pragma unroll
    for (u32 j = 0; j < RUN; ++j) {
      if (s + j >= a.num_streams) break;
      const u32 sj = (u32)s + j;
      // (beyond the capacity only when the call ends with ARGUS_ERR_CAPACITY: offsets then stay inside the array, so
      // that a call chained behind this one without a host check reads nothing it must not)
      a.interval_offsets[sj] = fin < a.interval_capacity ? fin : a.interval_capacity;
      const u64 next = a.bases[s + j + 1], told = next - base;
      // a stream with fewer intervals than foretold lies right, those after it do not; one with more has lost its tail to the
      // next stream's writes
      if (c[j] < told && sj + 1 < *bad) *bad = sj + 1;
      if (c[j] > told && sj < *bad) *bad = sj;
      if (c[j]) *used = sj;
      fin += c[j];
      base = next;
    }
    carry += total;
  }
  return carry;
}

// Block 0: exclusive scan of the per-stream counts; decides whether the second pass is needed, and from which stream on.
template <u32 RUN>
__device__ __forceinline__ void pair_offsets(const ArgusPairArgs& a) {
  __shared__ u64 sh[33];
  __shared__ u32 first_bad, last_used;
  if (threadIdx.x == 0) { first_bad = 0xffffffffu; last_used = 0; }
  __syncthreads();
  u32 bad = 0xffffffffu, used = 0;
  const u64 carry = final_offsets<RUN>(a, sh, &bad, &used);
  atomicMin(&first_bad, bad);
  atomicMax(&last_used, used);
  __syncthreads();
  if (threadIdx.x == 0) {
    a.interval_offsets[a.num_streams] = carry < a.interval_capacity ? carry : a.interval_capacity;
    a.ctl->total_intervals = carry;
    a.status->intervals_required = carry;
    a.ctl->redo_from = first_bad;
    if (carry > a.interval_capacity) {
      argus_set_error(a.status, ARGUS_ERR_CAPACITY, 0, carry);
      a.ctl->redo = 0;
    } else {
      a.ctl->redo = carry && first_bad <= last_used ? 1u : 0u;
    }
  }
}

// The other blocks, when there are notes: set bits before every group of words within its block of words, and, by the last block to
// be done, before every block of words. (142 M events with a prefix for every word 46 us, 12 so.)
template <u32 RUN>
__global__ void __launch_bounds__(kScanThreads) k_pair_offsets(AmbigArgs g) {
  // The second pass comes next, and its blocks spread evenly only over SMs that are free when they come (96 streams with a lost end
  // each: 5,993 us when they came beside this kernel's blocks, 4,111 us after them). Not so where there are enough of them to fill the
  // chip or few blocks here (up to 9.4 M events: 96 to 960 streams of 1.3, 4 and 8.5 M, whole malformed calls, early / late 450 / 450, 563 / 559
  // and 531 / 530 us at worst); and without notes it has nothing to do (coming early saves 0.5 us of the smallest call, 2 us of others).
  const bool early = gridDim.x <= 37 || g.p.num_streams >= 1036;
  if (early) argus_launch_next();
  argus_kernel_begin_long();
  if (!early && __ldcg(&g.p.ctl->n_notes) == 0) argus_launch_next();
  if (blockIdx.x == 0) { pair_offsets<RUN>(g.p); return; }
  if (__ldcg(&g.p.ctl->n_notes) == 0) return;
  __shared__ u32 sh[33];
  __shared__ u64 sh64[33];
  __shared__ u32 last;
  for (u64 blk = blockIdx.x - 1; blk < g.num_blocks; blk += gridDim.x - 1) {
    const u64 w = blk * kWordsPerBlock + threadIdx.x * kGroupWords;
    u32 c = 0;
    if (w < g.num_words) {  // (the last group is filled up with words that are zero)
      const uint4 x = *reinterpret_cast<const uint4*>(g.p.bits + w), y = *reinterpret_cast<const uint4*>(g.p.bits + w + 4);
      c = __popc(x.x) + __popc(x.y) + __popc(x.z) + __popc(x.w) + __popc(y.x) + __popc(y.y) + __popc(y.z) + __popc(y.w);
    }
    u32 total;
    const u32 ex = argus_block_exclusive_scan<u32>(c, sh, &total);
    if (w < g.num_words) g.group_prefix[w / kGroupWords] = ex;
    if (threadIdx.x == 0) g.block_prefix[blk] = total;
    __syncthreads();
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&g.p.ctl->prefix_done, 1u) == gridDim.x - 2;
  __syncthreads();
  if (!last) return;
  __threadfence();
  u64 carry = 0;
  for (u64 b0 = 0; b0 < g.num_blocks; b0 += kScanThreads) {
    const u64 b = b0 + threadIdx.x;
    const u64 c = b < g.num_blocks ? __ldcg(g.block_prefix + b) : 0;
    u64 total;
    const u64 ex = argus_block_exclusive_scan<u64>(c, sh64, &total);
    if (b < g.num_blocks) g.block_prefix[b] = carry + ex;
    carry += total;
  }
  if (threadIdx.x == 0) {
    g.block_prefix[g.num_blocks] = carry;
    g.p.ctl->total_ambig = carry;
    g.p.status->ambig_required = carry;
    if (carry > g.ambig_capacity || g.p.ctl->n_notes > g.p.note_capacity)
      argus_set_error(g.p.status, ARGUS_ERR_CAPACITY, 0, carry);
  }
}

// number of ambiguous markers at global positions < gpos
__device__ __forceinline__ u64 ambig_rank(const AmbigArgs& g, u64 gpos) {
  const u64 w = gpos >> 5;
  if (w >= g.num_words) return g.block_prefix[g.num_blocks];
  const uint4* const group = reinterpret_cast<const uint4*>(g.p.bits + w / kGroupWords * kGroupWords);
  const uint4 a = group[0], b = group[1];
  const u32 v[kGroupWords] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w}, k = (u32)w % kGroupWords;
  u32 c = 0;
#pragma unroll
  for (u32 q = 0; q < kGroupWords; ++q) c += q < k ? __popc(v[q]) : q == k ? __popc(v[q] & ((1u << (gpos & 31)) - 1u)) : 0;
  return g.block_prefix[w / kWordsPerBlock] + g.group_prefix[w / kGroupWords] + c;
}

__device__ __forceinline__ void ambig_offset(const AmbigArgs& g, u64 s) {
  if (__ldcg(&g.p.ctl->n_notes) == 0) { g.ambig_offsets[s] = 0; return; }
  const u64 off0 = g.p.num_streams ? g.p.stream_offsets[0] : 0;
  const u64 o = g.p.num_streams ? g.p.stream_offsets[s] : 0;
  const u64 r = o >= off0 ? ambig_rank(g, o - off0) : 0;
  g.ambig_offsets[s] = r < g.ambig_capacity ? r : g.ambig_capacity;  // inside the array also after ARGUS_ERR_CAPACITY
}

// ambig_offsets, and the notes as records in order
__global__ void __launch_bounds__(256) k_ambig_records(AmbigArgs g) {
  argus_kernel_begin_long();  // (a long kernel's blocks come next, as after k_pair_order)
  for (u64 s = (u64)blockIdx.x * blockDim.x + threadIdx.x; s <= g.p.num_streams; s += (u64)gridDim.x * blockDim.x) ambig_offset(g, s);
  const u64 n_notes = __ldcg(&g.p.ctl->n_notes);
  const u64 n = n_notes < g.p.note_capacity ? n_notes : g.p.note_capacity;
  const u64 off0 = n ? g.p.stream_offsets[0] : 0;
  for (u64 j = (u64)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (u64)gridDim.x * blockDim.x) {
    const u64 note = g.p.notes[j];
    const u64 gpos = note & ((1ull << ARGUS_NOTE_POS_BITS) - 1);
    const u64 r = ambig_rank(g, gpos);
    if (r >= g.ambig_capacity) continue;
    const u64 x = off0 + gpos;  // index into events
    // stream = last s with stream_offsets[s] <= x (empty streams skipped by taking the upper bound)
    u32 lo = 0, hi = g.p.num_streams;
    while (hi - lo > 1) {
      const u32 mid = lo + ((hi - lo) >> 1);
      if (g.p.stream_offsets[mid] <= x) lo = mid; else hi = mid;
    }
    u64 at = x;  // where the record lies: packed input, or its slot position in a ring container
    if (g.p.ring_written) {
      u64 pos = argus_ring_first(g.p, lo) + (x - g.p.stream_offsets[lo]);
      if (pos >= g.p.ring_capacity) pos -= g.p.ring_capacity;
      at = (u64)lo * g.p.ring_capacity + pos;
    }
    const argus_event_t e = g.p.events[at];
    argus_ambiguity_t rec;
    rec.ts = e.ts; rec.tag = e.tag; rec.ctx = e.ctx; rec.stream = lo;
    rec.event_idx = (u32)(x - g.p.stream_offsets[lo]);
    rec.kind = (u32)(note >> ARGUS_NOTE_POS_BITS) & 3u;
    rec.depth = (u32)(note >> (ARGUS_NOTE_POS_BITS + 2)) & 0x7fu;
    g.ambig[r] = rec;
  }
}

struct Layout {
  size_t ctl, counts, queue, bits, group_prefix, block_prefix, notes, records, order, bases, split, total;
  u64 num_words, num_blocks, queue_capacity;
  u32 record_capacity;
};

Layout make_layout(uint64_t num_events, uint32_t num_streams, uint64_t ambig_capacity) {
  Layout L;
  L.num_words = (num_events + 31) / 32;
  L.num_blocks = (L.num_words + kWordsPerBlock - 1) / kWordsPerBlock;
  size_t o = 0;
  L.ctl = o; o += argus_align_up(sizeof(ArgusPairCtl), 256);
  L.counts = o; o += argus_align_up(((size_t)num_streams + 1) * 8, 256);
  // every hand-over follows a chunk of at least kChunkEvents events, and only streams longer than that hand over (in small calls, for
  // which the static entry has little scratch, the longest of them)
  L.queue_capacity = num_events / kChunkEvents + 1;
  const u64 records = num_events > 1u << 20 ? L.queue_capacity : num_events / 32768 + 1;
  L.record_capacity = (u32)(records < num_streams ? records : num_streams);
  L.queue = o; o += argus_align_up((size_t)L.queue_capacity * 4, 256);
  L.bits = o; o += argus_align_up((size_t)L.num_words * 4 + 4, 256);  // (whole groups)
  static_assert(256 % (kGroupWords * 4) == 0, "whole groups");
  L.group_prefix = o; o += argus_align_up((size_t)(L.num_words + kGroupWords - 1) / kGroupWords * 4 + 4, 256);
  L.block_prefix = o; o += argus_align_up(((size_t)L.num_blocks + 1) * 8, 256);
  L.notes = o; o += argus_align_up((size_t)ambig_capacity * 8 + 8, 256);
  L.records = o; o += argus_align_up((size_t)L.record_capacity * sizeof(ArgusStreamRecord), 256);
  L.order = o; o += argus_align_up((size_t)num_streams * 4 + 4, 256);
  L.bases = o; o += argus_align_up(((size_t)num_streams + 1) * 8, 256);
  L.split = o; o += argus_split_bytes(num_events, num_streams);
  L.total = o;
  return L;
}

}  // namespace

// implemented in argus_pair_tiled.cu
int argus_launch_pair_tiled(const ArgusPairArgs& a, cudaStream_t stream, bool split);
bool argus_pair_tiled_usable(const ArgusPairArgs& a);

extern "C" void argus_testing_set_poll_limit(unsigned int polls) { g_poll_limit.store(polls ? polls : 1u << 19); }

extern "C" int argus_testing_pair_passes(const void* workspace, uint32_t* counted, uint32_t* second_pass) {
  ArgusPairCtl ctl;  // (the first thing in the workspace)
  ARGUS_CUDA_TRY(cudaMemcpy(&ctl, workspace, sizeof(ctl), cudaMemcpyDeviceToHost));
  *counted = ctl.recount_done != 0;
  *second_pass = ctl.redo != 0;
  return ARGUS_OK;
}
extern "C" void argus_testing_set_hand_overs(int always) { g_hand_on.store(always ? 1u : 0u); }
extern "C" int argus_testing_hand_overs(const void* workspace, uint64_t* first_pass, uint64_t* second_pass) {
  ArgusPairCtl ctl;
  ARGUS_CUDA_TRY(cudaMemcpy(&ctl, workspace, sizeof(ctl), cudaMemcpyDeviceToHost));
  *first_pass = ctl.q_tail[0];
  *second_pass = ctl.q_tail[1];
  return ARGUS_OK;
}

extern "C" size_t argus_pair_workspace_bytes(uint64_t num_events, uint32_t num_streams, uint64_t ambig_capacity) {
  return make_layout(num_events, num_streams, ambig_capacity).total;
}

// Whole pairing pipeline. kernel_choice: 0 = automatic, 1 = one thread per stream, 2 = tiled.
int argus_internal_pair(const argus_event_t* events, uint64_t num_events, const uint64_t* stream_offsets,
                        uint32_t num_streams, uint32_t num_regions, argus_interval_t* intervals,
                        uint64_t interval_capacity, uint64_t* interval_offsets, argus_ambiguity_t* ambig,
                        uint64_t ambig_capacity, uint64_t* ambig_offsets, argus_status_t* status, void* workspace,
                        size_t workspace_bytes, void* cuda_stream, int kernel_choice, bool reset_status,
                        uint64_t* digest, uint64_t digest_capacity,
                        const uint64_t* ring_written, uint32_t ring_capacity) {
  if (!stream_offsets || !interval_offsets || !ambig_offsets || !status || !workspace) return ARGUS_ERR_INVALID_ARG;
  if ((num_events && !events) || (interval_capacity && !intervals) || (ambig_capacity && !ambig)) return ARGUS_ERR_INVALID_ARG;
  if (num_regions == 0 || num_regions > ARGUS_MAX_REGIONS) return ARGUS_ERR_INVALID_ARG;
  if (num_events >> ARGUS_NOTE_POS_BITS) return ARGUS_ERR_INVALID_ARG;
  if (((uintptr_t)events & 15) || ((uintptr_t)intervals & 15) || ((uintptr_t)ambig & 15) || ((uintptr_t)status & 7) ||
      ((uintptr_t)workspace & 255) || ((uintptr_t)stream_offsets & 7) || ((uintptr_t)interval_offsets & 7) ||
      ((uintptr_t)ambig_offsets & 7))
    return ARGUS_ERR_INVALID_ARG;
  const Layout L = make_layout(num_events, num_streams, ambig_capacity);
  if (workspace_bytes < L.total) return ARGUS_ERR_WORKSPACE;
  cudaStream_t stream = (cudaStream_t)cuda_stream;
  char* ws = (char*)workspace;

  ArgusPairArgs a;
  a.events = events; a.stream_offsets = (const u64*)stream_offsets; a.num_events = num_events;
  a.num_streams = num_streams; a.num_regions = num_regions;
  a.intervals = intervals; a.interval_capacity = interval_capacity; a.interval_offsets = (u64*)interval_offsets;
  a.counts = (u64*)(ws + L.counts); a.bases = (u64*)(ws + L.bases);
  a.notes = (u64*)(ws + L.notes); a.note_capacity = ambig_capacity;
  a.bits = (u32*)(ws + L.bits);
  a.ctl = (ArgusPairCtl*)(ws + L.ctl);
  a.status = status;
  a.redo = 0;
  a.queue = (u32*)(ws + L.queue); a.queue_capacity = L.queue_capacity;
  a.records = (ArgusStreamRecord*)(ws + L.records); a.record_capacity = L.record_capacity;
  a.poll_limit = g_poll_limit.load(std::memory_order_relaxed);
  a.hand_on = g_hand_on.load(std::memory_order_relaxed);
  a.ring_written = (const u64*)ring_written; a.ring_capacity = ring_capacity;
  if (ring_written && (ring_capacity == 0 || kernel_choice == 1)) return ARGUS_ERR_INVALID_ARG;  // only the tiled kernel reads rings
  // Digests lie at their records' positions, so the digest array bounds both. A trace has num_events / 2 intervals at most, which is
  // what the array holds; only offsets that decrease, which are reported, make streams share events and reach further.
  a.digest = (u64*)digest;
  if (digest && digest_capacity < a.interval_capacity) a.interval_capacity = digest_capacity;

  const bool tiled = (kernel_choice != 1 && argus_pair_tiled_usable(a)) || ring_written != nullptr;
  // control block, counts, queue and bitmap are contiguous at the start of the workspace and start at zero
  uint4* const zeroed = (uint4*)ws;
  const u64 zeroed_words = L.group_prefix / 16;
  u32* const order = (u32*)(ws + L.order);
  // Small calls: one block clears and orders. Beyond that a grid clears, and looks at the ends of the streams.
  const bool alone = num_events < (1u << 20) && num_streams <= 8192;
  // Windows all over the trace are looked at where that is little against the whole call (see kSampledEvents).
  u32* const samples = num_events >= kSampledEvents && num_streams ? (u32*)(ws + L.group_prefix) : nullptr;  // (not used before the offsets kernel)
  static_assert(kSampledEvents / 32 / kGroupWords >= kSamples, "room for the samples");
  if (!alone) {
    // a stream a warp, up to what the chip holds of them
    const u32 per = num_streams <= 148u * 64u ? 1u : num_streams < 32u * 148u * 64u ? (num_streams + 148u * 64u - 1) / (148u * 64u) : 32u;
    u64 want = ((u64)num_streams / per + kInitThreads / 32 - 1) / (kInitThreads / 32) + zeroed_words / 4096 + 1;
    if (samples && want < kSamples * 32 / kInitThreads) want = kSamples * 32 / kInitThreads;  // a window a warp
    ARGUS_LAUNCH(k_pair_init, (unsigned)(want < 1184 ? want : 1184), kInitThreads, 0, stream, a, zeroed, zeroed_words, (int)reset_status, per, samples);
  }
  const bool many = num_streams > kScanThreads;
  const bool split = kernel_choice == 0 && tiled && !ring_written && argus_split_usable(num_events, num_streams);
  ARGUS_LAUNCH(many ? k_pair_order<kScanRun> : k_pair_order<1>, samples ? 148u : 1u, kScanThreads, 0, stream, a, order, zeroed, zeroed_words, (int)reset_status, (int)alone, (int)split,
               (const u32*)samples);
  a.order = tiled && num_streams > 1 ? order : nullptr;
  a.segments = nullptr; a.split_failed = nullptr; a.segment_tiles = 0;

  AmbigArgs g;
  g.p = a; g.num_words = L.num_words; g.span = num_events;
  g.group_prefix = (u32*)(ws + L.group_prefix); g.block_prefix = (u64*)(ws + L.block_prefix);
  g.num_blocks = L.num_blocks; g.ambig = ambig; g.ambig_capacity = ambig_capacity; g.ambig_offsets = (u64*)ambig_offsets;
  for (int pass = 0; pass < 2; ++pass) {
    a.redo = pass;
    if (num_streams) {
      if (pass == 0) argus_prof_mark(ARGUS_PROF_PAIR, stream, 0);
      if (tiled) {
        if (pass == 0 && split) {
          const int rc = argus_launch_pair_split(a, ws + L.split, stream);
          if (rc != ARGUS_OK) return rc;
        }
        const int rc = argus_launch_pair_tiled(a, stream, false);
        if (rc != ARGUS_OK) return rc;
      } else {
        ARGUS_LAUNCH(k_pair_thread_per_stream, (num_streams + 127) / 128, 128, 0, stream, a);
      }
      if (pass == 0) argus_prof_mark(ARGUS_PROF_PAIR, stream, 1);
    }
    if (pass == 0)
      ARGUS_LAUNCH(many ? k_pair_offsets<kScanRun> : k_pair_offsets<1>, (unsigned)(L.num_blocks < 295 ? L.num_blocks : 295) + 1, kScanThreads, 0, stream, g);
  }
  const u64 want = ((u64)num_streams + 1 + 255) / 256;
  ARGUS_LAUNCH(k_ambig_records, (unsigned)(alone ? (want > 16 ? want : 16) : 296), 256, 0, stream, g);
  return ARGUS_OK;
}

extern "C" int argus_pair_intervals_ex(const argus_event_t* events, uint64_t num_events, const uint64_t* stream_offsets,
                                       uint32_t num_streams, uint32_t num_regions, argus_interval_t* intervals,
                                       uint64_t interval_capacity, uint64_t* interval_offsets, argus_ambiguity_t* ambig,
                                       uint64_t ambig_capacity, uint64_t* ambig_offsets, argus_status_t* status,
                                       void* workspace, size_t workspace_bytes, void* cuda_stream, int kernel_choice) {
  return argus_internal_pair(events, num_events, stream_offsets, num_streams, num_regions, intervals, interval_capacity,
                             interval_offsets, ambig, ambig_capacity, ambig_offsets, status, workspace, workspace_bytes,
                             cuda_stream, kernel_choice, true);
}

extern "C" int argus_pair_intervals(const argus_event_t* events, uint64_t num_events, const uint64_t* stream_offsets,
                                    uint32_t num_streams, uint32_t num_regions, argus_interval_t* intervals,
                                    uint64_t interval_capacity, uint64_t* interval_offsets, argus_ambiguity_t* ambig,
                                    uint64_t ambig_capacity, uint64_t* ambig_offsets, argus_status_t* status,
                                    void* workspace, size_t workspace_bytes, void* cuda_stream) {
  return argus_pair_intervals_ex(events, num_events, stream_offsets, num_streams, num_regions, intervals,
                                 interval_capacity, interval_offsets, ambig, ambig_capacity, ambig_offsets, status,
                                 workspace, workspace_bytes, cuda_stream, 0);
}

extern "C" int argus_pair_intervals_ring(const argus_event_t* ring, uint32_t slot_capacity, const uint64_t* written,
                                         uint32_t num_streams, uint32_t num_regions, uint64_t* stream_offsets,
                                         uint64_t* dropped, argus_interval_t* intervals, uint64_t interval_capacity,
                                         uint64_t* interval_offsets, argus_ambiguity_t* ambig, uint64_t ambig_capacity,
                                         uint64_t* ambig_offsets, argus_status_t* status, void* workspace,
                                         size_t workspace_bytes, void* cuda_stream) {
  if (!status || !stream_offsets || slot_capacity == 0) return ARGUS_ERR_INVALID_ARG;
  if (num_streams && (!ring || !written)) return ARGUS_ERR_INVALID_ARG;
  if (((uintptr_t)written & 7) || ((uintptr_t)dropped & 7)) return ARGUS_ERR_INVALID_ARG;
  { const int rc = argus_internal_clear(status, nullptr, 0, cuda_stream); if (rc != ARGUS_OK) return rc; }
  const uint64_t bound = (uint64_t)num_streams * slot_capacity;  // what the slots can hold: sizes the workspace
  int rc = argus_internal_ring_offsets(written, slot_capacity, num_streams, bound, stream_offsets, dropped, status, cuda_stream);
  if (rc != ARGUS_OK) return rc;
  return argus_internal_pair(ring, bound, stream_offsets, num_streams, num_regions, intervals, interval_capacity, interval_offsets,
                             ambig, ambig_capacity, ambig_offsets, status, workspace, workspace_bytes, cuda_stream, 2, false,
                             nullptr, 0, written, slot_capacity);
}
