// argus_pair_tiled.cu — tiled pairing kernel for sm_100a.
//
// One CTA walks one stream tile by tile (T = NT * E events per tile); tiles arrive in shared
// memory by TMA bulk copies (double buffered, mbarrier completion) and interval records leave with
// 32- and 16-byte stores, one thread per record. The per-stream region stack is carried from tile
// to tile in shared memory; a CTA waits for another only when it has nothing to do (see ArgusStreamRecord).
//
// Inside a tile the stack height before each event is a count of begins and ends: among 32 in a row by vote, over the
// warps by one exchange. So every marker knows its level (stack position) without walking the stack:
//   - the begins of 32 markers in a row that open the same level are one word of that level's bitmap over the tile's
//     event positions, stored at once (a bit at a time where a window does not cover the tile);
//   - every end (one thread per end marker) finds its begin as the latest set bit of its own level
//     before it, and its parent as the latest set bit one level down before that begin; when there
//     is none in the tile, the frame is in the stack carried from earlier tiles;
//   - every finished interval adds its inclusive time to its parent frame's accumulator (shared
//     atomics), which gives exclusive time without ordering the threads. The accumulators hold what
//     the current window adds, in 32 bits (a frame carried from earlier tiles brings its 64-bit child
//     time along separately); an interval or a sum that does not fit breaks the rules below.
// This is exact when the tile is well nested (every end meets the frame on top with the same region
// id). A tile is consumed in windows: the first position where a rule fails (region mismatch, negative
// height, bad region id, depth overflow, level window exceeded, 2^32 ticks of child time in one
// window) cuts the window there; what lies before it counts (what ends behind it have added to their
// parents is taken back; if a sum wrapped, it is done again, up to the cut), the offending marker goes through the
// sequential stack machine on the carried stack, and a new window starts after it, so the result is always the
// sequential definition's.
//
// Bound by instruction issue and the latency of the phases (7 blocks = 28 warps per SM, capped by shared memory and registers
// alike), next by the way of shared-memory accesses through the load/store pipe. Looking an end up and writing its record in one
// go, with one barrier between, instead of two sweeps over all ends that each read both event records: a quarter fewer
// shared-memory wavefronts; together with a window that needs no bounds checks as the usual case and look-ups without range
// selects (decode trace, 614 M events: 5.42 -> 5.01 ms); then heights by vote over 32 markers in a row instead of a scan over the
// threads' own five, and a word of a level's bitmap stored at once, by the lowest lane of those that match in level, instead of
// a bit at a time (4.90 ms = 5.0 TB/s of 16 B read + 24 B written an event, 77 % of the copy rate, 5.5 TB/s with the digests;
// attention 1.50 -> 1.45 ms; with votes but a bit at a time 5.08 and 1.57); then records in whole sectors (tile_store_record) and streams that
// change hands where that keeps the SMs busy (ArgusStreamRecord): decode 4.61 ms, attention 1.18, GEMM 0.54. Tiles of 512 events with 8 blocks: GEMM 638 -> 707
// us, 160 threads with four events each and 6 blocks: 674.
#include "argus_internal.cuh"
#include "argus_bulk.cuh"
#include "argus_pair_common.cuh"

#include <atomic>
#include <mutex>
#include <type_traits>

namespace {

constexpr int kLevelWindow = 16;  // begins of a tile may sit at levels [lbase, lbase + 16)
constexpr int kCar = 80;          // slots of a carried-frame block: 64 frames, 1 sink for "no parent", padding
constexpr int kSink = 64;         // index of the sink slot inside a carried-frame block
constexpr int kBadRef = 0x3fff;   // reference that marks a window as not well nested
constexpr int kSeqChunk = 128;    // markers handed to the sequential machine at once when cuts come densely
constexpr u32 kNoRec = 0xffffffffu;
constexpr u64 kNoWork = ~0ull;

__device__ __forceinline__ void tile_progress(const ArgusPairArgs& a, u64 by) {
  atomicAdd(reinterpret_cast<unsigned long long*>(&a.ctl->progress[a.redo ? 1 : 0]), by);
}

// Claims a first position; false if another CTA has. The CTA that claims the last of a word's positions counts the word.
__device__ __forceinline__ bool tile_claim(ArgusPairCtl* ctl, int p, u32 at) {
  const u32 bit = 1u << (at & 31), word = at / 32, all = gridDim.x - word * 32 < 32 ? (1u << (gridDim.x & 31)) - 1u : ~0u;
  const u32 before = atomicOr(ctl->claimed[p][word], bit);
  if (before & bit) return false;
  if ((before | bit) == all) atomicAdd(&ctl->claimed_words[p], 1u);
  return true;
}

// A first position that no CTA has claimed; kNoRec if there is none.
__device__ __forceinline__ u32 tile_claim_any(ArgusPairCtl* ctl, int p) {
#pragma unroll 1
  for (u32 at = 0; at < gridDim.x; ++at) {
    const u32 open = ~__ldcg(ctl->claimed[p][at / 32]) >> (at & 31);
    if (!open) { at |= 31; continue; }
    at += __ffs((int)open) - 1;
    if (at < gridDim.x && tile_claim(ctl, p, at)) return at;
  }
  return kNoRec;
}

// Takes the next piece of work of pass `p`: a stream nobody has started (position below num_streams) or a
// hand-over from the queue. Returns false when every stream is done (or on a timeout). *rec: the stream's hand-over record (kNoRec: it
// has none), *resumed: what to start from is in there, *more: others wait. A CTA's first position is its own number, so that every SM
// gets its share of the long streams, which come first (the CTAs of an SM ask at the same time: with 296 long streams among
// 1,776 taken as they come, 42 SMs had seven of them each, the others none, and walked 791 tiles instead of 700: GEMM trace 545 -> 633 us; the
// first positions taken seven strata apart, whoever comes: 633, too). But a CTA may start late, when another kernel holds part of the
// chip, and nothing may wait for one that has not started: so the first position is claimed by a bit, and a CTA that would wait for
// a hand-over while not all are claimed takes one that is left instead. *drawn: a position that the CTA has, but has not used yet;
// first_stream: what lies at its own number. Whatever does not depend on one another is asked for together: a round trip is 0.7 us of
// the smallest call. One thread per CTA.
__device__ __forceinline__ bool tile_pop_work(const ArgusPairArgs& a, int p, u64* drawn, u64 first_stream, u64* stream, u32* rec, bool* resumed, bool* more) {
  u64 h = *drawn;
  const bool first = h < a.num_streams;
  u32 words = 0;
  u64 tail = 0;
  if (!first) {
    words = atomicAdd(&a.ctl->claimed_words[p], 0u);
    tail = atomicAdd(reinterpret_cast<unsigned long long*>(&a.ctl->q_tail[p]), 0ull);
  }
  if (h == kNoWork) h = gridDim.x + atomicAdd(reinterpret_cast<unsigned long long*>(&a.ctl->q_head[p]), 1ull);
  *drawn = kNoWork;
  *resumed = h >= a.num_streams;
  if (h < a.num_streams) {
    *stream = first ? first_stream : a.order ? a.order[h] : h;
    *rec = h < a.record_capacity ? (u32)h : kNoRec;  // (streams come longest first; those without a record are walked whole)
    *more = h + 1 < a.num_streams || (first ? atomicAdd(reinterpret_cast<unsigned long long*>(&a.ctl->q_tail[p]), 0ull) : tail);
    return true;
  }
  if (words < (gridDim.x + 31) / 32) {
    const u32 left = tile_claim_any(a.ctl, p);
    if (left != kNoRec) {
      *drawn = h;
      *resumed = false;
      *stream = a.order ? a.order[left] : left;
      *rec = left < a.record_capacity ? left : kNoRec;
      *more = true;
      return true;
    }
  }
  const u64 slot = h - a.num_streams;
  if (!a.queue || slot >= a.queue_capacity) return false;  // more positions than hand-overs can ever be published
  volatile u32* q = a.queue + slot;
  *more = tail > slot + 1;
  u64 seen = ~0ull;
  u32 idle = 0, nap = 64;
  for (;;) {
    // An entry that was stored before the counter moved has to be seen, since it is not looked for again until the counter moves. (Acquired by the read
    // itself: a fence in every round, by all who wait, took 10 K markers 41.3 -> 41.0 us, ring of 74 M 1,521 -> 1,512.)
    u64 now;
    asm volatile("atom.acquire.gpu.global.add.u64 %0, [%1], 0;" : "=l"(now) : "l"(&a.ctl->progress[p]) : "memory");
    if (now != seen) {
      if ((u32)now >= a.num_streams) return false;
      const u32 v = *q;
      if (v) {
        *q = 0;  // the second pass uses the same entries
        __threadfence();
        *rec = v - 1;
        *stream = *reinterpret_cast<volatile u32*>(&a.records[v - 1].stream);
        return true;
      }
      if (seen == ~0ull) atomicExch(&a.ctl->level[p], 0u);
      seen = now;
      idle = 0;
    }
    if (++idle > a.poll_limit) {  // ~1 s without any movement anywhere
      argus_set_error(a.status, ARGUS_ERR_TIMEOUT, 0, slot);
      return false;
    }
    __nanosleep(nap);
    if (nap < 2048) nap *= 2;
  }
}

// Shared memory of one CTA. Events of the two tile buffers and the frames carried from earlier tiles
// share one index space, so that "the frame an end closes" and "its parent" are plain indices:
//   ev0[0..T) | car0[0..80) | car1[0..80) | ev1[0..T)
// Seen from buffer 0, carried block c holds level L at T + 80 c + L; seen from buffer 1 at 80 c + L - 160.
// A window reads the current block and writes the stack it leaves behind into the other one.
template <int NT, int E>
struct TileSmem {
  static constexpr int T = NT * E;
  static constexpr int NW = NT / 32;
  static constexpr int NWORDS = T / 32;                 // bitmap words per level
  static constexpr int MAXI = T / 2 + ARGUS_MAX_DEPTH;  // intervals a well-nested tile can emit
  static constexpr int NI = (MAXI + NT - 1) / NT;       // intervals per thread in the emission phases
  static constexpr int kDescShift = T <= 1024 ? 10 : 16;
  using desc_t = typename std::conditional<(T <= 1024), unsigned short, u32>::type;
  uint4 evall[2 * T + 2 * kCar];
  alignas(16) u32 accall[T + 4 * kCar];      // child time each frame gathers in the current window (32 bits: an overflow cuts the
                                   // window), same index space shifted by 2 kCar
  desc_t desc[MAXI];               // per end, in end order: event index | level << kDescShift
  static constexpr int kBmVectors = ((kLevelWindow + 1) * NWORDS + 3) / 4;  // 16-byte vectors that cover bm
  union {
    alignas(16) u32 bm[kLevelWindow + 1][NWORDS];  // (the last row stays empty: levels outside the window) per level: bit e set = event e of the tile is a begin at that level
    uint4 bm_vectors[kBmVectors];      // the same, as it is cleared: all of it, the last words of the last row too
    ArgusFrame fstk[ARGUS_MAX_DEPTH];  // stack in the layout the sequential path uses (no bitmap is live while it runs)
  };
  u64 summ[kLevelWindow + 1];      // per level: bit w set = bm[level][w] != 0
  u32 cidx[2][ARGUS_MAX_DEPTH];    // begin index (within the stream) of each carried frame
  u64 cchild[2][ARGUS_MAX_DEPTH];  // child time of each carried frame as the window found it
  alignas(16) u32 warp_tot[32];
  u64 bar[2];
  u64 cur_stream;
  u32 cur_rec;                     // hand-over record of the stream being walked (kNoRec: none)
  int skip;                        // the piece of work taken is not to be walked
  int resumed;                     // its state is in the record
  int more, level;                 // others wait; and this CTA says how long they are
  int started;                     // this CTA has had work
  u64 drawn, first_stream;         // a position that it has and has not used yet; the stream at its own number
  u32 ti_end, look;                // where this CTA stops; the tile at which thread 0 looks up what waits
  int stop;                        // split pass: everything is left to the chained pass
  u64 n_int;                       // written by the sequential redo path
  int ch;
  u32 wrapped;                     // a sum of 32-bit child time wrapped in this window
  int badpos[2];                   // first position of the window where the parallel rules fail (INT_MAX = none); windows alternate
                                   // between the two, so that one can be reset while stragglers still read the other
  int dead, failed;
  int low;                         // split pass: lowest initial frame that the window closed
};

// Latest begin of the tile at level L and position < pos; -1 if there is none. INSIDE: pos < T, else pos <= T. Written without
// branches: the lanes of a warp would otherwise split over "same word", "earlier word" and "not in this tile" and run all
// three paths one after the other.
template <int NT, int E, bool INSIDE>
__device__ __forceinline__ int tile_latest_begin(const TileSmem<NT, E>& sm, int L, int lbase, int pos) {
  constexpr int NWORDS = TileSmem<NT, E>::NWORDS;
  const u32 l = (u32)(L - lbase) < (u32)kLevelWindow ? (u32)(L - lbase) : (u32)kLevelWindow;
  const int w = pos >> 5;
  const bool in_tile = INSIDE || w < NWORDS;     // pos == T: every word lies before it
  const u32 m = in_tile ? sm.bm[l][w] & ((1u << (pos & 31)) - 1u) : 0u;  // begins of the level in the same word, before pos
  int w2;                                        // last earlier word with a begin of the level
  bool earlier;
  if (NWORDS <= 32) {                            // one 32-bit word of the summary covers the tile
    const u32 s = reinterpret_cast<const u32*>(&sm.summ[l])[0] & ((INSIDE || w < 32) ? (1u << w) - 1u : ~0u);
    earlier = s != 0;
    w2 = earlier ? 31 - __clz(s) : 0;
  } else {
    const u64 s = sm.summ[l] & ((w >= 64) ? ~0ull : ((1ull << w) - 1ull));
    earlier = s != 0;
    w2 = earlier ? 63 - __clzll((long long)s) : 0;
  }
  const u32 m2 = sm.bm[l][w2];                   // not empty if its summary bit is set
  const int r = (m ? w : w2) * 32 + 31 - __clz(m ? m : m2);
  return m || earlier ? r : -1;
}


// An interval record, which starts on a 32-byte boundary or 16 bytes behind one, as its aligned 32 bytes and the other 16. Beside a neighbour's
// 16, stored by the same instruction, every 32-byte sector is written once and whole; three 16-byte stores write each in two
// halves, and the L2 takes as long for a half as for all of it. (GEMM 573 -> 549 us, attention 1,246 -> 1,191, decode 2,441 -> 2,339;
// as predicated stores, without selects, 599, 1,283 and 2,531: 16 bytes of registers spilled.)
__device__ __forceinline__ void tile_store_record(uint4* q, u32 t0, u32 t1, u32 incl, u32 excl, u32 region, u32 ctx, u32 stream, u32 parent,
                                                  u32 idx, u32 depth_flags) {
  const bool odd = (reinterpret_cast<uintptr_t>(q) & 16) != 0;
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(q + (odd ? 1 : 0)), "r"(odd ? excl : t0), "r"(odd ? 0u : t1),
               "r"(odd ? region : incl), "r"(odd ? ctx : 0u), "r"(odd ? stream : excl), "r"(odd ? parent : 0u), "r"(odd ? idx : region),
               "r"(odd ? depth_flags : ctx)
               : "memory");
  q[odd ? 0 : 2] = odd ? make_uint4(t0, t1, incl, 0u) : make_uint4(stream, parent, idx, depth_flags);
}

// One tile of a stream into shared memory: a bulk copy, or two when the stream lives in a ring slot and the
// tile straddles the slot's end. `src` is the stream's first record (packed input) or its slot (ring).
template <bool RING>
__device__ __forceinline__ void tile_fetch(const ArgusPairArgs& a, uint4* dst, const argus_event_t* src, u32 ring_first,
                                           u32 start, u32 count, u64* bar) {
  mbar_expect_tx(bar, count * 16u);
  if (!RING) {
    tma_load_1d(dst, src + start, count * 16u, bar);
  } else {
    u32 p = ring_first + start;  // both below the capacity
    if (p >= a.ring_capacity) p -= a.ring_capacity;
    const u32 room = a.ring_capacity - p;
    const u32 head = count < room ? count : room;
    tma_load_1d(dst, src + p, head * 16u, bar);
    if (count > head) tma_load_1d(dst + head, src, (count - head) * 16u, bar);
  }
}

// SPLIT: the work items are segments of streams instead of whole streams (see argus_pair_split.cu): the initial stack comes with
// the segment, and a marker that breaks the parallel rules gives the stream up to the chained pass that follows. Other blocks may
// give up the stream of this block's segment at any moment, so one thread reads that word and all threads follow its answer; the
// other words of global memory that a block branches on around its barriers (offsets, bases, segments, hand-over records, redo,
// redo_from, and after the split pass its outcome) are not written while the kernel runs, or are read by the one thread that takes the
// work, as is the word that calls the split pass off.
template <int NT, int E, int MINB, bool RING = false, bool SPLIT = false>
__global__ void __launch_bounds__(NT, MINB) k_pair_tiled(ArgusPairArgs a) {
  using SM = TileSmem<NT, E>;
  constexpr int T = SM::T, NW = SM::NW, NWORDS = SM::NWORDS, MAXI = SM::MAXI, NI = SM::NI;
  static_assert(NW <= 32 && NT % 32 == 0 && NT >= ARGUS_MAX_DEPTH && NWORDS <= 64 && T + kCar < kBadRef, "block shape");
  extern __shared__ __align__(128) unsigned char smem_raw[];
  SM& sm = *reinterpret_cast<SM*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  argus_kernel_begin_long();
  if (a.redo && !__ldcg(&a.ctl->redo)) return;
  bool failed = false;
  const bool segments = !SPLIT && !a.redo && a.segments && argus_split_in_force(a, &failed);  // the chained pass after a split one
  if (segments && !failed) return;
  if (!SPLIT && tid == 32) {  // (beside what thread 0 does)
    sm.first_stream = a.order ? a.order[blockIdx.x] : blockIdx.x;
    sm.drawn = tile_claim(a.ctl, a.redo ? 1 : 0, blockIdx.x) ? blockIdx.x : kNoWork;
  }
  if (tid == 0) {
    mbar_init(&sm.bar[0], 1);
    mbar_init(&sm.bar[1], 1);
    fence_mbar_init();
    sm.dead = sm.started = 0;
    for (int w = NW; w < 32; ++w) sm.warp_tot[w] = 0;
    // the sink of both carried blocks: its tag, shifted arithmetically, reads as ARGUS_NONE
    sm.evall[T + kSink] = sm.evall[T + kCar + kSink] = make_uint4(0, 0, 0xfffffffeu, 0);
    sm.badpos[0] = sm.badpos[1] = 0x7fffffff;
  }
  __syncthreads();
  u32 ph0 = 0, ph1 = 0;  // mbarrier phase parities
  int bp = 0;            // which of sm.badpos the next window uses
  const u64 off0 = a.stream_offsets[0];
  u32 tot_ctx = 0, tot_rev = 0, tot_clamp = 0;

  for (;;) {
    if (tid == 0) {
      u64 st = ~0ull;
      u32 rc = kNoRec;
      bool skip = false, resumed = false, more = false;
      if (SPLIT) {
        const uint4 w = __ldcg(reinterpret_cast<const uint4*>(&a.ctl->num_failed));  // num_failed, num_segments, split
        rc = atomicAdd(&a.ctl->seg_head, 1u);
        st = w.z && rc < w.y ? a.segments[rc].stream : ~0ull;
        skip = w.x && st < a.num_streams && __ldcg(a.split_failed + st);
      } else if (!tile_pop_work(a, a.redo ? 1 : 0, &sm.drawn, sm.first_stream, &st, &rc, &resumed, &more)) st = ~0ull;
      sm.cur_stream = st;
      sm.cur_rec = rc;
      if (!SPLIT) {
        sm.resumed = resumed;
        sm.level = sm.started || blockIdx.x == gridDim.x - 1;  // (not by all blocks at once when the kernel starts)
        sm.more = more;
        sm.started = 1;
      }
      if (!SPLIT && segments) skip = st < a.num_streams && !resumed && !__ldcg(a.split_failed + st);
      sm.skip = skip;
      sm.stop = 0;
    }
    __syncthreads();
    const u64 s64 = sm.cur_stream;
    if (s64 >= a.num_streams) break;
    const u32 s = (u32)s64;
    const u32 rec = sm.cur_rec;
    if (sm.skip) {
      if (!SPLIT && tid == 0) tile_progress(a, 1);  // walked by the split pass
      __syncthreads();
      continue;
    }
    ArgusSegment* const seg = SPLIT ? a.segments + rec : nullptr;
    const u64 lo = a.stream_offsets[s], hi = a.stream_offsets[s + 1];
    if (hi < lo || hi > a.num_events || lo < off0 || ((hi - lo) >> 32)) {
      if (tid == 0) {
        argus_set_error(a.status, ARGUS_ERR_BAD_OFFSETS, s, 0);
        if (!a.redo) a.counts[s] = 0;
        if (!SPLIT) tile_progress(a, 1);  // (the chained pass counts what the split pass has walked)
      }
      __syncthreads();
      continue;
    }
    const u32 n = (u32)(hi - lo);
    const u64 gpos0 = lo - off0;
    const u64 out_base = a.redo ? a.interval_offsets[s] : a.bases[s];
    if (a.redo && s < __ldcg(&a.ctl->redo_from)) {
      // second pass: this stream's intervals (and digests) already lie where they belong
      if (tid == 0) tile_progress(a, 1);
      __syncthreads();
      continue;
    }
    const argus_event_t* src = RING ? a.events + (u64)s * a.ring_capacity : a.events + lo;
    const u32 ring_first = RING ? argus_ring_first(a, s) : 0u;
    const u32 ntiles = (n + T - 1) / T;
    int ch = 0;          // carried stack height (uniform)
    u64 n_int = 0;       // intervals of this stream so far (uniform)
    bool stream_failed = false;
    u32 ti0 = 0;
    constexpr u32 kChunkTiles = (kChunkEvents + T - 1) / T < 2 ? 2 : (kChunkEvents + T - 1) / T;
    auto look_after = [](u32 left) { return left / 8 > kChunkTiles ? left / 8 : kChunkTiles; };  // tiles; a look costs half a us
    int init_h = 0;      // split: frames of the initial stack that are still open (uniform)
    u64 limit = a.interval_capacity;
    if (SPLIT) {
      ti0 = seg->first_tile;
      ch = init_h = seg->ch;
      n_int = ((u64)ti0 * T - (u64)ch) >> 1;  // every marker before is a begin or an end, and the open ones are the difference
      if (a.bases[s + 1] < limit) limit = a.bases[s + 1];
      if (tid < ch) {
        const u32 at = seg->idx[tid];
        sm.evall[T + tid] = __ldg(reinterpret_cast<const uint4*>(src + at));
        sm.cchild[0][tid] = 0;
        sm.cidx[0][tid] = at;
      }
      if (tid == 0) sm.low = 0x7fffffff;
    } else if (sm.resumed) {
      const ArgusStreamRecord* r = a.records + rec;
      ti0 = __ldcg(&r->next_tile);
      ch = __ldcg(&r->ch);
      n_int = __ldcg(&r->n_int);
      if (tid < ch) {  // the carried block 0 is where the first window looks
        sm.evall[T + tid] = __ldcg(&r->frames[tid]);
        sm.cchild[0][tid] = __ldcg(&r->child[tid]);
        sm.cidx[0][tid] = __ldcg(&r->idx[tid]);
      }
    }
    // thread 0 alone decides where the piece ends
    if (tid == 0) {
      const u32 end = SPLIT ? ti0 + seg->num_tiles : ntiles;
      sm.ti_end = end;
      if (ti0 < end) {  // first tile of this piece, into the buffer its index selects
        const u32 start = ti0 * (u32)T;
        tile_fetch<RING>(a, (ti0 & 1) ? sm.evall + T + 2 * kCar : sm.evall, src, ring_first, start,
                         (n - start) < (u32)T ? (n - start) : (u32)T, &sm.bar[ti0 & 1]);
      }
      if (!SPLIT) {
        sm.look = rec != kNoRec ? ti0 + look_after(ntiles - ti0) - 2 : 0xffffffffu;
        if (sm.level) atomicExch(&a.ctl->level[a.redo ? 1 : 0], sm.more ? n - ti0 * (u32)T : 0u);
      }
    }
    __syncthreads();

    int cpar = 0;        // which carried-frame block holds the current stack
    u32 ti = ti0;
    for (; ti < sm.ti_end; ++ti) {
      const int b = ti & 1;
      const u32 tile_start = ti * (u32)T;
      const int tn = (int)((n - tile_start) < (u32)T ? (n - tile_start) : (u32)T);
      uint4* const ev0 = sm.evall;
      uint4* const ev1 = sm.evall + T + 2 * kCar;
      const uint4* evb = b ? ev1 : ev0;                  // evb[ref] for every reference of this tile
      u32* accb = sm.accall + 2 * kCar;                  // accb[ref], ref in [-2 kCar, T + 2 kCar)
      const int carlo = b ? -2 * kCar : T;               // reference of slot 0 of carried block 0, seen from this buffer
      if (tid == 0 && ti + 1 < sm.ti_end) {  // prefetch the next tile into the other buffer
        const u32 nstart = tile_start + T;
        tile_fetch<RING>(a, b ? ev0 : ev1, src, ring_first, nstart, (n - nstart) < (u32)T ? (n - nstart) : (u32)T, &sm.bar[b ^ 1]);
      }
      {
        const u32 go_on = SPLIT && tid == 0 && (ti & 7u) == 7u ? __ldcg(&a.ctl->split) : 1u;
        const bool ok = mbar_wait_bounded(&sm.bar[b], b ? ph1 : ph0);
        if (b) ph1 ^= 1; else ph0 ^= 1;
        if (!ok) sm.dead = 1;
        if (SPLIT && !go_on) sm.stop = 1;
        if (!SPLIT && tid == 0) {
          if (ti == sm.look && ti + 2 + kLeastTiles <= ntiles) {  // (others read sm.ti_end after the tile's barriers)
            const u32 half = atomicOr(&a.ctl->level[a.redo ? 1 : 0], 0u) / 2;
            if (a.hand_on || (half > kLevelMargin && n - (ti + 2) * (u32)T < half - kLevelMargin)) sm.ti_end = ti + 2;
            sm.look = ti + look_after(ntiles - ti);
          }
          if ((ti & 31u) == 31u) tile_progress(a, 1ull << 32);  // whoever waits sees that streams get on
        }
      }

      // The tile is consumed in windows [w0, wend). A well-nested tile is one window. When the parallel
      // rules fail first at position p, the window is cut there: [w0, p) counts (it is well nested), the
      // marker at p goes through the sequential stack machine, and a new window starts after it.
      int w0 = 0, wend = tn, small_streak = 0;
      while (w0 < tn) {
        const int cbase = carlo + cpar * kCar;           // carried level L -> reference cbase + L
        uint4* const car_next = sm.evall + T + (cpar ^ 1) * kCar;

        // ---------------- phase A: heights by votes; begins into per-level bitmaps; ends into `desc` ----------
        const bool whole = w0 == 0 && wend == T;  // the usual window: no marker needs a look at the window's bounds
        // a warp looks at 32 E markers in a row, 32 at a time: what lies before a marker is a vote and a count of bits
        const int e0 = w0 + warp * (32 * E) + lane;
        u32 tags[E], begins[E], ends[E];
        u32 mine_cnt = 0;  // the warp's begins, ends: 16 bits each
#pragma unroll
        for (int k = 0; k < E; ++k) tags[k] = whole || e0 + 32 * k < wend ? reinterpret_cast<const u32*>(evb + e0 + 32 * k)[2] : 0xffffffffu;
        for (int i = tid; i < T / 4; i += NT) reinterpret_cast<uint4*>(accb)[i] = make_uint4(0, 0, 0, 0);
        for (int i = tid; i < SM::kBmVectors; i += NT) sm.bm_vectors[i] = make_uint4(0, 0, 0, 0);
        if (tid <= kLevelWindow) sm.summ[tid] = 0;
        if (tid < ch) accb[cbase + tid] = 0;  // what this window adds to the carried frames (a cut window starts clean again)
        if (tid == 0) { sm.failed = 0; sm.wrapped = 0; accb[cbase + kSink] = 0; }
        if (whole) {
#pragma unroll
          for (int k = 0; k < E; ++k) {
            ends[k] = __ballot_sync(0xffffffffu, tags[k] & 1u);
            begins[k] = ~ends[k];
            mine_cnt += __popc(ends[k]);
          }
          mine_cnt = (mine_cnt << 16) + (32 * E - mine_cnt);
        } else {
#pragma unroll
          for (int k = 0; k < E; ++k) {
            const bool valid = e0 + 32 * k < wend;
            ends[k] = __ballot_sync(0xffffffffu, valid && (tags[k] & 1u));
            begins[k] = __ballot_sync(0xffffffffu, valid && !(tags[k] & 1u));
            mine_cnt += (__popc(ends[k]) << 16) + __popc(begins[k]);
          }
        }
        // block prefix sum: one barrier
        if (lane == 0) sm.warp_tot[warp] = mine_cnt;
        __syncthreads();
        u32 before = 0, tot = 0;
#pragma unroll
        for (int w = 0; w < NW; w += 4) {
          const uint4 t4 = *reinterpret_cast<const uint4*>(sm.warp_tot + w);  // (entries past NW are zero)
          const u32 t[4] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            if (w + q < warp) before += t[q];
            tot += t[q];
          }
        }
        const u32 ex = before;
        const int win_ne = (int)(tot >> 16) < MAXI ? (int)(tot >> 16) : MAXI;  // more ends than that means a violation earlier
        const int h0 = ch + (int)(ex & 0xffffu) - (int)(ex >> 16);
        const int lbase = ch > kLevelWindow / 2 ? ch - kLevelWindow / 2 : 0;
        // levels a begin may open: inside the window of levels and below 64
        const u32 levels = ARGUS_MAX_DEPTH - lbase < kLevelWindow ? (u32)(ARGUS_MAX_DEPTH - lbase) : (u32)kLevelWindow;
        // flat, so that begins and ends of a warp are handled by predication, not by two passes. The parallel rules: known region
        // id, height never negative, levels as above; the first marker that breaks one is reported, later ones (whose heights may
        // mean nothing) at most leave bits and descriptors behind it.
        auto place = [&](auto WHOLE) {
          int h_base = h0, rank_base = (int)(ex >> 16);
          const u32 lower = (1u << lane) - 1u;
          u32 viol = 0;
#pragma unroll
          for (int k = 0; k < E; ++k) {
            const int e = e0 + 32 * k;
            const bool valid = decltype(WHOLE)::value || e < wend;  // (not "tag != all ones": that is a marker too, with a region id out of range)
            const bool is_e = valid && (tags[k] & 1u), is_b = valid && !(tags[k] & 1u);
            const int nb = __popc(begins[k] & lower);
            const int ne = decltype(WHOLE)::value ? lane - nb : __popc(ends[k] & lower);
            const int h = h_base + nb - ne, rank = rank_base + ne;
            const u32 l = (u32)(h - lbase);  // level of the frame a begin opens, inside the window
            const bool ok_b = l < levels;
            if ((valid && (tags[k] >> 1) >= a.num_regions) || (is_e && h < 1) || (is_b && !ok_b)) viol |= 1u << k;
            if (is_e && rank < MAXI) sm.desc[rank] = (typename SM::desc_t)((u32)e | ((u32)((h - 1) & 0x3f) << SM::kDescShift));
            if (decltype(WHOLE)::value) {  // the warp's 32 markers are one word of the bitmaps: a store for each level
              const u32 same = __match_any_sync(0xffffffffu, is_b && ok_b ? l : 0xffffffffu);
              if (is_b && ok_b && !(same & lower)) {
                sm.bm[l][e >> 5] = same;
                atomicOr(reinterpret_cast<u32*>(&sm.summ[l]) + (NWORDS <= 32 ? 0 : e >> 10), 1u << ((e >> 5) & 31));
              }
            } else if (is_b && ok_b) {
              atomicOr(&sm.bm[l][e >> 5], 1u << (e & 31));
              atomicOr(reinterpret_cast<u32*>(&sm.summ[l]) + (NWORDS <= 32 ? 0 : e >> 10), 1u << ((e >> 5) & 31));
            }
            rank_base += __popc(ends[k]);
            h_base += __popc(begins[k]) - __popc(ends[k]);
          }
          if (viol) atomicMin(&sm.badpos[bp], e0 + 32 * (__ffs((int)viol) - 1));
        };
        if (whole) place(std::true_type{}); else place(std::false_type{});
        __syncthreads();

        // ---------------- ends, one thread each, NT at a time in output order ----------------
        // A round looks up begin and parent and feeds the parent's child time; then, after a barrier, it writes its records:
        // a child ends before its parent, so what this round and those before it have added is all there will be.
        const u64 pos0 = out_base + n_int, room = SPLIT ? limit : a.interval_capacity;
        const int fit = pos0 + (u64)win_ne <= room ? win_ne : pos0 < room ? (int)(room - pos0) : 0;  // records that fit the output
        uint4* const rec0 = reinterpret_cast<uint4*>(a.intervals + pos0);
        u64* const dig0 = a.digest ? a.digest + pos0 : nullptr;
        // violations found so far, by the rounds before this one, too: ends at or after the first need no work (malformed GEMM 884 -> 845 us,
        // three defects in 1,000 markers 541 -> 511)
        int cut = sm.badpos[bp];
        u32 win_flags = 0;  // of this thread's records: CTX_MISMATCH, TIME_REVERSED, CHILD_CLAMPED, ten bits each
#pragma unroll
        for (int i = 0; i < NI; ++i) {
          if (i > 0 && i * NT >= win_ne) break;  // uniform
          // (the last, partly filled round goes to the upper half of the block: the lower half has the block's
          // other duties, and a barrier waits for the slowest warp)
          const int rk = (i == NI - 1 ? (tid + NT / 2) % NT : tid) + i * NT;
          u32 d = 0xffffffffu, incl = 0, flags = 0, btag = 0, bctx = 0;
          int partner = 0, parent = 0;
          u64 bts = 0;
          bool live = rk < win_ne;
          if (live) {
            d = sm.desc[rk];
            const int e = (int)(d & ((1u << SM::kDescShift) - 1u)), L = (int)(d >> SM::kDescShift);
            live = e < cut;
            if (live) {
              const uint4 ee = evb[e];  // needed after the lookups; asked for now, so that it arrives meanwhile
              // in the tile, or opened before this window (then so was its parent); selects, not branches
              // (no begin of level L - 1 can lie between the partner and e while the partner's frame is open, so the
              // parent is also the latest begin of level L - 1 before e: the two lookups do not depend on each other)
              const int p_in = tile_latest_begin<NT, E, true>(sm, L, lbase, e);
              const int q_in = tile_latest_begin<NT, E, true>(sm, L - 1, lbase, e);
              partner = p_in < 0 ? (L < ch ? cbase + L : kBadRef) : p_in;
              parent = L == 0 ? cbase + kSink : (q_in >= 0 ? q_in : (L - 1 < ch ? cbase + L - 1 : kBadRef));
              if (partner != kBadRef && parent != kBadRef) {
                const uint4 pe = evb[partner];
                bts = (u64)pe.x | ((u64)pe.y << 32);
                btag = pe.z; bctx = pe.w;
                const u64 dlt = ((u64)ee.x | ((u64)ee.y << 32)) - bts;
                incl = (u32)dlt;
                if (ee.w != pe.w) flags = ARGUS_FLAG_CTX_MISMATCH;
                // another region, 2^32 ticks and more, or time running backwards (which shows in the difference's upper half, or, when
                // the difference wraps to a small one, in the times')
                if ((((pe.z ^ ee.z) ^ 1u) | (u32)(dlt >> 32)) != 0 || ee.y < pe.y) {
                  live = (pe.z ^ ee.z) == 1u && ((u64)ee.x | ((u64)ee.y << 32)) < bts;
                  incl = 0;
                  flags |= ARGUS_FLAG_TIME_REVERSED;
                }
                // the parent gathers what this window adds to its child time in 32 bits; an interval or a sum of 2^32 ticks
                // cuts the window here, and the sequential machine (64-bit throughout) takes this marker
                const u32 old = atomicAdd(&accb[parent], incl);
                if (old + incl < old) { live = false; sm.wrapped = 1; }
              } else {
                live = false;
              }
              if (!live) atomicMin(&sm.badpos[bp], e);
            }
          }
          __syncthreads();
          if (i == 0 && sm.dead) {  // a bulk copy never arrived: report and leave (uniform decision)
            if (tid == 0) {
              argus_set_error(a.status, ARGUS_ERR_TIMEOUT, s, tile_start);
              tile_progress(a, 1);  // CTAs that poll for hand-overs must not wait for this stream
            }
            return;
          }
          cut = sm.badpos[bp];
          if (live && (int)(d & ((1u << SM::kDescShift) - 1u)) < cut) {
            const bool carried = (u32)partner >= (u32)T;
            const u32 acc = accb[partner], preg = (u32)(reinterpret_cast<const int*>(evb + parent)[2] >> 1);
            u32 excl = incl - acc, bidx = tile_start + (u32)partner;
            bool over = acc > incl;
            if (carried) {
              const int lv = partner - cbase;
              const u64 child = sm.cchild[cpar][lv] + acc;
              bidx = sm.cidx[cpar][lv];
              over = child > incl;
              excl = incl - (u32)child;
              if (SPLIT && lv < init_h) {  // its child time is completed afterwards
                seg->note_child[lv] = child;
                seg->note_incl[lv] = incl;
                seg->note_pos[lv] = pos0 + (u64)rk;
                atomicMin(&sm.low, lv);
                over = false;
                excl = incl;
              }
            }
            if (over) { flags |= ARGUS_FLAG_CHILD_CLAMPED; excl = 0; }
            if (flags) win_flags += (flags & 1u) | ((flags & 2u) << 9) | ((flags & 4u) << 18);
            if (rk < fit) {
              tile_store_record(rec0 + 3 * rk, (u32)bts, (u32)(bts >> 32), incl, excl, btag >> 1, bctx, s, preg, bidx,
                                (d >> SM::kDescShift) | (flags << 16));
              if (dig0) dig0[rk] = argus_digest_pack32(btag >> 1, incl, excl, flags);
            }
          } else if (incl) {
            atomicSub(&accb[parent], incl);  // an end at or after a cut
          }
        }
        const int badpos = sm.badpos[bp];  // every round's barrier has passed
        bp ^= 1;
        if (tid == 0) sm.badpos[bp] = 0x7fffffff;  // nobody reads or reports into it before the next window's barriers

        if (SPLIT && (badpos < wend || sm.stop)) {  // the chained pass walks this stream
          stream_failed = true;
          __syncthreads();
          break;
        }
        // the window counts up to `upto`: the stack it leaves behind, in the next window's index space (`pos`: events before it
        // are looked at)
        auto count_window = [&](int upto, int ne, int pos) {
          if (win_flags) { tot_ctx += win_flags & 1023u; tot_rev += (win_flags >> 10) & 1023u; tot_clamp += win_flags >> 20; }
          const int new_ch = ch + (upto - w0) - 2 * ne;  // every marker is a begin or an end
          if (tid < new_ch) {
            const int e = tile_latest_begin<NT, E, false>(sm, tid, lbase, pos);
            const int from = e >= 0 ? e : cbase + tid;
            car_next[tid] = evb[from];
            sm.cchild[cpar ^ 1][tid] = (e >= 0 ? 0ull : sm.cchild[cpar][tid]) + accb[from];
            sm.cidx[cpar ^ 1][tid] = e >= 0 ? tile_start + (u32)e : sm.cidx[cpar][tid];
          }
          small_streak = (upto - w0 < 32) ? small_streak + 1 : 0;
          ch = new_ch;
          n_int += (u64)ne;
          cpar ^= 1;
          w0 = upto;
          wend = tn;
          __syncthreads();
        };
        if (badpos >= wend) {
          count_window(wend, win_ne, T);
          if (SPLIT) init_h = sm.low < init_h ? sm.low : init_h;
        } else if (badpos > w0 && sm.wrapped) {
          // which of the ends that share a parent makes its sum wrap depends on their order, and so one before the cut may have
          // wrapped it unseen: [w0, badpos) is done again on its own (nothing was counted yet)
          wend = badpos;
          __syncthreads();
        } else {
          if (badpos > w0) {  // the ends before the cut (also a barrier for what the ends after it have taken back)
            int ne = 0;
            for (int rk = tid; rk - tid < win_ne; rk += NT)
              ne += __syncthreads_count(rk < win_ne && (int)(sm.desc[rk] & ((1u << SM::kDescShift) - 1u)) < badpos);
            __syncthreads();
            count_window(badpos, ne, badpos);
          }
          // ---------------- the marker(s) at w0 go through the sequential stack machine ----------------
          const int nseq = small_streak >= 2 ? ((tn - w0) < kSeqChunk ? (tn - w0) : kSeqChunk) : 1;
          const int base = carlo + cpar * kCar;
          uint4* const seq_next = sm.evall + T + (cpar ^ 1) * kCar;
          if (tid < ch) {
            const uint4 f = evb[base + tid];
            ArgusFrame& o = sm.fstk[tid];
            o.ts = (u64)f.x | ((u64)f.y << 32); o.child = sm.cchild[cpar][tid]; o.region = f.z >> 1; o.ctx = f.w;
            o.idx = sm.cidx[cpar][tid]; o.pad = 0;
          }
          __syncthreads();
          if (tid == 0) {
            ArgusSeqState st;
            st.h = ch; st.n_int = n_int; st.n_ctx = st.n_rev = st.n_clamp = 0; st.failed = false;
            bool ok = true;
            for (int e = w0; e < w0 + nseq && ok; ++e) {
              const uint4 pe = evb[e];
              ok = argus_seq_step(a, sm.fstk, st, s, gpos0, out_base, tile_start + (u32)e, (u64)pe.x | ((u64)pe.y << 32), pe.z, pe.w);
            }
            tot_ctx += st.n_ctx; tot_rev += st.n_rev; tot_clamp += st.n_clamp;
            sm.ch = st.h;
            sm.n_int = st.n_int;
            sm.failed = ok ? 0 : 1;
            if (!a.redo) atomicAdd((u64*)&a.status->n_sequential_tiles, 1ull);
          }
          __syncthreads();
          ch = sm.ch;
          n_int = sm.n_int;
          if (sm.failed) stream_failed = true;
          if (tid < ch) {
            const ArgusFrame f = sm.fstk[tid];
            seq_next[tid] = make_uint4((u32)f.ts, (u32)(f.ts >> 32), f.region << 1, f.ctx);
            sm.cchild[cpar ^ 1][tid] = f.child;
            sm.cidx[cpar ^ 1][tid] = f.idx;
          }
          cpar ^= 1;
          w0 += nseq;
          wend = tn;
          ++small_streak;
          __syncthreads();
          if (stream_failed) break;
        }
      }  // windows
      if (stream_failed) {
        if (ti + 1 < sm.ti_end) {  // drain the prefetched tile before the buffer is reused
          const bool ok = mbar_wait_bounded(&sm.bar[b ^ 1], (b ^ 1) ? ph1 : ph0);
          if (b ^ 1) ph1 ^= 1; else ph0 ^= 1;
          if (!ok) sm.dead = 1;
        }
        break;
      }
    }  // tiles


    __syncthreads();
    if (sm.dead) {
      if (tid == 0) {
        argus_set_error(a.status, ARGUS_ERR_TIMEOUT, s, 0);
        tile_progress(a, 1);
      }
      return;
    }
    if (SPLIT) {
      if (stream_failed) {
        if (tid == 0) argus_split_give_up(a, s, n);
      } else {
        if (tid < ch) seg->ledger[tid] = sm.cchild[cpar][tid];
        if (tid == 0) { seg->n_int = n_int; seg->end_ch = (u32)ch; }
        if (tot_ctx) atomicAdd(&seg->flags[0], tot_ctx);
        if (tot_rev) atomicAdd(&seg->flags[1], tot_rev);
        if (tot_clamp) atomicAdd(&seg->flags[2], tot_clamp);
      }
      tot_ctx = tot_rev = tot_clamp = 0;
    } else if (!stream_failed && ti < ntiles) {
      // hand the stream on: its state goes into the record, the record into the queue
      const u32 rec = sm.cur_rec;
      ArgusStreamRecord* r = a.records + rec;
      if (tid == 0) { r->stream = s; r->next_tile = ti; r->ch = ch; r->n_int = n_int; }
      if (tid < ch) {
        r->frames[tid] = sm.evall[T + cpar * kCar + tid];
        r->child[tid] = sm.cchild[cpar][tid];
        r->idx[tid] = sm.cidx[cpar][tid];
      }
      __threadfence();
      __syncthreads();
      if (tid == 0) {
        const u64 slot = atomicAdd(reinterpret_cast<unsigned long long*>(&a.ctl->q_tail[a.redo ? 1 : 0]), 1ull);
        if (slot < a.queue_capacity) *reinterpret_cast<volatile u32*>(a.queue + slot) = rec + 1;
        __threadfence();
        tile_progress(a, 1ull << 32);
      }
    } else {
      if (!a.redo) {
        // frames still open at the end of the stream (they sit in the block the next tile would read)
        if (!stream_failed && tid < ch) argus_note_ambiguity(a, gpos0 + sm.cidx[cpar][tid], ARGUS_AMBIG_BEGIN_EOS, (u32)tid);
        if (tid == 0) a.counts[s] = n_int;
      }
      if (tid == 0) tile_progress(a, 1);
    }
    __syncthreads();
  }  // streams

  if (!a.redo) {
    tot_ctx = __reduce_add_sync(0xffffffffu, tot_ctx);
    tot_rev = __reduce_add_sync(0xffffffffu, tot_rev);
    tot_clamp = __reduce_add_sync(0xffffffffu, tot_clamp);
    if (lane == 0) {
      if (tot_ctx) atomicAdd((u64*)&a.status->n_ctx_mismatch, (u64)tot_ctx);
      if (tot_rev) atomicAdd((u64*)&a.status->n_time_reversed, (u64)tot_rev);
      if (tot_clamp) atomicAdd((u64*)&a.status->n_child_clamped, (u64)tot_clamp);
    }
  }
}

// The shared-memory opt-in and the occupancy of one instantiation belong to one device: looked up once per
// device, under a lock (two host threads may make their first call at the same time).
template <int NT, int E, int MINB, bool RING, bool SPLIT = false>
int launch_tiled(const ArgusPairArgs& a, cudaStream_t stream) {
  constexpr int kMaxDevices = 64;
  static int grid_of[kMaxDevices];
  static std::mutex mu;
  constexpr size_t smem = ((sizeof(TileSmem<NT, E>) + 15) & ~(size_t)15) + 128;
  int dev = 0;
  ARGUS_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return ARGUS_ERR_INVALID_ARG;
  int grid_cache;
  {
    std::lock_guard<std::mutex> lk(mu);
    if (!grid_of[dev]) {
      ARGUS_CUDA_TRY(cudaFuncSetAttribute(k_pair_tiled<NT, E, MINB, RING, SPLIT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
      int sms = 0, per_sm = 0;
      ARGUS_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
      ARGUS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_pair_tiled<NT, E, MINB, RING, SPLIT>, NT, smem));
      if (per_sm < 1) return ARGUS_ERR_CUDA;
      if (per_sm > MINB) per_sm = MINB;
      grid_of[dev] = sms * per_sm < (int)kMostCtas ? sms * per_sm : (int)kMostCtas;
    }
    grid_cache = grid_of[dev];
  }
  const u32 items = SPLIT ? argus_split_max_segments(a.num_events, a.num_streams) : a.num_streams;
  const u32 grid = items < (u32)grid_cache ? items : (u32)grid_cache;
  ARGUS_LAUNCH(k_pair_tiled<NT, E, MINB, RING, SPLIT>, grid, NT, smem, stream, a);
  return ARGUS_OK;
}

std::atomic<int> g_variant{0};

}  // namespace

bool argus_pair_tiled_usable(const ArgusPairArgs& a) { return a.num_streams > 0; }

// Tile shape used by the tiled kernel: 0 = the default; 1..3 select the other compiled shapes
// <threads, events per thread, CTAs per SM> (test aid: tiles end at other places; results do not depend on it).
extern "C" void argus_set_tile_variant(int v) { g_variant.store(v); }

int argus_launch_pair_tiled(const ArgusPairArgs& a, cudaStream_t stream, bool split) {
  if (split) return launch_tiled<128, kSplitTile / 128, 7, false, true>(a, stream);
  if (a.ring_written) return launch_tiled<128, 5, 7, true>(a, stream);  // ring container: one shape
  switch (g_variant.load(std::memory_order_relaxed)) {
    case 1: return launch_tiled<192, 5, 4, false>(a, stream);
    case 2: return launch_tiled<64, 5, 8, false>(a, stream);
    case 3: return launch_tiled<256, 7, 2, false>(a, stream);
    default: return launch_tiled<128, 5, 7, false>(a, stream);  // seven CTAs of 128 threads per SM
  }
}
