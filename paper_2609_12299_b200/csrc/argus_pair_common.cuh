// argus_pair_common.cuh — the sequential per-stream stack machine (exact semantics) and the
// ambiguity side channel used by every pairing kernel.
//
// Ambiguity records cannot be written in final order in one pass: whether a begin ends up
// force-closed or open at end of stream is only known later. The pairing kernels therefore
//   (1) append a packed note {global event position, kind, depth} to an unordered list, and
//   (2) set the event's bit in a bitmap over all events;
// afterwards a rank query on the bitmap (popcount prefix) gives every note its slot in
// (stream, event index) order, and stream_offsets give ambig_offsets.
#ifndef ARGUS_PAIR_COMMON_CUH_
#define ARGUS_PAIR_COMMON_CUH_

#include "argus_common.cuh"
#include "argus_fuse.cuh"

struct ArgusFrame {  // one open region occurrence, 32 bytes
  u64 ts;
  u64 child;  // inclusive time of matched intervals directly below
  u32 region;
  u32 ctx;
  u32 idx;  // index of the begin marker within its stream
  u32 pad;
};

// Control block in the workspace, zeroed at the start of a call. A word that many blocks change while others look at it is looked at with
// an atomic, too, and lies on a line with nothing that is read in any other way: loads of a line that changes all the time held
// up everything else that half of the SMs asked the L2 for (2,368 streams of 16,208 events, blocks that load `level` every 3,840: 69 SMs walked
// 340 tiles each, the others 485, in 435 us; with atomics 416 each, in 340).
constexpr u32 kMostCtas = 2048;  // of the tiled kernel
struct ArgusPairCtl {
  // written by one kernel, read by the next
  u32 redo;            // 1 = provisional interval bases were wrong; second pass needed
  u32 redo_from;       // first stream whose intervals the second pass writes again
  u64 total_intervals;
  u64 total_ambig;
  u32 longest;         // events of the longest stream
  u32 prefix_done;     // blocks that have counted their share of the ambiguity bitmap
  u32 recount_head;    // streams taken to have their markers counted
  u32 recount_done;    // blocks that have found no more of them
  // atomics only
  alignas(128) u64 n_notes;  // ambiguity notes appended (may exceed the list capacity)
  // work queue of the tiled kernel, one set per pass (0 = first, 1 = redo): positions below num_streams are the
  // streams themselves, later positions are streams handed on after a chunk (see ArgusStreamRecord)
  u64 q_head[2];       // positions taken behind those that CTAs start with
  u64 q_tail[2];       // hand-overs published (queue entries written)
  u64 progress[2];     // low half: streams walked to their end (or given up on); high half: moves as long as streams are walked
  u32 level[2];        // events left of the stream that was taken last, 0 if nothing else waits
  u32 seg_head;        // segments taken (split pass)
  u32 claimed_words[2];  // words of `claimed` of which every position has been claimed
  // read by all blocks, changed when something is given up
  alignas(128) u32 num_failed;  // streams that the split pass has to leave to the chained one (read together with the next two)
  u32 num_segments;    // 0 where the segments do not fit their room, too
  u32 split;           // the split pass is worth it (argus_split_pays), and no long stream has been given up
  u32 pad;
  // atomics only: positions that CTAs start with, a bit each, a sector for a word (all CTAs claim at once)
  alignas(128) u32 claimed[2][kMostCtas / 32][8];
};

// A stream is a chain of tiles that one CTA at a time walks, and streams rarely share out evenly among the CTAs that the chip holds.
// So a CTA looks up now and then how much the stream that was taken last had left (ArgusPairCtl::level). If its own has less than half
// of that left it hands it on: it stores the stream's state here, puts the record into the work queue and takes the next
// position; whichever CTA is free when the record's turn comes carries on. Streams are taken longest first and what is handed
// on is about as long as what is taken for it, so what was taken last tells well enough what waits, and the streams that
// are left get shorter together. A hand-over costs the CTA about 8 us (it waits for its stores, then for a chain of loads), which
// is why it is not done for a little. Where nothing waits nothing is handed on. Hand-overs every 32,768 events, whatever waited, made
// long streams wait behind short ones, and left half of the CTAs idle for the last eighth of the time: GEMM trace (68.7 M events in streams
// of 72,000 and 32,000) 622 -> 571 us, attention (153.5 M in 112,684, 67,628 and 176) 1,412 -> 1,246, 131 x 12 streams (27,972 and
// 12,432) 244 -> 203, equal streams (2,368 of 129,664) 2,421 -> 2,442; looked up by three quarters instead of a half 576, 1,256 and 2,468.
// Positions are only ever taken by CTAs that run (tile_pop_work): other kernels may hold part of the chip, and nothing may wait for a CTA that
// has not started. So a CTA whose position has no entry yet is idle anyway (every unfinished stream is in a running CTA's hands):
// it polls until the entry appears or every stream is done, and gives up with ARGUS_ERR_TIMEOUT if nothing moves for about a second.
constexpr u32 kChunkEvents = 3840;   // walked by a CTA at least before it hands a stream on
constexpr u32 kLevelMargin = 1280;   // by which the stream has to have less left than half
constexpr u32 kLeastTiles = 3;       // and what is less than this is walked at once
struct ArgusStreamRecord {
  u32 stream, next_tile;
  int ch;                             // stack height at the hand-over
  u32 pad;
  u64 n_int;                          // intervals emitted so far
  uint4 frames[ARGUS_MAX_DEPTH];      // open begin markers as event records
  u64 child[ARGUS_MAX_DEPTH];         // their child time so far
  u32 idx[ARGUS_MAX_DEPTH];           // their index within the stream
};

// Few long streams: a stream is cut into segments that are walked at the same time (argus_pair_split.cu). What a segment
// needs to know and what it leaves behind.
struct ArgusSegment {
  u32 stream, first_tile, num_tiles;
  int ch;                             // frames open where it starts
  u32 unmatched_ends, unmatched_begins;  // by height, within the segment
  u32 flags[3];                       // intervals with CTX_MISMATCH, TIME_REVERSED, CHILD_CLAMPED
  u32 end_ch;                         // frames open where it ends
  u64 n_int;                          // intervals of the stream up to its end
  u32 idx[ARGUS_MAX_DEPTH];           // the open frames' begin markers, by level
  u32 open[ARGUS_MAX_DEPTH];          // the segment's unmatched begins, innermost first; of the stream's last segment, in the
                                      // end, the frames open at the end of the stream by level
  u64 ledger[ARGUS_MAX_DEPTH];        // child time that the segment gave to the frames open at its end, by level
  u64 note_pos[ARGUS_MAX_DEPTH];      // record of the initial frame of a level that the segment closed (~0: none): its child time
  u64 note_child[ARGUS_MAX_DEPTH];    // lacks what earlier segments gave it; what this one gave
  u64 note_incl[ARGUS_MAX_DEPTH];     // its inclusive time
};

struct ArgusPairArgs {
  const argus_event_t* events;
  const u64* stream_offsets;
  u64 num_events;
  u32 num_streams;
  u32 num_regions;
  argus_interval_t* intervals;
  u64 interval_capacity;
  u64* interval_offsets;  // final offsets (output of the offsets kernel)
  u64* counts;            // per-stream interval counts (workspace)
  u64* bases;             // [S + 1] provisional first interval of every stream: the sum of the counts foretold for those before it
  u64* notes;             // packed ambiguity notes (workspace)
  u64 note_capacity;
  u32* bits;              // one bit per event (workspace)
  ArgusPairCtl* ctl;
  argus_status_t* status;
  int redo;               // 0 = first pass with provisional bases, 1 = second pass with final bases (streams from ctl->redo_from on)
  u32* queue;             // hand-over queue entries (record index + 1; zeroed), null = streams are never split
  u64 queue_capacity;
  ArgusStreamRecord* records;
  u32 record_capacity;
  const u32* order;       // streams in the order in which the tiled kernel starts them: longest first (null = by index)
  u64* digest;            // one digest per interval record, same positions (null = none); interval_capacity is then no larger than
                          // what it holds
  const u64* ring_written; // non-null: `events` is a ring container, one slot of ring_capacity records per stream, record i of
  u32 ring_capacity;       // a stream at slot position i mod capacity; stream_offsets then describe the packed survivors
  ArgusSegment* segments;  // non-null: split pass; or, in the chained pass after it, what that left: only failed streams are walked
  u32* split_failed;       // [S]
  u32 segment_tiles;       // tiles of a segment
  u32 poll_limit;          // polls without any movement (ArgusPairCtl::progress) after which an idle CTA gives up (about a second)
  u32 hand_on;             // hand on at every look (a test)
};

// argus_pair_split.cu
constexpr u32 kSplitTile = 640;  // events of a tile of the split pass
bool argus_split_usable(uint64_t num_events, uint32_t num_streams);
uint32_t argus_split_max_segments(uint64_t num_events, uint32_t num_streams);
size_t argus_split_bytes(uint64_t num_events, uint32_t num_streams);
int argus_launch_pair_split(ArgusPairArgs& a, void* room, cudaStream_t stream);
// Is the split pass the faster one for streams of which the longest has `longest` events? The chained pass takes 4.05 ns an event of the
// longest stream with a stream on an SM and 0.75 ns more for each further one; the split pass 85 events a ns and 35 us more than the
// chained one with the split kernels launched for nothing (12 us). Measured (us, split / chained by itself; streams x events): decode
// trace, equal lengths, 96 x 12,156 71 / 66, 96 x 32,416 89 / 143, 320 x 12,156 103 / 90, 320 x 32,416 183 / 197, 448 x 32,416 239 /
// 209, 448 x 129,664 689 / 762, 512 x 32,416 259 / 211, 512 x 518,656 2,739 / 2,923, 592 x 518,656 3,231 / 3,005, 768 x 32,416 359 / 271;
// GEMM trace, two of twelve streams 2.3 times as long as the others, longest 25,200 of 288 99 / 140, of 768 181 / 213, longest 72,000 of
// 768 390 / 443.
__host__ __device__ __forceinline__ bool argus_split_pays(u32 longest, u64 num_events, u32 num_streams) {
  const u32 per_sm = (num_streams + 147) / 148;
  return (u64)longest * (280 + 64 * per_sm) > num_events + 3000000;  // both sides in 1 / 85 ns
}

// After the split pass: are its segments what counts, or is everything left to the chained pass? *failed: has a stream been given up?
__device__ __forceinline__ bool argus_split_in_force(const ArgusPairArgs& a, bool* failed) {
  const uint4 w = __ldcg(reinterpret_cast<const uint4*>(&a.ctl->num_failed));
  *failed = w.x != 0;
  return w.y && w.z;
}

// Gives a stream of `length` events up. The chained pass takes about as long for one long stream as for all of them, so one
// that is about as long as the longest takes all others with it. One thread.
__device__ __forceinline__ void argus_split_give_up(const ArgusPairArgs& a, u32 s, u32 length) {
  if (atomicExch(a.split_failed + s, 1u)) return;
  if (argus_split_pays(__ldcg(&a.ctl->longest) - length, a.num_events, a.num_streams)) atomicAdd(&a.ctl->num_failed, 1u);
  else atomicExch(&a.ctl->split, 0u);
}

// The markers of a stream are counted in rounds of kRecountStep. A stream may hold up to 2^32 - 1 markers, so the end of the last
// round need not fit 32 bits, and no loop may run up to it.
constexpr u32 kRecountStep = 32768;
__host__ __device__ constexpr u32 argus_recount_rounds(u32 n) { return n / kRecountStep + (n % kRecountStep != 0); }
__host__ __device__ constexpr u32 argus_recount_markers(u32 n, u32 round) {  // of that round
  return n - round * kRecountStep < kRecountStep ? n - round * kRecountStep : kRecountStep;
}

#define ARGUS_NOTE_POS_BITS 48

// Ring container: slot position of the oldest surviving record of stream s.
__device__ __forceinline__ u32 argus_ring_first(const ArgusPairArgs& a, u32 s) {
  const u64 w = a.ring_written[s];
  return w > a.ring_capacity ? (u32)(w % a.ring_capacity) : 0u;
}

__device__ __forceinline__ void argus_note_ambiguity(const ArgusPairArgs& a, u64 gpos, u32 kind, u32 depth) {
  const u64 slot = atomicAdd(&a.ctl->n_notes, 1ull);
  if (slot < a.note_capacity) a.notes[slot] = gpos | ((u64)kind << ARGUS_NOTE_POS_BITS) | ((u64)depth << (ARGUS_NOTE_POS_BITS + 2));
  atomicOr(&a.bits[gpos >> 5], 1u << (gpos & 31));
}

__device__ __forceinline__ void argus_store_interval(argus_interval_t* dst, u64 t_begin, u64 incl, u64 excl, u32 region,
                                                     u32 ctx, u32 stream, u32 parent, u32 begin_idx, u32 depth, u32 flags) {
  uint4* p = reinterpret_cast<uint4*>(dst);
  p[0] = make_uint4((u32)t_begin, (u32)(t_begin >> 32), (u32)incl, (u32)(incl >> 32));
  p[1] = make_uint4((u32)excl, (u32)(excl >> 32), region, ctx);
  p[2] = make_uint4(stream, parent, begin_idx, (depth & 0xffffu) | (flags << 16));
}

// Per-stream running state of the sequential machine.
struct ArgusSeqState {
  int h;            // stack height
  u64 n_int;        // intervals emitted so far in this stream
  u32 n_ctx, n_rev, n_clamp;  // flag counters (flushed by the caller)
  bool failed;
};

// Processes one event exactly as the definition states. `stk` holds ARGUS_MAX_DEPTH frames.
// `out_base` is the position of this stream's first interval. Returns false on a device error.
__device__ __forceinline__ bool argus_seq_step(const ArgusPairArgs& a, ArgusFrame* stk, ArgusSeqState& s, u32 stream,
                                               u64 stream_gpos0, u64 out_base, u32 i, u64 ts, u32 tag, u32 ctx) {
  const u32 region = tag >> 1;
  if (region >= a.num_regions) {
    argus_set_error(a.status, ARGUS_ERR_BAD_REGION, stream, i);
    return false;
  }
  if (!(tag & 1u)) {
    if (s.h == ARGUS_MAX_DEPTH) {
      argus_set_error(a.status, ARGUS_ERR_DEPTH, stream, i);
      return false;
    }
    ArgusFrame& f = stk[s.h++];
    f.ts = ts; f.child = 0; f.region = region; f.ctx = ctx; f.idx = i;
    return true;
  }
  int k = s.h - 1;
  while (k >= 0 && stk[k].region != region) --k;
  if (k < 0) {
    if (!a.redo) argus_note_ambiguity(a, stream_gpos0 + i, ARGUS_AMBIG_UNMATCHED_END, (u32)s.h);
    return true;
  }
  u64 moved = 0;
  while (s.h - 1 > k) {  // force-close mis-nested frames; their child time moves down the stack
    const ArgusFrame& f = stk[--s.h];
    if (!a.redo) argus_note_ambiguity(a, stream_gpos0 + f.idx, ARGUS_AMBIG_BEGIN_MISNESTED, (u32)s.h);
    moved += f.child;
  }
  const ArgusFrame f = stk[--s.h];
  const u64 child = f.child + moved;
  u32 flags = 0;
  u64 incl, excl;
  if (ctx != f.ctx) { flags |= ARGUS_FLAG_CTX_MISMATCH; s.n_ctx++; }
  if (ts < f.ts) { incl = 0; flags |= ARGUS_FLAG_TIME_REVERSED; s.n_rev++; } else { incl = ts - f.ts; }
  if (child > incl) { excl = 0; flags |= ARGUS_FLAG_CHILD_CLAMPED; s.n_clamp++; } else { excl = incl - child; }
  const u64 pos = out_base + s.n_int;
  if (pos < a.interval_capacity) {
    argus_store_interval(a.intervals + pos, f.ts, incl, excl, f.region, f.ctx, stream,
                         s.h > 0 ? stk[s.h - 1].region : ARGUS_NONE, f.idx, (u32)s.h, flags);
    if (a.digest) a.digest[pos] = argus_digest_pack(f.region, incl, excl, flags);
  }
  s.n_int++;
  if (s.h > 0) stk[s.h - 1].child += incl;
  return true;
}

// End of stream: every open frame becomes a BEGIN_EOS note.
__device__ __forceinline__ void argus_seq_finish(const ArgusPairArgs& a, const ArgusFrame* stk, const ArgusSeqState& s,
                                                 u64 stream_gpos0) {
  if (a.redo) return;
  for (int k = 0; k < s.h; ++k) argus_note_ambiguity(a, stream_gpos0 + stk[k].idx, ARGUS_AMBIG_BEGIN_EOS, (u32)k);
}

__device__ __forceinline__ void argus_flush_flag_counters(const ArgusPairArgs& a, const ArgusSeqState& s) {
  if (a.redo) return;
  if (s.n_ctx) atomicAdd((u64*)&a.status->n_ctx_mismatch, (u64)s.n_ctx);
  if (s.n_rev) atomicAdd((u64*)&a.status->n_time_reversed, (u64)s.n_rev);
  if (s.n_clamp) atomicAdd((u64*)&a.status->n_child_clamped, (u64)s.n_clamp);
}

#endif  // ARGUS_PAIR_COMMON_CUH_
