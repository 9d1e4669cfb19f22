// argus_pair_split.cu — few long streams: pairing of the segments of a stream at the same time.
//
// A stream is a chain: what a marker means depends on the stack that everything before it leaves. With fewer streams than the
// chip has room for blocks (a trace of some of the SMs) the chained pass leaves most of it idle. Here
//   k_split_scan  : one block per segment reads the markers' kinds only and finds, by heights, how many ends close a frame from
//                   before the segment and which begins stay open at its end;
//   k_split_chain : one block per stream; its first warp walks the segments, whose summaries the block brings into shared memory,
//                   and gives every one the stack where it starts;
//   (the SPLIT instantiation of the tiled kernel walks the segments: argus_pair_tiled.cu)
//   k_split_fix   : several blocks per stream complete the child time of the frames that were open across a segment's start; the
//                   first of them counts the stream's intervals and notes the frames open at its end.
// Heights know nothing of region ids. A segment that meets a marker which breaks the parallel rules gives its stream up; the
// chained pass, which follows and does nothing otherwise, walks such streams from their beginning. A stream about as long as the
// longest takes all others with it, and the blocks stop within eight tiles (384 streams of 129,664 events with a lost or doubled
// marker in two of three: 1,922 us when they went on, 1,582 us; 1,385 in the chained passes by themselves).
//
// The scan reads the events once more (16 of then 56 bytes an event). 96 streams of 518,656 events: pairing 2,412 -> 660 us
// (scan 132, chain 29, segments 450, fix 22; 36 and 27 for chain and fix with a warp and a block a stream).
#include "argus_internal.cuh"
#include "argus_pair_common.cuh"

namespace {

constexpr int kScanThreads = 256;
constexpr int kFixThreads = 512;
constexpr u32 kRun = 32;  // consecutive events a thread looks at
constexpr u32 kBlockEvents = kScanThreads * kRun;

__device__ __forceinline__ u32 split_length(const ArgusPairArgs& a, u32 s) {
  const u64 off0 = a.stream_offsets[0], lo = a.stream_offsets[s], hi = a.stream_offsets[s + 1];
  return hi < lo || hi > a.num_events || lo < off0 || ((hi - lo) >> 32) ? 0u : (u32)(hi - lo);
}
__device__ __forceinline__ u32 split_segments(const ArgusPairArgs& a, u32 s) {  // an empty or bad stream has one, of no tiles
  const u64 per = (u64)a.segment_tiles * kSplitTile, n = split_length(a, s);
  return n ? (u32)((n + per - 1) / per) : 1u;
}

__global__ void __launch_bounds__(kScanThreads) k_split_scan(ArgusPairArgs a, u32* first_segment) {
  argus_kernel_begin();
  const u32 split = __ldcg(&a.ctl->split);
  __shared__ u32 sh[33], sh_stream, sh_before;
  __shared__ int shi[33], low_of[kScanThreads / 32];
  const u32 tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // the block's segment: streams' segments one after the other
  if (tid == 0) sh_stream = 0xffffffffu;
  __syncthreads();
  u32 carry = 0;
  for (u32 s0 = 0; s0 < a.num_streams; s0 += kScanThreads) {
    const u32 s = s0 + tid, c = s < a.num_streams ? split_segments(a, s) : 0u;
    u32 total;
    const u32 ex = carry + argus_block_exclusive_scan<u32>(c, sh, &total);
    if (blockIdx.x == 0 && s < a.num_streams) { first_segment[s] = ex; a.split_failed[s] = 0; }
    if (blockIdx.x >= ex && blockIdx.x < ex + c) { sh_stream = s; sh_before = ex; }
    carry += total;
  }
  __syncthreads();
  // No segments where the chained pass is the faster one. Offsets that decrease let streams share events, and then there may be more
  // segments than blocks and room: the chained pass, which reports such offsets, walks all streams.
  if (!split || carry > gridDim.x) return;
  if (blockIdx.x == 0 && tid == 0) { first_segment[a.num_streams] = carry; a.ctl->num_segments = carry; }
  if (sh_stream == 0xffffffffu) return;
  const u32 s = sh_stream, j = blockIdx.x - sh_before, n = split_length(a, s), per = a.segment_tiles * kSplitTile;
  ArgusSegment* const g = a.segments + blockIdx.x;
  const u32 start = j * per, count = n - start < per ? n - start : per;
  const uint4* const src = reinterpret_cast<const uint4*>(a.events + a.stream_offsets[s]) + start;
  // from the last event back: a begin without an end behind it goes below every height so far
  int height = 0, lowest = 0;
  for (u32 i0 = 0; i0 < count; i0 += kBlockEvents) {
    u32 ends = 0;  // bit j: event i0 + (32 tid + j) from the end is an end
    const u32 w0 = i0 + warp * 32 * kRun;
#pragma unroll 16
    for (u32 r = 0; r < kRun; ++r) {
      const u32 i = w0 + r * 32 + lane;
      const u32 tag = i < count ? __ldg(reinterpret_cast<const u32*>(src + (count - 1 - i)) + 2) : 0u;
      const u32 b = __ballot_sync(0xffffffffu, tag & 1u);
      if (lane == r) ends = b;
    }
    const u32 mine = i0 + tid * kRun, have = mine < count ? (count - mine < kRun ? count - mine : kRun) : 0u;
    const u32 begins = have ? ~ends & (0xffffffffu >> (32 - have)) : 0u;
    int total;
    const int h0 = height + argus_block_exclusive_scan<int>(__popc(ends) - __popc(begins), shi, &total);
    int h = h0, low = h0;
#pragma unroll
    for (u32 r = 0; r < kRun; ++r) {
      h += (int)((ends >> r) & 1u) - (int)((begins >> r) & 1u);
      low = h < low ? h : low;
    }
    int upto = low;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) { const int o = __shfl_up_sync(0xffffffffu, upto, d); if (lane >= (u32)d && o < upto) upto = o; }
    if (lane == 31) low_of[warp] = upto;
    __syncthreads();
    int before = __shfl_up_sync(0xffffffffu, upto, 1);
    if (lane == 0 || before > lowest) before = lowest;
    int all = lowest;
    for (u32 w = 0; w < kScanThreads / 32; ++w) {
      const int o = low_of[w];
      if (w < warp && o < before) before = o;
      if (o < all) all = o;
    }
    if (low < before) {
      h = h0;
      for (u32 r = 0; r < kRun; ++r) {
        h += (int)((ends >> r) & 1u) - (int)((begins >> r) & 1u);
        if (h < before) {
          before = h;
          if (-h <= ARGUS_MAX_DEPTH) g->open[-h - 1] = start + (count - 1 - (mine + r));
        }
      }
    }
    lowest = all;
    height += total;
    __syncthreads();
  }
  if (tid < ARGUS_MAX_DEPTH) g->note_pos[tid] = ~0ull;
  if (tid < 3) g->flags[tid] = 0;
  if (tid == 0) {
    g->stream = s; g->first_tile = j * a.segment_tiles; g->num_tiles = (count + kSplitTile - 1) / kSplitTile;
    g->unmatched_begins = (u32)-lowest;
    g->unmatched_ends = (u32)(height - lowest);
  }
}

// The summaries of up to kChainBatch segments come into shared memory at once; then one warp goes through them, a round of shared
// memory per segment (96 streams of 32 segments: 37 us when that warp asked for them itself, four segments ahead, 29 us, of which 20 pass beside the
// end of the scan).
constexpr u32 kChainThreads = 256, kChainBatch = 64;
__global__ void __launch_bounds__(kChainThreads) k_split_chain(ArgusPairArgs a, const u32* first_segment) {
  argus_kernel_begin_long();
  static_assert(ARGUS_MAX_DEPTH == 64, "two levels a lane");
  __shared__ u32 stack[ARGUS_MAX_DEPTH];
  __shared__ u32 ends[kChainBatch], begins[kChainBatch], open[kChainBatch][ARGUS_MAX_DEPTH];
  const u32 s = blockIdx.x, lane = threadIdx.x;
  if (!__ldcg(&a.ctl->num_segments)) return;  // all streams are left
  const u32 g0 = first_segment[s], g1 = first_segment[s + 1];
  int h = 0;
  bool fail = false;
  for (u32 k0 = g0; k0 < g1; k0 += kChainBatch) {
    const u32 have = g1 - k0 < kChainBatch ? g1 - k0 : kChainBatch;
    const ArgusSegment* const from = a.segments + k0;
    for (u32 i = threadIdx.x; i < have * ARGUS_MAX_DEPTH; i += kChainThreads) open[i / ARGUS_MAX_DEPTH][i % ARGUS_MAX_DEPTH] = __ldcg(from[i / ARGUS_MAX_DEPTH].open + i % ARGUS_MAX_DEPTH);
    for (u32 i = threadIdx.x; i < have; i += kChainThreads) { ends[i] = __ldcg(&from[i].unmatched_ends); begins[i] = __ldcg(&from[i].unmatched_begins); }
    __syncthreads();
    for (u32 i = 0; lane < 32 && i < have && !fail; ++i) {
      ArgusSegment* const g = a.segments + k0 + i;
      const int ue = (int)ends[i], ub = (int)begins[i], low = h - ue;
      if ((int)lane < h) g->idx[lane] = stack[lane];
      if ((int)lane + 32 < h) g->idx[lane + 32] = stack[lane + 32];
      if (lane == 0) g->ch = h;
      if (low < 0 || ub > ARGUS_MAX_DEPTH || low + ub > ARGUS_MAX_DEPTH) { fail = true; break; }
      __syncwarp();
      if ((int)lane < ub) stack[low + ub - 1 - (int)lane] = open[i][lane];
      if ((int)lane + 32 < ub) stack[low + ub - 1 - (int)lane - 32] = open[i][lane + 32];
      h = low + ub;
      __syncwarp();
      if (k0 + i + 1 == g1) {
        if ((int)lane < h) g->open[lane] = stack[lane];
        if ((int)lane + 32 < h) g->open[lane + 32] = stack[lane + 32];
      }
    }
    __syncthreads();
  }
  if (fail && lane == 0) argus_split_give_up(a, s, split_length(a, s));
}

__global__ void __launch_bounds__(kFixThreads) k_split_fix(ArgusPairArgs a, const u32* first_segment, u32 parts) {
  argus_kernel_begin_long();
  const u32 s = blockIdx.x / parts, part = blockIdx.x % parts;  // (blocks that share a stream: a frame a thread)
  bool any_failed;
  if (!argus_split_in_force(a, &any_failed) || (any_failed && __ldcg(a.split_failed + s))) return;
  const u32 g0 = first_segment[s], g1 = first_segment[s + 1], per = a.segment_tiles * kSplitTile;
  const u64 off0 = a.stream_offsets[0];
  u32 ctx = 0, rev = 0, clamp = 0;
  const u64 limit = a.bases[s + 1] < a.interval_capacity ? a.bases[s + 1] : a.interval_capacity;
  for (u32 i = part * kFixThreads + threadIdx.x; i < (g1 - g0) * ARGUS_MAX_DEPTH; i += parts * kFixThreads) {
    const u32 k = g0 + i / ARGUS_MAX_DEPTH, l = i % ARGUS_MAX_DEPTH;
    const ArgusSegment* const g = a.segments + k;
    if (l == 0) { ctx += g->flags[0]; rev += g->flags[1]; clamp += g->flags[2]; }
    const u64 pos = g->note_pos[l];
    if (pos == ~0ull) continue;
    u64 child = g->note_child[l];
    const u64 incl = g->note_incl[l];
#pragma unroll 4
    for (u32 q = g0 + g->idx[l] / per; q < k; ++q) child += a.segments[q].ledger[l];
    const bool clamped = child > incl;
    clamp += clamped;
    if (pos >= limit) continue;  // not written: such a stream is written by the second pass
    argus_interval_t* const r = a.intervals + pos;
    const u32 flags = r->flags | (clamped ? ARGUS_FLAG_CHILD_CLAMPED : 0u);
    const u64 excl = clamped ? 0 : incl - child;
    r->exclusive = excl;
    r->flags = (uint16_t)flags;
    if (a.digest) a.digest[pos] = argus_digest_pack(r->region, incl, excl, flags);
  }
  if (ctx) atomicAdd((u64*)&a.status->n_ctx_mismatch, (u64)ctx);
  if (rev) atomicAdd((u64*)&a.status->n_time_reversed, (u64)rev);
  if (clamp) atomicAdd((u64*)&a.status->n_child_clamped, (u64)clamp);
  if (part) return;
  const u32 n = split_length(a, s);
  const ArgusSegment* const last = a.segments + (g1 - 1);
  if (threadIdx.x == 0) a.counts[s] = n ? last->n_int : 0;
  if (n && threadIdx.x < last->end_ch) argus_note_ambiguity(a, a.stream_offsets[s] - off0 + last->open[threadIdx.x], ARGUS_AMBIG_BEGIN_EOS, threadIdx.x);
}

}  // namespace

// Fewer streams than three quarters of the blocks of the pairing kernel that run at a time (7 x 148), and long ones: the chained
// pass would leave the rest of the chip idle. Whether that outweighs the scan is decided on the device, by the longest stream.
bool argus_split_usable(uint64_t num_events, uint32_t num_streams) {
  return num_streams > 0 && num_streams < 777 && num_events > (1u << 20) && num_events / num_streams >= 16 * kSplitTile;
}

static u32 split_tiles(uint64_t num_events) {  // about three segments for every block that runs at a time, of 8 tiles at least
  const u64 tiles = (num_events / 3072 + kSplitTile - 1) / kSplitTile;
  return (u32)(tiles < 8 ? 8 : tiles);
}

uint32_t argus_split_max_segments(uint64_t num_events, uint32_t num_streams) {
  return (u32)(num_events / ((u64)split_tiles(num_events) * kSplitTile)) + num_streams;
}

size_t argus_split_bytes(uint64_t num_events, uint32_t num_streams) {
  if (!argus_split_usable(num_events, num_streams)) return 0;
  return argus_align_up((size_t)argus_split_max_segments(num_events, num_streams) * sizeof(ArgusSegment), 256) +
         argus_align_up(((size_t)num_streams + 1) * 4, 256) + argus_align_up((size_t)num_streams * 4, 256);
}

int argus_launch_pair_tiled(const ArgusPairArgs& a, cudaStream_t stream, bool split);

// The whole split pass; `room` holds argus_split_bytes(). Leaves a.segments and a.split_failed set for the chained pass.
int argus_launch_pair_split(ArgusPairArgs& a, void* room, cudaStream_t stream) {
  const u32 most = argus_split_max_segments(a.num_events, a.num_streams);
  char* w = (char*)room;
  a.segments = (ArgusSegment*)w;
  w += argus_align_up((size_t)most * sizeof(ArgusSegment), 256);
  u32* const first_segment = (u32*)w;
  w += argus_align_up(((size_t)a.num_streams + 1) * 4, 256);
  a.split_failed = (u32*)w;
  a.segment_tiles = split_tiles(a.num_events);
  ARGUS_LAUNCH(k_split_scan, most, kScanThreads, 0, stream, a, first_segment);
  ARGUS_LAUNCH(k_split_chain, a.num_streams, kChainThreads, 0, stream, a, (const u32*)first_segment);
  const int rc = argus_launch_pair_tiled(a, stream, true);
  if (rc != ARGUS_OK) return rc;
  // a level of a segment a thread, on average
  const u32 each = most / a.num_streams * ARGUS_MAX_DEPTH, parts = (each + kFixThreads - 1) / kFixThreads;
  ARGUS_LAUNCH(k_split_fix, a.num_streams * parts, kFixThreads, 0, stream, a, (const u32*)first_segment, parts);
  return ARGUS_OK;
}
