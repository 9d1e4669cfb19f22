// argus_synthesize.cu — the whole hot path in one call: pair -> aggregate -> overlap.
//
// Pairing writes, beside every 48-byte interval record, an 8-byte digest (region, both durations, a flag
// bit); then ONE pass over the digests both aggregates the intervals and selects the overlap candidates (a pass
// over the records themselves reads six times the bytes). More than 400 regions, or a call that
// asks for no table: the three plain calls. Results are identical in every mode. argus_synthesize_ring is the
// same pipeline on a ring container.
#include "argus_internal.cuh"

#include <atomic>

namespace {

std::atomic<int> g_synth_mode_knob{-1};  // -1 = automatic

struct SynLayout {
  size_t pair, pair_bytes, agg, agg_bytes, ov, ov_bytes, pieces, spans, digest, starts, total;
  uint64_t digest_capacity;
  uint32_t parts, slices;
};

SynLayout syn_layout(uint64_t num_events, uint32_t num_streams, uint32_t num_regions, uint64_t ambig_capacity,
                     uint32_t num_pairs, uint32_t num_sms, uint64_t max_overlap_spans) {
  SynLayout L;
  size_t o = 0;
  L.pair = o; L.pair_bytes = argus_pair_workspace_bytes(num_events, num_streams, ambig_capacity); o += argus_align_up(L.pair_bytes, 256);
  L.agg = o; L.agg_bytes = argus_aggregate_workspace_bytes(num_events / 2, num_streams, num_regions); o += argus_align_up(L.agg_bytes, 256);
  // Overlap: the plain call's workspace, or control block, first pieces of the slices and 32 bytes a span (the entries
  // lie in the digest array).
  const bool digests = argus_aggregate_can_read_digests(num_regions);
  L.parts = argus_aggregate_digest_parts(num_streams, num_events);
  L.slices = argus_aggregate_digest_slices(num_streams, num_events);
  const size_t pieces = (size_t)num_streams * L.slices * sizeof(ArgusOvPiece);
  L.ov = o;
  L.pieces = o + argus_align_up(sizeof(ArgusOvCtl), 256);
  L.spans = L.pieces + argus_align_up(pieces, 256);
  const size_t from_entries = L.spans - o + (size_t)max_overlap_spans * 32, plain = argus_internal_overlap_bytes(max_overlap_spans, num_streams);
  L.ov_bytes = num_pairs ? argus_align_up(from_entries > plain ? from_entries : plain, 256) : 0;
  o += L.ov_bytes;
  // one digest per interval (two events each, so num_events / 2 at most; pairing and the pass over the digests stay inside the array)
  L.digest_capacity = digests ? num_events / 2 + 1 : 0;
  L.digest = o; o += argus_align_up((size_t)L.digest_capacity * 8, 256);
  L.starts = o; o += num_pairs ? argus_align_up((size_t)L.digest_capacity * 8, 256) : 0;  // begin times of overlap candidates
  L.total = o;
  return L;
}

}  // namespace

// Where argus_synthesize aggregates and selects overlap spans: -1 automatic, 1 in one pass over the intervals'
// digests, 2 and 3 the plain calls (test aid; results are identical).
extern "C" void argus_set_synthesize_mode(int mode) { g_synth_mode_knob.store(mode); }

extern "C" size_t argus_synthesize_workspace_bytes(uint64_t num_events, uint32_t num_streams, uint32_t num_regions,
                                                   uint64_t ambig_capacity, uint32_t num_pairs, uint32_t num_sms,
                                                   uint64_t max_overlap_spans) {
  return syn_layout(num_events, num_streams, num_regions, ambig_capacity, num_pairs, num_sms, max_overlap_spans).total;
}

// ring_written non-null: `events` is a ring container whose packed offsets are already in stream_offsets (device);
// num_events then bounds the surviving records and the status block has been cleared by the caller.
static int synthesize_impl(const argus_event_t* events, uint64_t num_events, const uint64_t* stream_offsets,
                           uint32_t num_streams, uint32_t num_regions, argus_interval_t* intervals,
                           uint64_t interval_capacity, uint64_t* interval_offsets, argus_ambiguity_t* ambig,
                           uint64_t ambig_capacity, uint64_t* ambig_offsets, uint32_t warps_per_cta,
                           const uint32_t* cta_sm, uint32_t num_sms, argus_agg_t* warp_tab, argus_agg_t* cta_tab,
                           argus_agg_t* sm_tab, argus_agg_t* kernel_tab, const uint32_t* pairs, uint32_t num_pairs,
                           argus_overlap_t* overlap_out, uint64_t max_overlap_spans, argus_status_t* status,
                           void* workspace, size_t workspace_bytes, void* cuda_stream, const uint64_t* ring_written,
                           uint32_t ring_capacity) {
  if (!status || !workspace || ((uintptr_t)workspace & 255)) return ARGUS_ERR_INVALID_ARG;
  if (warps_per_cta == 0 || num_streams % warps_per_cta != 0) return ARGUS_ERR_INVALID_ARG;
  if (num_regions == 0 || num_regions > ARGUS_MAX_REGIONS) return ARGUS_ERR_INVALID_ARG;
  if ((sm_tab || num_pairs) && ((!cta_sm && num_streams) || num_sms == 0)) return ARGUS_ERR_INVALID_ARG;
  if (num_pairs && (!pairs || !overlap_out)) return ARGUS_ERR_INVALID_ARG;
  const SynLayout L = syn_layout(num_events, num_streams, num_regions, ambig_capacity, num_pairs, num_sms, max_overlap_spans);
  if (workspace_bytes < L.total) return ARGUS_ERR_WORKSPACE;
  const int g_synth_mode = g_synth_mode_knob.load(std::memory_order_relaxed);
  char* ws = (char*)workspace;
  const bool want_agg = warp_tab || cta_tab || sm_tab || kernel_tab;

  // where aggregation and overlap selection happen: 1 = in one pass over the intervals' digests after pairing (or over the
  // records, and then the plain overlap call), 2 = the plain calls
  const bool can_one_pass = num_streams > 0 && want_agg && argus_aggregate_can_read_digests(num_regions) && num_pairs <= ARGUS_MAX_PAIRS;
  const bool use_digest = can_one_pass && L.digest_capacity != 0 && g_synth_mode != 2 && g_synth_mode != 3;  // (test aid: modes 2 and 3)
  ArgusOvCtl* const ov_ctl = (ArgusOvCtl*)(ws + L.ov);
  ArgusFuseArgs f = ArgusFuseArgs();
  if (use_digest && num_pairs) {
    f.pairs = pairs; f.num_pairs = num_pairs; f.entries = (u64*)(ws + L.digest); f.starts = (u64*)(ws + L.starts); f.pieces = (ArgusOvPiece*)(ws + L.pieces);
    f.ctl = ov_ctl;
  }
  int rc = argus_internal_pair(events, num_events, stream_offsets, num_streams, num_regions, intervals, interval_capacity,
                               interval_offsets, ambig, ambig_capacity, ambig_offsets, status, ws + L.pair, L.pair_bytes,
                               cuda_stream, ring_written ? 2 : 0, ring_written == nullptr,
                               use_digest ? (uint64_t*)(ws + L.digest) : nullptr, L.digest_capacity, ring_written, ring_capacity);
  if (rc != ARGUS_OK) return rc;

  if (want_agg) {
    rc = argus_internal_aggregate_scoped(intervals, interval_offsets, ambig, ambig_offsets, num_streams, warps_per_cta,
                                         cta_sm, num_sms, num_regions, nullptr, warp_tab, cta_tab, sm_tab, kernel_tab,
                                         nullptr, nullptr, status, ws + L.agg, L.agg_bytes, cuda_stream, false,
                                         f.num_pairs ? &f : nullptr,
                                         use_digest ? (const uint64_t*)(ws + L.digest) : nullptr, L.parts, L.slices, interval_capacity);
    if (rc != ARGUS_OK) return rc;
  }
  if (num_pairs) {
    if (f.num_pairs) {
      rc = argus_internal_overlap_from_digests(intervals, (const uint64_t*)f.starts, (const uint64_t*)f.entries, f.pieces,
                                               L.slices, num_streams, warps_per_cta, cta_sm, num_sms, pairs,
                                               num_pairs, overlap_out, status, ov_ctl, ws + L.spans, max_overlap_spans, L.digest_capacity, cuda_stream);
    } else {
      rc = argus_internal_overlap(intervals, interval_capacity, interval_offsets, num_streams, warps_per_cta, cta_sm, num_sms,
                                  pairs, num_pairs, overlap_out, status, ws + L.ov, L.ov_bytes, cuda_stream, false);
    }
    if (rc != ARGUS_OK) return rc;
  }
  return ARGUS_OK;
}

extern "C" int argus_synthesize(const argus_event_t* events, uint64_t num_events, const uint64_t* stream_offsets,
                                uint32_t num_streams, uint32_t num_regions, argus_interval_t* intervals,
                                uint64_t interval_capacity, uint64_t* interval_offsets, argus_ambiguity_t* ambig,
                                uint64_t ambig_capacity, uint64_t* ambig_offsets, uint32_t warps_per_cta,
                                const uint32_t* cta_sm, uint32_t num_sms, argus_agg_t* warp_tab, argus_agg_t* cta_tab,
                                argus_agg_t* sm_tab, argus_agg_t* kernel_tab, const uint32_t* pairs, uint32_t num_pairs,
                                argus_overlap_t* overlap_out, uint64_t max_overlap_spans, argus_status_t* status,
                                void* workspace, size_t workspace_bytes, void* cuda_stream) {
  return synthesize_impl(events, num_events, stream_offsets, num_streams, num_regions, intervals, interval_capacity,
                         interval_offsets, ambig, ambig_capacity, ambig_offsets, warps_per_cta, cta_sm, num_sms, warp_tab, cta_tab,
                         sm_tab, kernel_tab, pairs, num_pairs, overlap_out, max_overlap_spans, status, workspace, workspace_bytes,
                         cuda_stream, nullptr, 0);
}

extern "C" int argus_synthesize_ring(const argus_event_t* ring, uint32_t slot_capacity, const uint64_t* written,
                                     uint32_t num_streams, uint32_t num_regions, uint64_t* stream_offsets, uint64_t* dropped,
                                     argus_interval_t* intervals, uint64_t interval_capacity, uint64_t* interval_offsets,
                                     argus_ambiguity_t* ambig, uint64_t ambig_capacity, uint64_t* ambig_offsets,
                                     uint32_t warps_per_cta, const uint32_t* cta_sm, uint32_t num_sms, argus_agg_t* warp_tab,
                                     argus_agg_t* cta_tab, argus_agg_t* sm_tab, argus_agg_t* kernel_tab, const uint32_t* pairs,
                                     uint32_t num_pairs, argus_overlap_t* overlap_out, uint64_t max_overlap_spans,
                                     argus_status_t* status, void* workspace, size_t workspace_bytes, void* cuda_stream) {
  if (!status || !stream_offsets || slot_capacity == 0) return ARGUS_ERR_INVALID_ARG;
  if (num_streams && (!ring || !written)) return ARGUS_ERR_INVALID_ARG;
  if (((uintptr_t)written & 7) || ((uintptr_t)dropped & 7) || ((uintptr_t)stream_offsets & 7)) return ARGUS_ERR_INVALID_ARG;
  { const int rc = argus_internal_clear(status, nullptr, 0, cuda_stream); if (rc != ARGUS_OK) return rc; }
  const uint64_t bound = (uint64_t)num_streams * slot_capacity;  // what the slots can hold: sizes the workspace
  const int rc = argus_internal_ring_offsets(written, slot_capacity, num_streams, bound, stream_offsets, dropped, status, cuda_stream);
  if (rc != ARGUS_OK) return rc;
  // without streams there is nothing to read from a ring: the plain path writes the empty results
  return synthesize_impl(ring, bound, stream_offsets, num_streams, num_regions, intervals, interval_capacity, interval_offsets,
                         ambig, ambig_capacity, ambig_offsets, warps_per_cta, cta_sm, num_sms, warp_tab, cta_tab, sm_tab,
                         kernel_tab, pairs, num_pairs, overlap_out, max_overlap_spans, status, workspace, workspace_bytes,
                         cuda_stream, num_streams ? written : nullptr, slot_capacity);
}
