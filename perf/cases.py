"""Workloads by which the speed of this framework is measured: marker traces of the shapes that the repository's own
configurations, tests and benchmark use, taken through the public entry points as a program that analyses traces does.

A case names an operation and the trace that it works on:
  op    synth   argus_synthesize: the whole path in one call (the benchmark's step)
        calls   argus_pair_intervals, argus_aggregate and argus_overlap, one after the other
        ring    argus_synthesize_ring on a ring container whose slots have wrapped
        scoped  argus_aggregate_scoped (all tables, one row per iteration of a window) and argus_overlap_scoped
        pcmap   a mapping run: argus_pair_intervals, argus_map_pc_counts, argus_attribute
        join    queries of a reference run against probe runs (`how`: hashed, grouped or plain)
  kind  tiny, gemm, attention or decode, with `ctas`, `iters` and `inner` (see tracegen.TraceSpec) and defect rates.

Every trace comes from the seed alone and lies in GPU memory before the call, beside the output buffers and the
workspace where the entry point lets a program keep them. Results are whole numbers and have to be the same to the
bit, except what argus_attribute computes in fp64."""
from __future__ import annotations

import random
from dataclasses import replace

import numpy as np
import torch

import paper_2609_12299_b200 as argus
from paper_2609_12299_b200 import tracegen as tg
from paper_2609_12299_b200.tracegen.mapping import mapping_trace

KINDS = {"tiny": tg.TINY, "gemm": tg.GEMM, "attention": tg.ATTENTION, "decode": tg.DECODE}
MOST_EVENTS = 300_000_000  # no drawn case handles more marker records than this; the largest listed one has twice as many
DEV = "cuda:0"


def _case(name, op, kind, ctas, iters, inner=0, dup=0.0, drop=0.0, trunc=0.0, **more):
    return {"name": name, "op": op, "kind": kind, "ctas": ctas, "iters": iters, "inner": inner, "dup": dup, "drop": drop,
            "trunc": trunc, **more}


def listed():
    return [
        # the smallest call: 10 thousand records of four CTAs, as a test or an interactive query of one launch has them
        _case("synth_tiny", "synth", "tiny", 4, 626),
        # one short kernel: a GEMM of 40 tiles a CTA, 1.4 million records, all of it in the L2
        _case("synth_gemm_short", "synth", "gemm", 148, 40),
        # the persistent GEMM of the benchmark's secondary records: roles of unequal length, five regions
        _case("synth_gemm", "synth", "gemm", 148, 2000),
        # the attention trace: producer and consumer spans that overlap, 22 tiles of 512 KV iterations
        _case("synth_attention", "synth", "attention", 148, 22, 512),
        # the benchmark's decode megakernel at half its tokens, so that three of them fit the card: the largest call
        _case("synth_decode", "synth", "decode", 148, 128, 22),
        # the same kernel recorded on six CTAs only: few streams, each of them long
        _case("synth_decode_few", "synth", "decode", 6, 256, 22),
        # a lossy tracer: doubled begins, lost ends and streams cut short all over the GEMM trace
        _case("synth_malformed", "synth", "gemm", 148, 2000, 0, 0.0005, 0.001, 0.01),
        # the three plain calls, on an odd number of CTAs and iterations; one stream in a hundred is cut short
        _case("calls_gemm_ragged", "calls", "gemm", 131, 777, 0, 0.0, 0.0, 0.01),
        # a ring container that has wrapped: each warp's last 60,001 records, cut in the middle of a token
        _case("ring_decode", "ring", "decode", 148, 48, 22, slot=60_001),
        # a scoped query on a traced run: sixteen iterations, all regions, with role and iteration tables, and their overlap
        _case("scoped_decode", "scoped", "decode", 148, 48, 22, window=16),
        # PC-to-region attribution: a mapping run of the decode kernel with 70,560 PCs
        _case("pcmap_decode", "pcmap", "decode", 148, 8, 22, pcs=70_560, execs=2),
        # 2,000 reference operations looked up in three probe runs at once
        _case("join_decode", "join", "decode", 148, 16, 22, how="hashed", queries=2000, runs=3),
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def _draw_trace(rng, kind):
    if kind == "tiny":
        return {"ctas": rng.randint(1, 64), "iters": 2 * _log(rng, 8, 2048), "inner": 0}
    ctas = 148 if rng.random() < 0.5 else rng.randint(1, 147)  # the whole chip, or a subset of its SMs
    if kind == "gemm":
        return {"ctas": ctas, "iters": _log(rng, 5, 2000), "inner": 0}
    if kind == "attention":
        return {"ctas": ctas, "iters": _log(rng, 1, 22), "inner": _log(rng, 16, 512)}
    return {"ctas": ctas, "iters": _log(rng, 1, 256), "inner": rng.choice((8, 16, 22, 32))}


def draw(rng):
    while True:
        op = rng.choice(("synth", "synth", "synth", "synth", "calls", "calls", "ring", "scoped", "pcmap", "join"))
        kind = rng.choice({"synth": ("tiny", "gemm", "gemm", "attention", "decode", "decode"),
                           "calls": ("tiny", "gemm", "attention", "decode")}.get(op, ("gemm", "attention", "decode")))
        case = {"op": op, "kind": kind, "dup": 0.0, "drop": 0.0, "trunc": 0.0, **_draw_trace(rng, kind)}
        if op in ("synth", "calls") and kind != "tiny" and rng.random() < 0.3:
            case["trunc"] = 0.01
            if rng.random() < 0.5:
                case["dup"], case["drop"] = 0.0005, 0.001
        per_stream = _clean_events(case) // _spec(case, 0).num_streams
        if op == "ring":
            case["slot"] = max(3, int(per_stream * rng.uniform(0.4, 1.2)))  # above 1: nothing is overwritten
        elif op == "scoped":
            case["window"] = rng.randint(1, 16)
        elif op == "pcmap":
            case["pcs"], case["execs"] = rng.randint(43_856, 70_560), rng.randint(1, 3)
        elif op == "join":
            case["how"] = rng.choice(("hashed", "grouped", "plain"))
            case["queries"] = _log(rng, 80, 2000) if case["how"] != "plain" else rng.randint(5, 80)
            case["runs"] = rng.randint(1, 4)
        records = _records(case)
        if case["op"] == "join" and case["how"] == "plain":
            records *= case["queries"]  # one pass over the samples for each query
        if records <= MOST_EVENTS:
            return case


def _spec(case, seed):
    return tg.TraceSpec(KINDS[case["kind"]], case["ctas"], case["iters"], case["inner"], tg.BASE_SEED + 1000 * (seed + 1), case["dup"],
                        case["drop"], case["trunc"], name=case["op"])


def _clean_events(case):
    """Records of the trace without its defects (these change the number by a percent at most)."""
    return int(tg.host_offsets(replace(_spec(case, 0), p_dup_begin=0.0, p_drop_end=0.0, p_trunc=0.0))[-1])


def _records(case):
    """Marker records that one pass handles, for an operation on intervals twice the intervals."""
    n = _clean_events(case)
    if case["op"] == "ring":
        return min(n, case["slot"] * _spec(case, 0).num_streams)
    if case["op"] == "pcmap":
        return n + n * case["execs"]
    if case["op"] == "join":
        return n * (case["runs"] + 1)
    return n


def _whole(t):
    """A byte buffer of 8-byte-aligned records as 64-bit words, which is how the outputs are handed over."""
    return t.view(torch.int64)


def _status(t):
    return _whole(t)[:7]  # all but the last word, a diagnostic about the kernel's own way of working


def _device(a):
    return torch.from_numpy(a.view(np.int32)).to(DEV)


def _counts(pair):
    """(intervals, ambiguity records) that a pairing found: what a program reads from the status block before it looks at either."""
    st = pair.fetch_status()
    assert int(st["code"]) == 0, st
    return int(st["intervals_required"]), int(st["ambig_required"])


def _paired(spec):
    ev, off = tg.generate_cuda(spec, DEV)
    n = ev.numel() // 16
    p = argus.argus_pair_intervals(ev, off, spec.num_regions, interval_capacity=max(n // 2, 1), ambig_capacity=max(n // 64, 4096))
    return p, _counts(p)


def _ring(spec, slot):
    """The trace as a tracer with fixed slots leaves it: record i of a stream at position i mod slot, later ones over earlier ones."""
    ev, off = tg.generate_cuda(spec, DEV)
    words, at = ev.view(torch.int64).view(-1, 2), off.tolist()
    ring = torch.zeros((spec.num_streams, slot, 2), dtype=torch.int64, device=DEV)
    for s in range(spec.num_streams):
        n = at[s + 1] - at[s]
        kept, first = min(n, slot), max(n - slot, 0) % slot
        src = words[at[s + 1] - kept:at[s + 1]]
        head = min(kept, slot - first)
        ring[s, first:first + head] = src[:head]
        if kept > head:
            ring[s, :kept - head] = src[head:]
    return ring.view(-1).view(torch.uint8), off[1:] - off[:-1]


def prepare(case, seed):
    op, spec = case["op"], _spec(case, seed)
    s = {"op": op, "spec": spec, "case": case, "out": None, "cta_sm": _device(spec.cta_sm), "pairs": _device(spec.overlap_pairs)}
    if op in ("synth", "calls"):
        s["events"], s["offsets"] = tg.generate_cuda(spec, DEV)
        n = _clean_events(case)
        # room as the benchmark gives it: every second record can close an interval, few markers are ambiguous
        s["icap"], s["acap"], s["spans"] = n // 2, max(n // 64, 4096), max(n // 8, 1 << 16)
        if not spec.well_formed:
            s["icap"] += n // 1000 + 64  # doubled begins make a trace longer
        if op == "calls":
            need = argus.argus_overlap_workspace_bytes(s["icap"], spec.num_streams, len(spec.overlap_pairs), spec.num_sms)
            s["ov_ws"] = torch.empty(min(need, 2 << 30), dtype=torch.uint8, device=DEV)
            s["agg"] = None
        s["found"] = (n // 2, 0)
        if not spec.well_formed:  # how much a seed's trace holds differs: its results are handed over in buffers of one size
            run(s)
            p = s["out"].pair if op == "synth" else s["out"]
            s["found"], s["rest"] = (s["icap"], s["acap"]), p.intervals[_counts(p)[0] * 48:]
            p.ambig[_counts(p)[1] * 32:].zero_()
    elif op == "ring":
        s["ring"], s["written"] = _ring(spec, case["slot"])
        bound = spec.num_streams * case["slot"]
        # a cut leaves the ends of up to five open frames in each slot
        s["icap"], s["acap"], s["spans"] = bound // 2, max(bound // 64, 8 * spec.num_streams, 4096), max(bound // 8, 1 << 16)
        p, _, _ = argus.argus_pair_intervals_ring(s["ring"], case["slot"], s["written"], spec.num_regions, interval_capacity=s["icap"],
                                                  ambig_capacity=s["acap"])
        s["found"] = _counts(p)
    elif op == "scoped":
        p, (n_iv, n_amb) = _paired(spec)
        lo = max(spec.iters * max(spec.inner if spec.kind == tg.ATTENTION else 1, 1) // 2 - case["window"] // 2, 0)
        s.update(pair=p, icap=n_iv, scope=argus.ArgusScope(lo, lo + case["window"] - 1))
    elif op == "pcmap":
        ev, off = tg.generate_cuda(spec, DEV)
        s["events"], s["offsets"] = mapping_trace(ev, off, spec.num_regions, case["pcs"], case["execs"])
        s["icap"], s["acap"] = s["events"].numel() // 32, 4096
        g = torch.Generator(device=DEV).manual_seed(seed + 1)
        s["metric"] = torch.rand(case["pcs"], dtype=torch.float64, device=DEV, generator=g)
    else:
        p, (n_ref, _) = _paired(spec)
        s["reference"] = p.intervals[:n_ref * 48].clone()
        probes, offs, base = [], [], 0
        for r in range(case["runs"]):  # probe runs of the same kernel: other times, the same stream, region and iteration keys
            p, (n_iv, _) = _paired(replace(spec, seed=spec.seed + 1 + r))
            probes.append(p.intervals[:n_iv * 48].clone())
            offs.append(p.interval_offsets + base)
            base += n_iv
        s["samples"], s["sample_offsets"] = torch.cat(probes), torch.stack(offs)
        pick = random.Random(seed + 1)
        s["queries"] = torch.tensor([pick.randrange(n_ref) for _ in range(case["queries"])], dtype=torch.int64, device=DEV)
        if case["how"] == "hashed":
            need = argus.load_library().argus_join_workspace_bytes(case["queries"])
            s["join_ws"] = torch.empty(need, dtype=torch.uint8, device=DEV)
    return s


def _pair_outputs(p, found, rest=None):
    n_iv, n_amb = found
    if rest is not None:
        rest.zero_()  # what lies behind the last interval is unspecified
    return {"intervals": _whole(p.intervals[:n_iv * 48]), "interval_offsets": p.interval_offsets,
            "ambig": _whole(p.ambig[:n_amb * 32]), "ambig_offsets": p.ambig_offsets, "status": _status(p.status)}


def _tables(a, levels):
    return {lv: _whole(getattr(a, lv)) for lv in levels}


def run(s):
    op, spec, case = s["op"], s["spec"], s["case"]
    R, W, M = spec.num_regions, spec.warps_per_cta, spec.num_sms
    levels = ("warp", "cta", "sm", "kernel")
    if op == "synth":
        s["out"] = r = argus.argus_synthesize(s["events"], s["offsets"], R, W, s["cta_sm"], M, s["pairs"], interval_capacity=s["icap"],
                                              ambig_capacity=s["acap"], max_overlap_spans=s["spans"], out=s["out"])
        return {**_pair_outputs(r.pair, s["found"], s.get("rest")), **_tables(r.agg, levels), "overlap": _whole(r.overlap)}
    if op == "calls":
        s["out"] = p = argus.argus_pair_intervals(s["events"], s["offsets"], R, interval_capacity=s["icap"], ambig_capacity=s["acap"],
                                                  out=s["out"])
        s["agg"] = a = argus.argus_aggregate(p.intervals, p.interval_offsets, p.ambig, p.ambig_offsets, W, s["cta_sm"], M, R, out=s["agg"])
        ov, ov_status = argus.argus_overlap(p.intervals, s["icap"], p.interval_offsets, W, s["cta_sm"], M, s["pairs"], workspace=s["ov_ws"])
        return {**_pair_outputs(p, s["found"], s.get("rest")), **_tables(a, levels), "overlap": _whole(ov), "agg_status": _status(a.status),
                "ov_status": _status(ov_status)}
    if op == "ring":
        r, offsets, dropped = argus.argus_synthesize_ring(s["ring"], case["slot"], s["written"], R, W, s["cta_sm"], M, s["pairs"],
                                                          interval_capacity=s["icap"], ambig_capacity=s["acap"], max_overlap_spans=s["spans"])
        return {**_pair_outputs(r.pair, s["found"]), **_tables(r.agg, levels), "overlap": _whole(r.overlap), "offsets": offsets,
                "dropped": dropped}
    if op == "scoped":
        p = s["pair"]
        a = argus.argus_aggregate_scoped(p.intervals, p.interval_offsets, p.ambig, p.ambig_offsets, W, s["cta_sm"], M, R, s["scope"],
                                         levels=levels + ("role", "iter"))
        ov, ov_status = argus.argus_overlap_scoped(p.intervals, s["icap"], p.interval_offsets, W, s["cta_sm"], M, s["pairs"], s["scope"])
        return {**_tables(a, levels + ("role", "iter")), "overlap": _whole(ov), "agg_status": _status(a.status), "ov_status": _status(ov_status)}
    if op == "pcmap":
        s["out"] = p = argus.argus_pair_intervals(s["events"], s["offsets"], R + 1, interval_capacity=s["icap"], ambig_capacity=s["acap"],
                                                  out=s["out"])
        counts, map_status = argus.argus_map_pc_counts(p.intervals, p.interval_offsets, R, case["pcs"])
        mhat, entropy, alpha = argus.argus_attribute(counts, s["metric"])
        return {**_pair_outputs(p, (s["icap"], 0)), "counts": counts, "mhat": mhat, "entropy": entropy, "alpha": alpha,
                "map_status": _status(map_status)}
    if case["how"] == "hashed":
        out, status = argus.argus_join_samples_hashed(s["reference"], s["queries"], s["samples"], s["join_ws"])
    elif case["how"] == "grouped":
        out, status = argus.argus_join_samples_grouped(s["reference"], s["queries"], s["samples"], s["sample_offsets"], spec.num_streams)
    else:
        out, status = argus.argus_join_samples(s["reference"], s["queries"], s["samples"])
    return {"join": _whole(out), "status": _status(status)}


def work(case):
    """Records read once (16 B), intervals (48 B), tables (576 B a cell) and the other results written once; an operation on
    intervals reads them once. Sorting, matching and counting are whole-number work: no floating-point operations are claimed."""
    spec, op, n = _spec(case, 0), case["op"], _records(case)
    S, C, M, R = spec.num_streams, spec.num_ctas, spec.num_sms, spec.num_regions
    tables, overlap, offsets = (S + C + M + 1) * R * 576, len(spec.overlap_pairs) * M * 32, (S + 1) * 8
    if op in ("synth", "calls"):
        return {"bytes": 40 * n + 3 * offsets + tables + overlap, "flops": 0}
    if op == "ring":
        return {"bytes": 40 * n + 5 * offsets + tables + overlap, "flops": 0}
    if op == "scoped":
        return {"bytes": 24 * n + 2 * offsets + tables + overlap + (spec.warps_per_cta + case["window"]) * R * 576, "flops": 0}
    if op == "pcmap":
        return {"bytes": 40 * n + 3 * offsets + (R + 1) * case["pcs"] * 16 + case["pcs"] * 16 + (R + 1) * 8, "flops": 0}
    return {"bytes": 24 * n * case["runs"] // (case["runs"] + 1) + case["queries"] * (48 + 8 + 64), "flops": 0}


def tolerance(case):
    if case["op"] == "pcmap":
        return {"rel": 3e-15}  # fp64 quotients, logarithms and sums over the PCs; in another order they differ by up to 7e-16 of the value (2-norm), measured
    return "exact"
