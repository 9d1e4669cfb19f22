"""Calls that get only part of the chip, because a kernel of another stream holds SMs for longer than the call takes, or because calls on streams of
different priority share it: nothing waits for a block that has not started, so every call ends before that kernel does and is right."""
import ctypes
import time

import numpy as np
import pytest
import torch

import oracle
import paper_2609_12299_b200 as argus
from paper_2609_12299_b200 import tracegen as tg
from paper_2609_12299_b200.binding import argus_set_tile_variant

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
HELD_US = 300_000


def _while_sms_are_held(sms, call):
    lib, stream = argus.load_library(), torch.cuda.Stream()
    call()  # (buffers, shared-memory limits)
    torch.cuda.synchronize()
    assert lib.argus_testing_hold_sms(sms, HELD_US, ctypes.c_void_p(stream.cuda_stream)) == 0
    held = stream.record_event()
    time.sleep(0.02)
    out = call()
    done = torch.cuda.current_stream().record_event()
    while not done.query() and not held.query():
        time.sleep(0.001)
    before = not held.query()
    torch.cuda.synchronize()
    assert before, "the call waited for the other stream's kernel"
    return out


def _trace(idx, ctas, iters):
    spec = tg.config(idx).scaled(ctas, iters)
    ev, offs = tg.generate_host(spec)
    _, iv, ioffs, am, aoffs, st = oracle.pair(ev, offs, spec.num_regions)
    assert int(st["code"]) == 0
    d_ev, d_off = torch.from_numpy(ev.view(np.uint8).reshape(-1).copy()).to(DEV), torch.from_numpy(offs.view(np.int64).copy()).to(DEV)
    return spec, ev, offs, d_ev, d_off, iv, am


# more streams than the chip holds blocks, and fewer; a malformed trace, whose second pass does some streams again
@pytest.mark.parametrize("idx,ctas,iters", [(1, 148, 30), (1, 50, 200), (3, 70, 1), (4, 100, 40)])
@pytest.mark.parametrize("sms", [40, 100, 147])
def test_part_of_the_chip(idx, ctas, iters, sms):
    spec, ev, offs, d_ev, d_off, iv, am = _trace(idx, ctas, iters)
    for variant in (0, 1, 2, 3) if sms == 100 else (0,):
        argus_set_tile_variant(variant)
        try:
            p = _while_sms_are_held(sms, lambda: argus.argus_pair_intervals(d_ev, d_off, spec.num_regions, ambig_capacity=len(am) + 16))
        finally:
            argus_set_tile_variant(0)
        assert int(p.fetch_status()["code"]) == 0
        assert p.intervals_numpy().tobytes() == iv.tobytes() and p.ambig_numpy().tobytes() == am.tobytes()


@pytest.mark.parametrize("sms", [100, 147])
def test_ring_and_one_call_pipeline(sms):
    spec, ev, offs, d_ev, d_off, iv, am = _trace(1, 120, 25)
    lengths, S = np.diff(offs).astype(np.int64), spec.num_streams
    slot = int(lengths.max())
    ring = np.zeros((S, slot), argus.EVENT_DTYPE)
    for s in range(S):
        ring[s, :lengths[s]] = ev[offs[s]:offs[s + 1]]
    d_ring, written = torch.from_numpy(ring.view(np.uint8).reshape(-1)).to(DEV), torch.from_numpy(lengths).to(DEV)
    p, _, _ = _while_sms_are_held(sms, lambda: argus.argus_pair_intervals_ring(d_ring, slot, written, spec.num_regions, ambig_capacity=64))
    assert int(p.fetch_status()["code"]) == 0 and p.intervals_numpy().tobytes() == iv.tobytes()
    d_sm, pairs = (torch.from_numpy(a.view(np.int32).copy()).to(DEV) for a in (spec.cta_sm, spec.overlap_pairs))
    r = _while_sms_are_held(sms, lambda: argus.argus_synthesize(d_ev, d_off, spec.num_regions, spec.warps_per_cta, d_sm, spec.num_sms, pairs))
    assert int(r.fetch_status()["code"]) == 0 and r.pair.intervals_numpy().tobytes() == iv.tobytes()


def test_calls_on_streams_of_different_priority():
    """Equal calls on four streams, two of them of higher priority, at the same time."""
    spec, ev, offs, d_ev, d_off, iv, am = _trace(1, 148, 60)
    streams = [torch.cuda.Stream(priority=p) for p in (0, -1, 0, -1)]
    outs = []
    for st in streams:
        with torch.cuda.stream(st):
            outs.append(argus.argus_pair_intervals(d_ev, d_off, spec.num_regions, ambig_capacity=64))
    torch.cuda.synchronize()
    t0 = time.time()
    for _ in range(200):
        for st, out in zip(streams, outs):
            with torch.cuda.stream(st):
                argus.argus_pair_intervals(d_ev, d_off, spec.num_regions, out=out)
    torch.cuda.synchronize()
    assert time.time() - t0 < 1.0  # (a wait that runs out takes about that long)
    for out in outs:
        assert int(out.fetch_status()["code"]) == 0 and out.intervals_numpy().tobytes() == iv.tobytes()
