"""More streams than the chip holds blocks of the pairing kernel, of lengths that do not share out evenly: streams change hands between
blocks, with frames open (some all along the stream), their child time, and defects. Against the oracle, every tile shape and the ring container."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_12299_b200 as argus
from helpers import random_wellformed
from paper_2609_12299_b200.binding import argus_set_tile_variant

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
R = 7


def _streams(lengths, S, defects):
    """Streams of about these lengths, some inside two frames that are open all along, some with lost ends or doubled begins."""
    rng = np.random.default_rng(41)
    kinds = {}
    for n in set(lengths):
        ev = random_wellformed(rng, max(n // 2 - 2, 0), R - 2, max_height=9)
        for deep in (False, True):
            if deep and len(ev):
                out = np.zeros(len(ev) + 4, argus.EVENT_DTYPE)
                out[2:-2] = ev
                out[0], out[1] = (ev["ts"][0] - 5, (R - 2) << 1, 1), (ev["ts"][0] - 3, (R - 1) << 1, 1)
                out[-2], out[-1] = (ev["ts"][-1] + 2, ((R - 1) << 1) | 1, 1), (ev["ts"][-1] + 9, ((R - 2) << 1) | 1, 1)
            else:
                out = ev.astype(argus.EVENT_DTYPE)
            kinds[n, deep] = out
    streams = []
    for s in range(S):
        ev = kinds[lengths[s % len(lengths)], s % 3 == 0].copy()
        ev["ts"] += np.uint64(1000 * s)
        if defects and s % 5 == 1 and len(ev) > 100:
            ev = np.delete(ev, np.nonzero(ev["tag"] & 1)[0][rng.integers(10, 40, 2)])
            ev = np.insert(ev, len(ev) // 3, ev[len(ev) // 3])
        streams.append(ev)
    return streams


@pytest.mark.parametrize("lengths,S,defects", [
    ((30_000,) + (9_000,) * 5, 1_260, False),   # a few long ones: these are never handed on
    ((14_000,), 1_110, True),                    # equal ones, some left for a second round
    ((0, 641, 25_000, 3_840, 7_681, 12_345), 1_560, True),
])
def test_streams_change_hands(lengths, S, defects):
    streams = _streams(lengths, S, defects)
    ev = np.concatenate(streams)
    offs = np.cumsum([0] + [len(e) for e in streams]).astype(np.uint64)
    assert len(ev) > 1 << 20
    _, iv, ioffs, am, aoffs, o_st = oracle.pair(ev, offs, R)
    assert int(o_st["code"]) == 0
    d_ev = torch.from_numpy(ev.view(np.uint8).reshape(-1).copy()).to(DEV)
    d_off = torch.from_numpy(offs.view(np.int64).copy()).to(DEV)

    def check(p):
        st = p.fetch_status()
        assert int(st["code"]) == 0
        assert np.array_equal(p.interval_offsets.cpu().numpy().view(np.uint64), ioffs)
        assert np.array_equal(p.ambig_offsets.cpu().numpy().view(np.uint64), aoffs)
        assert p.intervals_numpy().tobytes() == iv.tobytes() and p.ambig_numpy().tobytes() == am.tobytes()
        for f in ("n_ctx_mismatch", "n_time_reversed", "n_child_clamped", "intervals_required", "ambig_required"):
            assert int(st[f]) == int(o_st[f]), f

    for variant in (0, 1, 2, 3):
        argus_set_tile_variant(variant)
        try:
            for _ in range(3):  # who hands what on to whom differs from run to run
                check(argus.argus_pair_intervals(d_ev, d_off, R))
        finally:
            argus_set_tile_variant(0)
    slot = max(len(e) for e in streams)
    ring = np.zeros((S, slot), argus.EVENT_DTYPE)
    for s, e in enumerate(streams):
        ring[s, :len(e)] = e
    written = torch.from_numpy(np.diff(offs).astype(np.int64)).to(DEV)
    p, _, _ = argus.argus_pair_intervals_ring(torch.from_numpy(ring.view(np.uint8).reshape(-1)).to(DEV), slot, written, R, ambig_capacity=len(am) + 64)
    check(p)
