"""Interval counts foretold from the ends of the streams (calls of 2^20 events and more): streams cut short at the back, at the
front, at both, and malformed ones for which the foretold count is wrong, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_12299_b200 as argus
from paper_2609_12299_b200 import tracegen as tg

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _cut_streams(rng, ev, offs, front, back, every):
    parts, out = [], [0]
    for s in range(len(offs) - 1):
        e = ev[offs[s]:offs[s + 1]]
        if s % every == 1:
            e = e[int(rng.integers(1, 2000)) * front:]
        if s % every in (1, 2):
            e = e[:len(e) - int(rng.integers(1, 2000)) * back]
        parts.append(e)
        out.append(out[-1] + len(e))
    return np.concatenate(parts), np.array(out, np.uint64)


@pytest.mark.parametrize("idx,ctas,iters,front,back,every", [(1, 4, 900, 0, 1, 50), (1, 4, 900, 1, 0, 3), (2, 2, 4, 1, 1, 3), (3, 4, 10, 1, 1, 3), (4, 4, 900, 1, 1, 5)])
def test_cut_streams(idx, ctas, iters, front, back, every):
    rng = np.random.default_rng(idx)
    spec = tg.config(idx).scaled(ctas, iters)
    ev, offs = tg.generate_host(spec)
    ev, offs = _cut_streams(rng, ev, offs.astype(np.int64), front, back, every)
    while len(ev) < 1 << 20:  # more streams of the same
        offs = np.concatenate([offs, offs[1:] + offs[-1]])
        ev = np.concatenate([ev, ev])
    d_ev = torch.from_numpy(ev.view(np.uint8).reshape(-1).copy()).to(DEV)
    d_off = torch.from_numpy(offs.view(np.int64).copy()).to(DEV)
    rc, iv, ioffs, am, aoffs, _ = oracle.pair(ev, offs, spec.num_regions)
    for kernel in (1, 2):
        p = argus.argus_pair_intervals(d_ev, d_off, spec.num_regions, kernel=kernel)
        assert int(p.fetch_status()["code"]) == 0
        assert np.array_equal(p.interval_offsets.cpu().numpy().view(np.uint64), ioffs)
        assert np.array_equal(p.ambig_offsets.cpu().numpy().view(np.uint64), aoffs)
        assert p.intervals_numpy().tobytes() == iv.tobytes()
        assert p.ambig_numpy().tobytes() == am.tobytes()


@pytest.mark.parametrize("slot", [7001, 9001])
def test_wrapped_ring(slot):
    """Every slot has wrapped in the middle of a token: the packed records through the oracle."""
    spec = tg.config(3).scaled(10, 6)
    ev, offs = tg.generate_host(spec)
    S = spec.num_streams
    ring = np.zeros((S, slot), argus.EVENT_DTYPE)
    kept = []
    for s in range(S):
        e = ev[offs[s]:offs[s + 1]]
        n = len(e)
        idx = np.arange(max(n - slot, 0), n)
        ring[s, idx % slot] = e[idx]
        kept.append(e[idx])
    packed = np.concatenate(kept)
    poffs = np.cumsum([0] + [len(k) for k in kept]).astype(np.uint64)
    assert len(packed) >= 1 << 20
    rc, iv, ioffs, am, aoffs, _ = oracle.pair(packed, poffs, spec.num_regions)
    d_ring = torch.from_numpy(ring.view(np.uint8).reshape(-1).copy()).to(DEV)
    written = torch.from_numpy(np.diff(offs).astype(np.int64)).to(DEV)
    p, o, dropped = argus.argus_pair_intervals_ring(d_ring, slot, written, spec.num_regions)
    assert int(p.fetch_status()["code"]) == 0
    assert p.intervals_numpy().tobytes() == iv.tobytes()
    assert p.ambig_numpy().tobytes() == am.tobytes()
    assert np.array_equal(p.ambig_offsets.cpu().numpy().view(np.uint64), aoffs)
