"""Interval counts foretold from the ends of the streams (calls of 2^20 events and more): streams cut short at the back, at the
front, at both, and malformed ones for which the foretold count is wrong, against the oracle."""
import ctypes

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


@pytest.mark.parametrize("S,length,cut", [(1025, 1200, 0.0), (1500, 9000, 0.3), (1500, 9000, 0.02), (11_000, 200, 0.5), (40_000, 30, 0.1), (300_001, 6, 0.1)])
def test_streams_of_several_outermost_regions(S, length, cut):
    """Streams that begin and end with different regions although they are whole, and streams among them that lack some of their
    front or back; more streams than a block, and than all warps, take at a time."""
    rng = np.random.default_rng(S)
    n = 3 * rng.integers(length // 6, length // 3 + 2, S)
    offs = np.concatenate([[0], np.cumsum(2 * n)])
    inner = np.arange(offs[-1]) - np.repeat(offs[:-1], 2 * n)      # index within the stream: a pair around another, then a pair
    ev = np.zeros(offs[-1], argus.EVENT_DTYPE)
    ev["ts"] = np.arange(len(ev)) * 3
    six = inner % 6
    region = np.where((six == 1) | (six == 2), 6, (inner // 6 * 2 + (six >= 4)) % 5)
    ev["tag"] = region * 2 + np.isin(six, (2, 3, 5))
    keep = np.ones(len(ev), bool)
    for s in np.nonzero(rng.random(S) < cut)[0]:
        k = int(rng.integers(1, 2 * n[s] + 1))
        if rng.random() < 0.5:
            keep[offs[s]:offs[s] + k // 4] = False
        else:
            keep[offs[s + 1] - k:offs[s + 1]] = False
    kept = np.concatenate([[0], np.cumsum(keep)])
    ev, offs = ev[keep], kept[offs].astype(np.uint64)
    assert len(ev) > 1 << 20
    _, iv, ioffs, am, aoffs, _ = oracle.pair(ev, offs, 7)
    p = argus.argus_pair_intervals(torch.from_numpy(ev.view(np.uint8).reshape(-1).copy()).to(DEV), torch.from_numpy(offs.view(np.int64).copy()).to(DEV), 7)
    assert int(p.fetch_status()["code"]) == 0
    assert np.array_equal(p.interval_offsets.cpu().numpy().view(np.uint64), ioffs)
    assert np.array_equal(p.ambig_offsets.cpu().numpy().view(np.uint64), aoffs)
    assert p.intervals_numpy().tobytes() == iv.tobytes()
    assert p.ambig_numpy().tobytes() == am.tobytes()


@pytest.mark.parametrize("defect,where,streams", [("lost ends", 0.0, 900), ("doubled begins", 0.0, 1100), ("lost begins", 0.0, 900), ("lost ends", 0.9, 900),
                                                  ("cut fronts", 0.0, 900), ("lost ends", 0.0, 300), ("lost ends", 0.98, 300)])
def test_defects_inside_streams(defect, where, streams):
    """Defects that show at neither end of a stream, in calls of 2^22 events and more, where windows all over the trace tell them and
    all markers are counted: in all streams, and in the last ones only; few long streams, too. Stray ends make the count wrong."""
    rng = np.random.default_rng(streams)
    spec = tg.config(1).scaled(4, 700)
    ev, offs = tg.generate_host(spec)
    source = [ev[offs[s]:offs[s + 1]] for s in range(spec.num_streams)]
    parts, total = [], 0
    for s in range(streams):
        e = source[s % len(source)]
        if s >= where * streams:
            is_end = (e["tag"] & 1) == 1
            hit = rng.random(len(e)) < 0.002
            hit[0] = hit[-1] = False
            if defect == "lost ends":
                e = e[~(hit & is_end)]
            elif defect == "lost begins":
                e = e[~(hit & ~is_end)]
            elif defect == "doubled begins":
                e = np.repeat(e, 1 + (hit & ~is_end))
            else:
                e = e[int(rng.integers(0, 60)):]
                e = e[~(hit[-len(e):] & ((e["tag"] & 1) == 1))]
        parts.append(e)
        total += len(e)
    while total < 1 << 22:
        parts += parts[:streams]
        total *= 2
    ev = np.concatenate(parts)
    offs = np.cumsum([0] + [len(e) for e in parts]).astype(np.uint64)
    _, iv, ioffs, am, aoffs, o_st = oracle.pair(ev, offs, spec.num_regions)
    assert int(o_st["code"]) == 0 and len(am) > 0
    p = argus.argus_pair_intervals(torch.from_numpy(ev.view(np.uint8).reshape(-1).copy()).to(DEV), torch.from_numpy(offs.view(np.int64).copy()).to(DEV),
                                   spec.num_regions, ambig_capacity=len(am) + 16)
    assert int(p.fetch_status()["code"]) == 0
    assert np.array_equal(p.interval_offsets.cpu().numpy().view(np.uint64), ioffs)
    assert np.array_equal(p.ambig_offsets.cpu().numpy().view(np.uint64), aoffs)
    assert p.intervals_numpy().tobytes() == iv.tobytes()
    assert p.ambig_numpy().tobytes() == am.tobytes()


def test_wrapped_ring_with_defects():
    """The same in a ring container: the slots have wrapped, so streams start with ends of lost begins, and ends are missing inside."""
    rng = np.random.default_rng(3)
    spec = tg.config(1).scaled(75, 300)
    ev, offs = tg.generate_host(spec)
    slot = 4801
    ring, kept, written = np.zeros((spec.num_streams, slot), argus.EVENT_DTYPE), [], []
    for s in range(spec.num_streams):
        e = ev[offs[s]:offs[s + 1]]
        hit = (rng.random(len(e)) < 0.002) & ((e["tag"] & 1) == 1)
        e = np.tile(e[~hit], 2)
        idx = np.arange(max(len(e) - slot, 0), len(e))
        ring[s, idx % slot] = e[idx]
        kept.append(e[idx])
        written.append(len(e))
    packed = np.concatenate(kept)
    poffs = np.cumsum([0] + [len(k) for k in kept]).astype(np.uint64)
    assert len(packed) >= 1 << 22
    _, iv, ioffs, am, aoffs, o_st = oracle.pair(packed, poffs, spec.num_regions)
    assert int(o_st["code"]) == 0
    p, _, _ = argus.argus_pair_intervals_ring(torch.from_numpy(ring.view(np.uint8).reshape(-1).copy()).to(DEV), slot,
                                              torch.from_numpy(np.array(written, np.int64)).to(DEV), spec.num_regions, ambig_capacity=len(am) + 16)
    assert int(p.fetch_status()["code"]) == 0
    assert p.intervals_numpy().tobytes() == iv.tobytes()
    assert p.ambig_numpy().tobytes() == am.tobytes()
    assert np.array_equal(p.ambig_offsets.cpu().numpy().view(np.uint64), aoffs)


def _passes(p):
    lib, counted, second = argus.load_library(), ctypes.c_uint32(), ctypes.c_uint32()
    assert lib.argus_testing_pair_passes(ctypes.c_void_p(p.workspace.data_ptr()), ctypes.byref(counted), ctypes.byref(second)) == 0
    return bool(counted.value), bool(second.value)


def _spoil(e, defect, rng, num_regions):
    is_end = (e["tag"] & 1) == 1
    hit = rng.random(len(e)) < 0.002
    hit[0] = hit[-1] = False
    if defect == "lost ends":
        return e[~(hit & is_end)]
    if defect == "lost begins":
        return e[~(hit & ~is_end)]
    if defect == "lost both":
        return e[~hit]
    if defect == "doubled begins":
        return np.repeat(e, 1 + (hit & ~is_end))
    if defect == "doubled ends":
        return np.repeat(e, 1 + (hit & is_end))
    e = e.copy()
    hit &= is_end == (defect == "changed ends")
    e["tag"][hit] = (((e["tag"][hit] >> 1) + rng.integers(1, num_regions, hit.sum()).astype(np.uint32)) % num_regions << 1) | (e["tag"][hit] & 1)
    return e


@pytest.mark.parametrize("defect,where,counted,second", [
    (None, 0.0, False, False), ("lost ends", 0.0, True, False), ("doubled begins", 0.0, True, False), ("lost begins", 0.0, True, False),
    ("doubled ends", 0.0, True, False), ("changed ends", 0.0, False, True), ("changed begins", 0.0, False, True), ("lost both", 0.0, False, True),
    ("lost ends", 329.0, False, False), ("one stream", 0.0, False, False)])
def test_what_is_counted_and_what_is_done_again(defect, where, counted, second):
    """Markers are counted where that tells the number of intervals, and then nothing is written twice; not where it cannot (markers that
    have changed, lost begins among lost ends), and not where no stream lies behind the first malformed one. 330 streams."""
    rng = np.random.default_rng(11)
    spec = tg.config(1).scaled(4, 700)
    ev, offs = tg.generate_host(spec)
    source = [ev[offs[s]:offs[s + 1]] for s in range(spec.num_streams)]
    parts = [source[s % len(source)] for s in range(330)]
    if defect == "one stream":
        parts = [np.concatenate([_spoil(e, "doubled ends", rng, spec.num_regions) for e in parts])]
    elif defect:
        parts = [_spoil(e, defect, rng, spec.num_regions) if s >= where else e for s, e in enumerate(parts)]
    ev = np.concatenate(parts)
    offs = np.cumsum([0] + [len(e) for e in parts]).astype(np.uint64)
    assert len(ev) >= 1 << 22
    _, iv, ioffs, am, aoffs, o_st = oracle.pair(ev, offs, spec.num_regions)
    assert int(o_st["code"]) == 0
    p = argus.argus_pair_intervals(torch.from_numpy(ev.view(np.uint8).reshape(-1).copy()).to(DEV), torch.from_numpy(offs.view(np.int64).copy()).to(DEV),
                                   spec.num_regions, ambig_capacity=len(am) + 16)
    assert int(p.fetch_status()["code"]) == 0
    assert _passes(p) == (counted, second)
    assert np.array_equal(p.interval_offsets.cpu().numpy().view(np.uint64), ioffs)
    assert p.intervals_numpy().tobytes() == iv.tobytes()
    assert p.ambig_numpy().tobytes() == am.tobytes()
