"""Child time beyond 2^32 ticks inside a tile whose windows are cut by lost markers: the ends before a cut count, and their sums must
be whole whatever the order in which the block's threads add to a parent. Against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_12299_b200 as argus
from paper_2609_12299_b200.binding import KERNEL_AUTO, KERNEL_TILED

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", [KERNEL_AUTO, KERNEL_TILED])
@pytest.mark.parametrize("share,lost", [(0.01, 0.002), (0.3, 0.002), (1.0, 0.002), (1.0, 0.0), (0.3, 0.05)])
def test_child_time_wraps_in_a_cut_window(share, lost, kernel):
    rng = np.random.default_rng(31)
    streams = []
    for s in range(96):
        n = int(rng.integers(1, 12000))
        dur = np.where(rng.random(n) < share, rng.integers(1 << 28, 1 << 32, n), rng.integers(0, 300, n)).astype(np.uint64)
        ev = np.zeros(2 * n, argus.EVENT_DTYPE)
        ev["ts"][0::2] = np.cumsum(dur + np.uint64(3)) - dur
        ev["ts"][1::2] = ev["ts"][0::2] + dur
        ev["tag"][0::2] = rng.integers(0, 5, n).astype(np.uint32) << 1
        ev["tag"][1::2] = ev["tag"][0::2] | 1
        ev = ev[rng.random(2 * n) >= lost]           # lost ends leave frames open, which gather all that follows
        if s % 2 and len(ev):                        # the stream inside one interval of a region of its own
            ev = np.concatenate([ev[:1], ev, ev[-1:]])
            ev["tag"][0], ev["tag"][-1] = 10, 11
        streams.append(ev)
    ev = np.concatenate(streams)
    offs = np.cumsum([0] + [len(e) for e in streams]).astype(np.uint64)
    rc, iv, ioffs, am, aoffs, o_st = oracle.pair(ev, offs, 6)
    p = argus.argus_pair_intervals(torch.from_numpy(ev.view(np.uint8).reshape(-1).copy()).cuda(),
                                   torch.from_numpy(offs.view(np.int64).copy()).cuda(), 6, kernel=kernel)
    st = p.fetch_status()
    assert int(st["code"]) == int(o_st["code"])
    if int(o_st["code"]):                            # more than 64 frames left open
        return
    assert np.array_equal(p.interval_offsets.cpu().numpy().view(np.uint64), ioffs)
    assert p.intervals_numpy().tobytes() == iv.tobytes()
    assert p.ambig_numpy().tobytes() == am.tobytes()
    for f in ("n_ctx_mismatch", "n_time_reversed", "n_child_clamped"):
        assert int(st[f]) == int(o_st[f]), f


@pytest.mark.parametrize("kernel", [KERNEL_AUTO, KERNEL_TILED])
def test_times_at_both_ends_of_the_64_bit_range(kernel):
    """An end whose time lies nearly 2^64 ticks before its begin's: the difference wraps to a few ticks, but the time runs backwards."""
    rng = np.random.default_rng(5)
    streams = []
    for s in range(20):
        n = int(rng.integers(1, 4000))
        ev = np.zeros(4 * n, argus.EVENT_DTYPE)      # an outer interval around an inner one, n times
        ev["tag"] = np.tile(np.array([0, 2, 3, 1], np.uint32), n)
        near = rng.integers(0, 1 << 40 if s % 2 else 200, 4 * n).astype(np.uint64)
        ev["ts"] = np.where(rng.random(4 * n) < 0.5, near, ~near)
        streams.append(ev)
    # begin near the top, end near the bottom: a step of 15, of 2^32 - 1, of 2^32, of 0 (no step back), and the other way round
    top = np.uint64(2**64 - 1)
    for b, e in ((top - np.uint64(9), 5), (top, (1 << 32) - 2), (top, (1 << 32) - 1), (top, top), (5, top - np.uint64(9)), (top, 0)):
        ev = np.zeros(2, argus.EVENT_DTYPE)
        ev["ts"], ev["tag"] = [b, e], [0, 1]
        streams.append(ev)
    ev = np.concatenate(streams)
    offs = np.cumsum([0] + [len(e) for e in streams]).astype(np.uint64)
    _, iv, ioffs, am, _, o_st = oracle.pair(ev, offs, 2)
    p = argus.argus_pair_intervals(torch.from_numpy(ev.view(np.uint8).reshape(-1).copy()).cuda(),
                                   torch.from_numpy(offs.view(np.int64).copy()).cuda(), 2, kernel=kernel)
    st = p.fetch_status()
    assert int(st["code"]) == 0 and int(o_st["code"]) == 0 and len(am) == 0
    assert p.intervals_numpy().tobytes() == iv.tobytes()
    for f in ("n_ctx_mismatch", "n_time_reversed", "n_child_clamped"):
        assert int(st[f]) == int(o_st[f]), f
