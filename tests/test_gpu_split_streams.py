"""Few long streams: the segments of a stream are paired at the same time. Frames that stay open over many segments, streams that
end in the middle, empty and short ones among them, and markers that make a stream fall back to the chained pass, against the
oracle; both pairing alone and the one-call pipeline."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_12299_b200 as argus
from paper_2609_12299_b200 import tracegen as tg

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _wrap(ev, region, ctx=0):
    """The stream inside one interval of `region` that is open over all of it."""
    out = np.zeros(len(ev) + 2, argus.EVENT_DTYPE)
    out[1:-1] = ev
    out[0] = (ev["ts"][0] - 5, region << 1, ctx)
    out[-1] = (ev["ts"][-1] + 7, (region << 1) | 1, ctx)
    return out


def _trace(kind, rng):
    idx, ctas, iters = {"gemm": (1, 3, 1300), "attention": (2, 2, 8), "decode": (3, 1, 40)}[kind]
    spec = tg.config(idx).scaled(ctas, iters)
    ev, offs = tg.generate_host(spec)
    streams = [ev[offs[s]:offs[s + 1]] for s in range(spec.num_streams)]
    return spec, streams


@pytest.mark.parametrize("change", ["none", "wrapped", "cut", "lengths", "clamped", "defects"])
@pytest.mark.parametrize("kind", ["gemm", "attention", "decode"])
def test_segments(kind, change):
    rng = np.random.default_rng(7)
    spec, streams = _trace(kind, rng)
    R = spec.num_regions + 2
    if change == "wrapped":      # two levels that are open over every segment
        streams = [_wrap(_wrap(e, R - 1), R - 2) for e in streams]
    elif change == "cut":        # ends missing at the back
        streams = [e[:len(e) - int(rng.integers(0, 40))] for e in streams]
    elif change == "lengths":    # exact multiples of a tile and of a segment, one event more, one tile, nothing
        for s, n in enumerate([640, 641, 0, 8 * 640, 8 * 640 + 1, 1]):
            streams[s] = streams[s][:n]
    elif change == "clamped":    # outer intervals shorter than their children
        streams = [_wrap(e, R - 1) for e in streams]
        for e in streams:
            e["ts"][-1] = e["ts"][0] + np.uint64(9)
    elif change == "defects":    # one stream loses an end, one has a stray one, one has an outlier in time
        streams = [_wrap(e, R - 1) for e in streams]
        streams[0] = np.delete(streams[0], len(streams[0]) // 2)
        streams[1]["tag"][len(streams[1]) // 3] ^= 1
        streams[2]["ts"][len(streams[2]) // 2:] += np.uint64(1 << 33)
    while sum(len(e) for e in streams) <= 1 << 20:
        streams = streams + streams[:spec.warps_per_cta]
    ev = np.concatenate(streams)
    offs = np.cumsum([0] + [len(e) for e in streams]).astype(np.uint64)
    S, W = len(streams), spec.warps_per_cta
    assert S < 777 and len(ev) > 1 << 20 and len(ev) // S >= 10240
    d_ev = torch.from_numpy(ev.view(np.uint8).reshape(-1).copy()).to(DEV)
    d_off = torch.from_numpy(offs.view(np.int64).copy()).to(DEV)
    _, iv, ioffs, am, aoffs, o_st = oracle.pair(ev, offs, R)

    def check(p):
        st = p.fetch_status()
        assert int(st["code"]) == 0
        assert np.array_equal(p.interval_offsets.cpu().numpy().view(np.uint64), ioffs)
        assert np.array_equal(p.ambig_offsets.cpu().numpy().view(np.uint64), aoffs)
        assert p.intervals_numpy().tobytes() == iv.tobytes()
        assert p.ambig_numpy().tobytes() == am.tobytes()
        for f in ("n_ctx_mismatch", "n_time_reversed", "n_child_clamped", "intervals_required", "ambig_required"):
            assert int(st[f]) == int(o_st[f]), f

    check(argus.argus_pair_intervals(d_ev, d_off, R))
    cta_sm = (np.arange(S // W) % 2).astype(np.uint32)
    pairs = np.concatenate([spec.overlap_pairs, [[0, 1]]]).astype(np.uint32)
    r = argus.argus_synthesize(d_ev, d_off, R, W, torch.from_numpy(cta_sm.view(np.int32)).to(DEV), 2, torch.from_numpy(pairs.view(np.int32)).to(DEV))
    check(r.pair)
    _, tabs, _ = oracle.aggregate(iv, ioffs, am, aoffs, W, cta_sm, 2, R)
    for lv in ("warp", "cta", "sm", "kernel"):
        assert r.agg.table_numpy(lv).tobytes() == tabs[lv].tobytes(), lv
    _, ov, _ = oracle.overlap(iv, ioffs, W, cta_sm, 2, pairs)
    assert r.overlap_numpy(2).tobytes() == ov.tobytes()


@pytest.mark.parametrize("kind", ["gemm", "decode"])
def test_streams_given_up_while_their_segments_are_walked(kind):
    """Half of the streams have markers in the wrong order all over their length, which only the segments that meet them see, so that
    many blocks give up a stream while others take up its segments. The healthy streams between them must not notice. Every run
    against the oracle."""
    rng = np.random.default_rng(11)
    spec, streams = _trace(kind, rng)
    R = spec.num_regions + 1
    streams = streams * -(-(1 << 24) // sum(len(e) for e in streams))  # segments for every block, three times over
    streams = [_wrap(e, R - 1) for e in streams]
    for s in range(len(streams)):
        if s % 2 == 0:
            continue
        at = np.unique(rng.integers(1, len(streams[s]) - 2, 40) | 1)   # no neighbours
        tag = streams[s]["tag"]
        at = at[(tag[at] ^ tag[at + 1]) > 1][:4 + s % 9]                # two that follow one another, of different regions
        tag[at], tag[at + 1] = tag[at + 1], tag[at].copy()
    ev = np.concatenate(streams)
    offs = np.cumsum([0] + [len(e) for e in streams]).astype(np.uint64)
    S = len(streams)
    assert S < 777 and len(ev) // S >= 10240
    d_ev = torch.from_numpy(ev.view(np.uint8).reshape(-1).copy()).to(DEV)
    d_off = torch.from_numpy(offs.view(np.int64).copy()).to(DEV)
    _, iv, ioffs, am, aoffs, o_st = oracle.pair(ev, offs, R)
    assert int(o_st["code"]) == 0 and len(am)
    want = [torch.from_numpy(x.view(np.uint8).reshape(-1).copy()).to(DEV) for x in (iv, am, ioffs, aoffs)]
    p = None
    for _ in range(60):
        p = argus.argus_pair_intervals(d_ev, d_off, R, out=p)
        assert int(p.fetch_status()["code"]) == 0
        assert torch.equal(p.interval_offsets.view(torch.uint8), want[2]) and torch.equal(p.ambig_offsets.view(torch.uint8), want[3])
        assert torch.equal(p.intervals[:len(want[0])], want[0]) and torch.equal(p.ambig[:len(want[1])], want[1])
        p.intervals.zero_()
        p.ambig.zero_()


@pytest.mark.parametrize("S,n", [(110, 11_000), (320, 12_000), (592, 12_000), (776, 10_250)])
def test_few_streams_that_the_chained_pass_walks(S, n):
    """Streams of equal length, too short or too many for their segments to pay: the split kernels are launched and leave them all."""
    i = np.arange(S * n) % n
    ev = np.zeros(S * n, argus.EVENT_DTYPE)
    ev["ts"] = np.arange(S * n) * 5
    ev["tag"] = np.array([0, 2, 3, 1], np.uint32)[i % 4]
    ev["tag"][(i >= n // 2) & (i < n // 2 + 4)] = 2          # four begins without an end in the middle of every stream
    offs = (np.arange(S + 1) * n).astype(np.uint64)
    _, iv, ioffs, am, aoffs, _ = oracle.pair(ev, offs, 2)
    p = argus.argus_pair_intervals(torch.from_numpy(ev.view(np.uint8).reshape(-1).copy()).to(DEV), torch.from_numpy(offs.view(np.int64).copy()).to(DEV), 2)
    assert int(p.fetch_status()["code"]) == 0 and len(am)
    assert np.array_equal(p.interval_offsets.cpu().numpy().view(np.uint64), ioffs)
    assert p.intervals_numpy().tobytes() == iv.tobytes() and p.ambig_numpy().tobytes() == am.tobytes()
