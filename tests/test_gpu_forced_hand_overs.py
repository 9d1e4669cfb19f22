"""Streams that change hands at every look, whatever the others have left: deep stacks, child time beyond 32 bits and defects carried from block to
block in records, in both passes, every tile shape and the ring container, against the oracle. Each case counts the hand-overs, so that none passes
with streams walked whole. And the default rule: streams that do not share out evenly are handed on."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import paper_2609_12299_b200 as argus
from helpers import make_events, random_wellformed
from paper_2609_12299_b200 import tracegen as tg
from paper_2609_12299_b200.binding import KERNEL_TILED, argus_set_tile_variant
from test_gpu_hand_overs import _streams
from test_gpu_parity import _synthesize_matches, assert_pair_matches

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture
def at_every_look():
    lib = argus.load_library()
    lib.argus_testing_set_hand_overs(1)
    yield
    lib.argus_testing_set_hand_overs(0)


def _hand_overs(p):
    lib, first, second = argus.load_library(), ctypes.c_uint64(), ctypes.c_uint64()
    assert lib.argus_testing_hand_overs(ctypes.c_void_p(p.workspace.data_ptr()), ctypes.byref(first), ctypes.byref(second)) == 0
    return first.value, second.value


def _lose_ends_and_double_begins(ev, rng):
    ev = np.delete(ev, rng.choice(np.nonzero(ev["tag"] & 1)[0], 40, replace=False))
    dup = np.sort(rng.choice(np.nonzero((ev["tag"] & 1) == 0)[0], 25, replace=False))
    return np.insert(ev, dup, ev[dup])


def _deep(defects):
    rng = np.random.default_rng(35)
    evs = [random_wellformed(rng, 60_000, 6, max_height=h) for h in (40, 12)] + [random_wellformed(rng, 2_500, 6, max_height=3)]
    if defects:
        evs = [_lose_ends_and_double_begins(e, rng) for e in evs]
    return evs


def _long_child_time():
    rows, t = [], 1_700_000_000_000_000_000
    rows += [(t, "B", 0, 1), (t + 1, "B", 1, 1)]
    for i in range(20_000):  # 6e10 ticks under both frames, all along the stream
        rows.append((t + 9, "B", 2, 2)); t += 3_000_000; rows.append((t, "E", 2, 2))
    rows += [(t + 1, "E", 1, 1), (t + 5, "E", 0, 1)]
    return [make_events(rows)] * 3


@pytest.mark.parametrize("variant", [0, 1, 2, 3])
@pytest.mark.parametrize("evs", [_deep(False), _deep(True), _long_child_time()], ids=["deep", "defects", "child-time"])
def test_open_frames_change_hands(evs, variant, at_every_look):
    offs = np.cumsum([0] + [len(e) for e in evs]).astype(np.uint64)
    argus_set_tile_variant(variant)
    try:
        p, _ = assert_pair_matches(np.concatenate(evs), offs, 6, KERNEL_TILED)
    finally:
        argus_set_tile_variant(0)
    assert _hand_overs(p)[0] > 0


def test_second_pass(at_every_look):
    """More streams than blocks, of which the first has lost markers inside: the intervals of those behind it are written again."""
    streams = _streams((14_000,), 1_110, True)
    ev, offs = np.concatenate(streams), np.cumsum([0] + [len(e) for e in streams]).astype(np.uint64)
    p, _ = assert_pair_matches(ev, offs, 7, KERNEL_TILED)
    first, second = _hand_overs(p)
    assert first > 0 and second > 0


@pytest.mark.parametrize("defects", [False, True])
def test_ring(defects, at_every_look):
    evs = _deep(defects)
    slot = max(len(e) for e in evs) - 777  # the longer ones have wrapped
    ring, kept = np.zeros((len(evs), slot), argus.EVENT_DTYPE), []
    for s, e in enumerate(evs):
        idx = np.arange(max(len(e) - slot, 0), len(e))
        ring[s, idx % slot] = e[idx]
        kept.append(e[idx])
    offs = np.cumsum([0] + [len(k) for k in kept]).astype(np.uint64)
    _, iv, ioffs, am, aoffs, st = oracle.pair(np.concatenate(kept), offs, 6)
    assert int(st["code"]) == 0
    p, _, _ = argus.argus_pair_intervals_ring(torch.from_numpy(ring.view(np.uint8).reshape(-1).copy()).to(DEV), slot,
                                              torch.from_numpy(np.array([len(e) for e in evs], np.int64)).to(DEV), 6, ambig_capacity=len(am) + 16)
    assert int(p.fetch_status()["code"]) == 0
    assert p.intervals_numpy().tobytes() == iv.tobytes() and p.ambig_numpy().tobytes() == am.tobytes()
    assert np.array_equal(p.interval_offsets.cpu().numpy().view(np.uint64), ioffs)
    assert np.array_equal(p.ambig_offsets.cpu().numpy().view(np.uint64), aoffs)
    assert _hand_overs(p)[0] > 0


def test_synthesize(at_every_look):
    spec = tg.config(4).scaled(2, 3000)  # malformed: few long streams without defects are walked in segments, all at once
    res, _ = _synthesize_matches(spec, *tg.generate_host(spec))
    assert _hand_overs(res)[0] > 0


def test_default_rule_hands_on():
    """Streams of 30,000, 20,000 and 12,000 events, more of them than the chip holds blocks: the longest are taken first, and those who walk them have little
    left when the others, which wait, are as long as what was taken last."""
    streams = _streams((30_000, 20_000, 12_000), 2_400, False)
    ev, offs = np.concatenate(streams), np.cumsum([0] + [len(e) for e in streams]).astype(np.uint64)
    p, _ = assert_pair_matches(ev, offs, 7, KERNEL_TILED)
    print("hand-overs by the default rule:", _hand_overs(p))
    assert _hand_overs(p)[0] > 0
