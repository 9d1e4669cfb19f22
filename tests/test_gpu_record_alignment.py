"""Interval records are written 32 bytes at a time where they lie on such a boundary: arrays that start on one and 16 bytes behind one, streams
whose first record lies on either, and nothing written outside the array's capacity."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
import paper_2609_12299_b200 as argus
from paper_2609_12299_b200 import tracegen as tg

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("shift", [0, 16])
@pytest.mark.parametrize("short", [0, 1, 2, 701])
def test_array_that_starts_on_a_16_byte_boundary(shift, short):
    spec = tg.config(1).scaled(3, 37)
    ev, offs = tg.generate_host(spec)
    ev = np.concatenate([ev[:2], ev])  # a first stream of two begins more, which close no interval: the others' records move by one
    offs = offs + np.uint64(2)
    offs[0] = 0
    R = spec.num_regions
    _, iv, ioffs, am, aoffs, _ = oracle.pair(ev, offs, R)
    d_ev = torch.from_numpy(ev.view(np.uint8).reshape(-1).copy()).to(DEV)
    d_off = torch.from_numpy(offs.view(np.int64).copy()).to(DEV)
    cap = len(iv) - short
    p = argus.argus_pair_intervals(d_ev, d_off, R, interval_capacity=cap)
    room = torch.full((cap * 48 + 256,), 0x5A, dtype=torch.uint8, device=DEV)
    assert room.data_ptr() % 32 == 0
    p = dataclasses.replace(p, intervals=room[64 + shift:64 + shift + cap * 48])
    p = argus.argus_pair_intervals(d_ev, d_off, R, interval_capacity=cap, out=p)
    assert int(p.fetch_status()["code"]) == (4 if short else 0)
    got = room.cpu().numpy()
    assert (got[:64 + shift] == 0x5A).all() and (got[64 + shift + cap * 48:] == 0x5A).all()
    if not short:
        assert got[64 + shift:64 + shift + cap * 48].tobytes() == iv.tobytes()
