"""An interval array that is too small: the call reports it, and the records that fit are right and lie where they belong, on arrays that start on a
32-byte boundary and 16 bytes behind one."""
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
@pytest.mark.parametrize("short", [1, 2, 3, 701])
def test_records_that_fit(shift, short):
    spec = tg.config(1).scaled(3, 37)
    ev, offs = tg.generate_host(spec)
    _, iv, _, _, _, _ = oracle.pair(ev, offs, spec.num_regions)
    d_ev, d_off = torch.from_numpy(ev.view(np.uint8).reshape(-1).copy()).to(DEV), torch.from_numpy(offs.view(np.int64).copy()).to(DEV)
    cap = len(iv) - short
    room = torch.full((cap * 48 + 256,), 0x5A, dtype=torch.uint8, device=DEV)
    assert room.data_ptr() % 32 == 0
    p = argus.argus_pair_intervals(d_ev, d_off, spec.num_regions, interval_capacity=cap)
    p = argus.argus_pair_intervals(d_ev, d_off, spec.num_regions, out=dataclasses.replace(p, intervals=room[64 + shift:64 + shift + cap * 48]))
    st = p.fetch_status()
    assert int(st["code"]) == 4 and int(st["intervals_required"]) == len(iv)
    assert p.intervals_numpy().tobytes() == iv[:cap].tobytes()
    got = room.cpu().numpy()
    assert (got[:64 + shift] == 0x5A).all() and (got[64 + shift + cap * 48:] == 0x5A).all()
