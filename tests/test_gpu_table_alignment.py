"""Tables that start on 8 bytes but not on 16: rows are written 16 bytes at a time only where they lie on such a boundary. The passes over the
digests and over the records, one block a stream and several, against the oracle, and nothing written beside the tables."""
from dataclasses import replace

import numpy as np
import pytest
import torch

import oracle
import paper_2609_12299_b200 as argus
from paper_2609_12299_b200 import tracegen as tg
from paper_2609_12299_b200.binding import _synthesize_buffers

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
LEVELS = ("warp", "cta", "sm", "kernel")


# idx 1: five regions; idx 3: 202, of which most cells of a short stream stay empty
@pytest.mark.parametrize("idx,ctas,iters,defects", [(1, 2, 40, False), (1, 80, 12, False), (1, 3, 1500, False), (3, 30, 1, False), (4, 80, 30, True)])
@pytest.mark.parametrize("shift", [0, 8])
def test_rows_on_8_bytes(idx, ctas, iters, defects, shift):
    spec = tg.config(idx).scaled(ctas, iters)
    ev, offs = tg.generate_host(spec)
    R, W, M, S, C = spec.num_regions, spec.warps_per_cta, spec.num_sms, spec.num_streams, spec.num_streams // spec.warps_per_cta
    _, iv, ioffs, am, aoffs, _ = oracle.pair(ev, offs, R)
    assert bool(len(am)) == defects
    _, want, _ = oracle.aggregate(iv, ioffs, am, aoffs, W, spec.cta_sm, M, R)
    d_ev, d_off = torch.from_numpy(ev.view(np.uint8).reshape(-1).copy()).to(DEV), torch.from_numpy(offs.view(np.int64).copy()).to(DEV)
    d_sm, pairs = torch.from_numpy(spec.cta_sm.view(np.int32)).to(DEV), torch.from_numpy(spec.overlap_pairs.view(np.int32)).to(DEV)
    sizes = {lv: n * R * 576 for lv, n in zip(LEVELS, (S, C, M, 1))}

    def shifted(agg):
        room = {lv: torch.full((n + 256,), 0x5A, dtype=torch.uint8, device=DEV) for lv, n in sizes.items()}
        assert all(t.data_ptr() % 16 == 0 for t in room.values())
        return room, replace(agg, **{lv: t[64 + shift:64 + shift + sizes[lv]] for lv, t in room.items()})

    def check(room, agg):
        for lv in LEVELS:
            assert agg.table_numpy(lv).tobytes() == want[lv].tobytes(), lv
            assert bool((room[lv][:64 + shift] == 0x5A).all()) and bool((room[lv][64 + shift + sizes[lv]:] == 0x5A).all()), lv

    out = _synthesize_buffers(d_ev.device, len(ev), S, len(spec.overlap_pairs), R, W, M, None, None, None, LEVELS)
    room, agg = shifted(out.agg)
    res = argus.argus_synthesize(d_ev, d_off, R, W, d_sm, M, pairs, out=replace(out, agg=agg))
    assert int(res.fetch_status()["code"]) == 0
    check(room, res.agg)

    p = argus.argus_pair_intervals(d_ev, d_off, R)
    args = (p.intervals, p.interval_offsets, p.ambig, p.ambig_offsets, W, d_sm, M, R)
    room, agg = shifted(argus.argus_aggregate(*args))
    got = argus.argus_aggregate(*args, out=agg)
    assert int(argus.argus_status_fetch(got.status)["code"]) == 0
    check(room, got)
