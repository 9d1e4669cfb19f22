"""CTAs that are mapped to an SM that does not exist: every entry point names the first such CTA's first stream, as the oracle does,
whichever of their streams is met first."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_12299_b200 as argus
from paper_2609_12299_b200 import tracegen as tg

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _told(st):
    return int(st["code"]), int(st["bad_stream"]), int(st["bad_event"])


@pytest.mark.parametrize("bad", [(22,), (5, 9, 21), tuple(range(1, 23)), (0, 22)])
def test_first_stream_of_the_first_bad_cta(bad):
    spec = tg.config(0).scaled(23, 120)
    W, M, R = spec.warps_per_cta, 7, spec.num_regions
    cta_sm = (np.arange(spec.num_ctas) % M).astype(np.uint32)
    cta_sm[list(bad)] = M + np.arange(len(bad), dtype=np.uint32) % 3
    ev, offs = tg.generate_host(spec)
    _, iv, ioffs, am, aoffs, _ = oracle.pair(ev, offs, R)
    pairs = spec.overlap_pairs
    want = (1, min(bad) * W, int(cta_sm[min(bad)]))
    assert _told(oracle.aggregate(iv, ioffs, am, aoffs, W, cta_sm, M, R)[-1]) == want
    assert _told(oracle.overlap(iv, ioffs, W, cta_sm, M, pairs)[-1]) == want
    d_ev, d_off = torch.from_numpy(ev.view(np.uint8).reshape(-1).copy()).to(DEV), torch.from_numpy(offs.view(np.int64).copy()).to(DEV)
    d_sm, d_pairs = torch.from_numpy(cta_sm.view(np.int32)).to(DEV), torch.from_numpy(pairs.view(np.int32).copy()).to(DEV)
    scope = argus.ArgusScope(0, 1 << 30, sm_mask=torch.full((1,), -1, dtype=torch.int32, device=DEV))
    p = argus.argus_pair_intervals(d_ev, d_off, R)
    for _ in range(20):
        a = argus.argus_aggregate(p.intervals, p.interval_offsets, p.ambig, p.ambig_offsets, W, d_sm, M, R)
        _, ov_st = argus.argus_overlap(p.intervals, p.interval_capacity, p.interval_offsets, W, d_sm, M, d_pairs)
        sc = argus.argus_aggregate_scoped(p.intervals, p.interval_offsets, p.ambig, p.ambig_offsets, W, d_sm, M, R, scope)
        _, sc_st = argus.argus_overlap_scoped(p.intervals, p.interval_capacity, p.interval_offsets, W, d_sm, M, d_pairs, scope)
        r = argus.argus_synthesize(d_ev, d_off, R, W, d_sm, M, d_pairs)
        for st in (a.status, ov_st, sc.status, sc_st):
            assert _told(argus.argus_status_fetch(st)) == want
        assert _told(r.fetch_status()) == want
