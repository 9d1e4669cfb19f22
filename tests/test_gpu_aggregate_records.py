"""argus_aggregate's pass over the records: streams that end at, before and behind the edges of a tile of 256, 192 or 128 records and of the four tiles from
which on frequent regions get copies of their cells, streams that several blocks share, durations around 2^32, one region and 400, and a record
of a region that does not exist, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_12299_b200 as argus

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
EDGES = [0, 1, 127, 128, 129, 191, 192, 193, 255, 256, 257, 385, 511, 512, 513, 767, 768, 769, 1023, 1024, 1025, 3000]


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.uint8).reshape(-1).copy()).to(DEV)


@pytest.mark.parametrize("R", [1, 5, 65, 148, 400])
@pytest.mark.parametrize("S,W", [(12, 3), (24, 1), (900, 12), (1080, 12), (736, 16)])  # sixteen blocks a stream, sixteen, one (of 256, 192 and 128 threads, by R)
def test_tables(S, W, R):
    rng = np.random.default_rng(S + R)
    lengths = np.array([EDGES[s % len(EDGES)] for s in range(S)])
    offs = np.concatenate([[0], np.cumsum(lengths)]).astype(np.uint64)
    n = int(offs[-1])
    iv = np.zeros(n, argus.INTERVAL_DTYPE)
    iv["stream"] = np.repeat(np.arange(S), lengths)
    iv["region"] = np.minimum(rng.geometric(0.3, n) - 1, R - 1)   # a few regions own most
    iv["region"][rng.random(n) < 0.2] = rng.integers(0, R)
    iv["inclusive"] = (2.0 ** rng.uniform(0, 31.99, n)).astype(np.uint64)
    far = rng.random(n) < 0.003
    iv["inclusive"][far] = rng.choice(np.array([0, (1 << 32) - 2, (1 << 32) - 1, 1 << 32, (1 << 63) + 5], np.uint64), int(far.sum()))
    iv["exclusive"] = iv["inclusive"] - iv["inclusive"] // np.uint64(3)
    iv["flags"] = rng.random(n) < 0.01
    am = np.zeros(3 * S, argus.AMBIG_DTYPE)
    am["tag"] = (rng.integers(0, R, len(am)) << 1) | rng.integers(0, 2, len(am))
    am["kind"] = rng.integers(0, 3, len(am))
    aoffs = (np.arange(S + 1) * 3).astype(np.uint64)
    C = S // W
    M = max(1, C // 2)
    cta_sm = (np.arange(C) % M).astype(np.uint32)
    _, want, st = oracle.aggregate(iv, offs, am, aoffs, W, cta_sm, M, R)
    assert int(st["code"]) == 0
    d_sm = torch.from_numpy(cta_sm.view(np.int32)).to(DEV)
    args = (torch.from_numpy(offs.view(np.int64)).to(DEV), _dev(am), torch.from_numpy(aoffs.view(np.int64)).to(DEV), W, d_sm, M, R)
    got = argus.argus_aggregate(_dev(iv), *args)
    assert int(argus.argus_status_fetch(got.status)["code"]) == 0
    for lv in ("warp", "cta", "sm", "kernel"):
        assert got.table_numpy(lv).tobytes() == want[lv].tobytes(), lv
    iv["region"][n // 2] = R
    bad = argus.argus_aggregate(_dev(iv), *args)
    assert int(argus.argus_status_fetch(bad.status)["code"]) == 6 and int(argus.argus_status_fetch(bad.status)["bad_event"]) == n // 2
