"""Iteration tables: iterations in order and out of order within a stream, with gaps, many and few streams, more iterations than
a block holds at a time and one only; and warp-role tables of CTA counts that are no multiple of a group, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_12299_b200 as argus

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("order", ["in-order", "shuffled", "sparse", "two-phases"])
@pytest.mark.parametrize("S,W,R,window", [(3, 1, 5, 7), (96, 4, 202, 16), (640, 16, 9, 1), (4800, 16, 3, 40)])
def test_iteration_table(order, S, W, R, window):
    rng = np.random.default_rng(S + window)
    per = 200_000 // S + 33
    lo = 11
    iv = np.zeros(S * per, argus.INTERVAL_DTYPE)
    base = np.sort(rng.integers(0, window + 20, per)) if order != "sparse" else np.sort(rng.choice([3, lo, lo + window // 2, lo + window - 1, lo + window], per))
    if order == "two-phases":
        base = np.concatenate([base[per // 2:], base[:per // 2]])
    for s in range(S):
        sl = slice(s * per, (s + 1) * per)
        iv["ctx"][sl] = rng.permutation(base) if order == "shuffled" else base
        iv["stream"][sl] = s
    iv["region"] = rng.integers(0, R, len(iv))
    iv["t_begin"] = rng.integers(0, 1 << 40, len(iv)).astype(np.uint64)
    iv["inclusive"] = (2.0 ** rng.uniform(0, 38, len(iv))).astype(np.uint64)
    iv["exclusive"] = iv["inclusive"] // np.uint64(3)
    iv["flags"] = rng.random(len(iv)) < 0.01
    offs = (np.arange(S + 1) * per).astype(np.uint64)
    C = S // W
    M = max(1, C // 2)
    cta_sm = (np.arange(C) % M).astype(np.uint32)
    levels = ("warp", "cta", "sm", "kernel", "role", "iter")
    _, want, _ = oracle.aggregate_scoped(iv, offs, None, None, W, cta_sm, M, R, scope={"ctx": (lo, lo + window - 1)}, levels=levels)
    d_iv = torch.from_numpy(iv.view(np.uint8).reshape(-1).copy()).to(DEV)
    d_off = torch.from_numpy(offs.view(np.int64).copy()).to(DEV)
    got = argus.argus_aggregate_scoped(d_iv, d_off, None, None, W, torch.from_numpy(cta_sm.view(np.int32)).to(DEV), M, R,
                                       argus.ArgusScope(lo, lo + window - 1), levels=levels)
    assert int(argus.argus_status_fetch(got.status)["code"]) == 0
    for lv in levels:
        assert got.table_numpy(lv).tobytes() == want[lv].tobytes(), lv


@pytest.mark.parametrize("shares", ["uniform", "skewed"])
@pytest.mark.parametrize("S,W,R,window", [(96, 4, 200, 16), (640, 16, 292, 9), (320, 16, 400, 16), (2400, 16, 400, 3)])
def test_many_regions(shares, S, W, R, window):
    """Up to the most regions that the tables in shared memory have room for, with regions that have copies of their cells among many
    that have none: a few hold most intervals, in some streams other ones than in the rest."""
    rng = np.random.default_rng(S + R)
    per = 400_000 // S + 65
    iv = np.zeros(S * per, argus.INTERVAL_DTYPE)
    iv["ctx"] = np.tile(np.sort(rng.integers(0, window + 6, per)), S)
    iv["stream"] = np.repeat(np.arange(S), per)
    iv["region"] = rng.integers(0, R, len(iv))
    if shares == "skewed":
        hot = rng.random(len(iv)) < 0.8
        iv["region"][hot] = (R - 1 - rng.choice(5, hot.sum(), p=[0.5, 0.2, 0.15, 0.1, 0.05]) - iv["stream"][hot] % 2 * 7).astype(np.uint32)
    iv["t_begin"] = rng.integers(0, 1 << 40, len(iv)).astype(np.uint64)
    iv["inclusive"] = (2.0 ** rng.uniform(0, 33, len(iv))).astype(np.uint64)  # (some of 2^32 ticks and more)
    iv["exclusive"] = iv["inclusive"] // np.uint64(2)
    iv["flags"] = rng.random(len(iv)) < 0.02
    offs = (np.arange(S + 1) * per).astype(np.uint64)
    cta_sm = (np.arange(S // W) % 5).astype(np.uint32)
    levels = ("warp", "kernel", "role", "iter")
    scope = (4, 4 + window - 1)
    _, want, _ = oracle.aggregate_scoped(iv, offs, None, None, W, cta_sm, 5, R, scope={"ctx": scope}, levels=levels)
    got = argus.argus_aggregate_scoped(torch.from_numpy(iv.view(np.uint8).reshape(-1).copy()).to(DEV), torch.from_numpy(offs.view(np.int64).copy()).to(DEV), None,
                                       None, W, torch.from_numpy(cta_sm.view(np.int32)).to(DEV), 5, R, argus.ArgusScope(*scope), levels=levels)
    assert int(argus.argus_status_fetch(got.status)["code"]) == 0
    for lv in levels:
        assert got.table_numpy(lv).tobytes() == want[lv].tobytes(), lv
