"""argus_overlap's kernel at the sizes where its branches change: spans in order or not, one role or both, around the number of
spans it holds in shared memory and the number of intervals an SM at which blocks have more threads, starts that crowd, many CTAs
an SM, and a workspace too small for the plain layout of the entries."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_12299_b200 as argus

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
TILE = 9216  # spans of both roles that fit shared memory at a time


def _intervals(rng, per_stream, S, order, other):
    """S streams of per_stream intervals of regions 0 and 1 (every `other`-th of region 2), as pairing orders them: by end."""
    iv = np.zeros(S * per_stream, argus.INTERVAL_DTYPE)
    for s in range(S):
        t = (1 << 40) + np.cumsum(rng.integers(1, 400, per_stream)).astype(np.uint64)
        d = np.minimum(rng.integers(0, 300, per_stream), np.append(np.diff(t.astype(np.int64)), 100)).astype(np.uint64)
        if order == "overlapping":
            d += np.uint64(900)
        elif order == "shuffled":
            p = rng.permutation(per_stream)
            t, d = t[p], d[p]
        elif order == "crowded":
            t = (1 << 40) + rng.integers(0, 50, per_stream).astype(np.uint64)
            t[:2] += np.uint64(1 << 35)
        sl = slice(s * per_stream, (s + 1) * per_stream)
        iv["stream"][sl], iv["t_begin"][sl], iv["inclusive"][sl] = s, t, d
        r = rng.integers(0, 2, per_stream)
        r[::other] = 2
        iv["region"][sl] = r
    return iv


@pytest.mark.parametrize("order", ["disjoint", "overlapping", "shuffled", "crowded"])
@pytest.mark.parametrize("per_stream", [1, 33, TILE // 4, TILE // 2, TILE // 2 + 1, 23_000, 65_535, 65_536])
def test_overlap_sizes_and_orders(order, per_stream):
    rng = np.random.default_rng(per_stream)
    S, W, M, other = 4, 2, 2, 3
    iv = _intervals(rng, per_stream, S, order, other)
    offs = (np.arange(S + 1) * per_stream).astype(np.uint64)
    cta_sm = np.array([1, 0], np.uint32)
    d_iv = torch.from_numpy(iv.view(np.uint8).reshape(-1).copy()).to(DEV)
    d_off = torch.from_numpy(offs.view(np.int64).copy()).to(DEV)
    d_sm = torch.from_numpy(cta_sm.view(np.int32)).to(DEV)
    for pairs in ([(0, 1)], [(1, 0), (2, 2), (0, 9)]):
        pairs_np = np.array(pairs, np.uint32)
        d_pairs = torch.from_numpy(pairs_np.view(np.int32)).to(DEV)
        _, want, _ = oracle.overlap(iv, offs, W, cta_sm, M, pairs_np)
        spans = sum(int(((iv["region"] == r) & (iv["inclusive"] > 0)).sum()) for p in pairs for r in p)
        # the whole workspace, and one with room for just the spans selected (fewer than the intervals)
        for ws in (None, argus.argus_overlap_workspace_bytes((spans + 1) // 2, S, 1, M)):
            out, st = argus.argus_overlap(d_iv, len(iv), d_off, W, d_sm, M, d_pairs, workspace_bytes=ws)
            assert int(argus.argus_status_fetch(st)["code"]) == 0
            assert out.cpu().numpy().view(argus.OVERLAP_DTYPE).reshape(want.shape).tobytes() == want.tobytes()


@pytest.mark.parametrize("order", ["disjoint", "overlapping", "shuffled", "crowded"])
@pytest.mark.parametrize("per_stream,S,W,M", [(1727, 4, 2, 2), (1729, 4, 2, 2), (3455, 4, 2, 2), (3457, 4, 2, 2), (4095, 4, 2, 2), (4096, 4, 2, 2), (100, 16, 16, 1), (700, 32, 16, 1),
                                              (6900, 4, 2, 2), (6912, 4, 2, 2), (6925, 4, 2, 2),
                                              (9, 48, 16, 7)])
def test_block_sizes(order, per_stream, S, W, M):
    """Around the spans that a block of 512 threads merges and sorts at a time, and with more slices of streams than a block takes at a
    time."""
    rng = np.random.default_rng(per_stream)
    iv = _intervals(rng, per_stream, S, order, 3)
    offs = (np.arange(S + 1) * per_stream).astype(np.uint64)
    cta_sm = (np.arange(S // W) % M).astype(np.uint32)
    pairs_np = np.array([(0, 1), (1, 1), (2, 0)], np.uint32)
    _, want, _ = oracle.overlap(iv, offs, W, cta_sm, M, pairs_np)
    out, st = argus.argus_overlap(torch.from_numpy(iv.view(np.uint8).reshape(-1).copy()).to(DEV), len(iv), torch.from_numpy(offs.view(np.int64).copy()).to(DEV),
                                  W, torch.from_numpy(cta_sm.view(np.int32)).to(DEV), M, torch.from_numpy(pairs_np.view(np.int32)).to(DEV))
    assert int(argus.argus_status_fetch(st)["code"]) == 0
    assert out.cpu().numpy().view(argus.OVERLAP_DTYPE).reshape(want.shape).tobytes() == want.tobytes()


@pytest.mark.parametrize("order", ["disjoint", "overlapping", "crowded"])
@pytest.mark.parametrize("S,W,M,per_stream", [(2080, 4, 4, 12), (640, 2, 2, 24), (96, 16, 1, 64)])
def test_many_ctas_an_sm_and_three_pairs(order, S, W, M, per_stream):
    """Few intervals an SM that lie in more CTAs than a block looks at at a time, and in several batches of
    slices for each of them: what a block keeps of its CTAs outlives the scans in between. Plain call and one-call pipeline."""
    rng = np.random.default_rng(S)
    iv = _intervals(rng, per_stream, S, order, 3)
    ev = np.zeros((S, per_stream, 2), argus.EVENT_DTYPE)
    ev["ts"][:, :, 0] = iv["t_begin"].reshape(S, -1)
    ev["ts"][:, :, 1] = (iv["t_begin"] + iv["inclusive"]).reshape(S, -1)
    ev["tag"] = np.stack([iv["region"] << 1, (iv["region"] << 1) | 1], axis=-1).reshape(S, per_stream, 2)
    offs = (np.arange(S + 1) * per_stream).astype(np.uint64)
    cta_sm = rng.integers(0, M, S // W).astype(np.uint32)
    pairs_np = np.array([(0, 1), (1, 1), (2, 0)], np.uint32)
    _, want, _ = oracle.overlap(iv, offs, W, cta_sm, M, pairs_np)
    d_sm, d_pairs = torch.from_numpy(cta_sm.view(np.int32)).to(DEV), torch.from_numpy(pairs_np.view(np.int32)).to(DEV)
    out, st = argus.argus_overlap(torch.from_numpy(iv.view(np.uint8).reshape(-1).copy()).to(DEV), len(iv), torch.from_numpy(offs.view(np.int64).copy()).to(DEV),
                                  W, d_sm, M, d_pairs)
    assert int(argus.argus_status_fetch(st)["code"]) == 0
    assert out.cpu().numpy().view(argus.OVERLAP_DTYPE).reshape(want.shape).tobytes() == want.tobytes()
    r = argus.argus_synthesize(torch.from_numpy(ev.reshape(-1).view(np.uint8).copy()).to(DEV), torch.from_numpy((2 * offs).view(np.int64).copy()).to(DEV), 3, W,
                               d_sm, M, d_pairs, max_overlap_spans=2 * 3 * len(iv))
    assert int(r.fetch_status()["code"]) == 0
    assert r.overlap_numpy(M).tobytes() == want.tobytes()


def test_sm_index_out_of_range_leaves_zeros_and_the_other_tables():
    """A CTA mapped to an SM that does not exist: the call reports it; the overlap is all zeros, and the tables hold every other
    CTA's intervals."""
    spec_sm = np.array([0, 1, 2], np.uint32)      # num_sms = 2
    S, W, R = 6, 2, 3
    ev = np.zeros((S, 4), argus.EVENT_DTYPE)
    ev["ts"] = np.arange(4) * 10
    ev["tag"] = [0, 2, 3, 1]
    offs = (np.arange(S + 1) * 4).astype(np.uint64)
    d_ev = torch.from_numpy(ev.reshape(-1).view(np.uint8).copy()).to(DEV)
    d_off = torch.from_numpy(offs.view(np.int64).copy()).to(DEV)
    d_pairs = torch.tensor([[0, 1]], dtype=torch.int32, device=DEV)
    r = argus.argus_synthesize(d_ev, d_off, R, W, torch.from_numpy(spec_sm.view(np.int32)).to(DEV), 2, d_pairs)
    st = r.fetch_status()
    assert int(st["code"]) == 1
    assert not r.overlap.cpu().numpy().any()
    assert int(r.agg.table_numpy("cta")["count"].sum()) == 12
    assert int(r.agg.table_numpy("sm")["count"].sum()) == int(r.agg.table_numpy("kernel")["count"].sum()) == 8
