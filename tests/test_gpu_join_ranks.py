"""Order statistics of the join for numbers of samples and distributions that take the different ways: few samples, one bin that holds
more than a warp ranks, equal values, the whole 64-bit range; all three joins against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_12299_b200 as argus

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _dev(a):
    return torch.from_numpy(a.view(np.uint8).reshape(-1).copy()).to(DEV)


@pytest.mark.parametrize("values", ["spread", "equal", "two", "narrow", "one-huge", "all-bits"])
def test_ranks(values):
    rng = np.random.default_rng(len(values))
    sizes = [1, 2, 5, 63, 64, 65, 257, 1000, 2049, 4096]
    ref = np.zeros(len(sizes), argus.INTERVAL_DTYPE)
    ref["region"] = np.arange(len(sizes))
    parts = []
    for r, n in enumerate(sizes):
        v = {"spread": lambda: np.exp(rng.normal(6, 0.8, n)).astype(np.uint64),
             "equal": lambda: np.full(n, 1234567, np.uint64),
             "two": lambda: rng.integers(0, 2, n).astype(np.uint64) * np.uint64((1 << 40) + 1),
             "narrow": lambda: rng.integers(100_000, 100_900, n).astype(np.uint64),
             "one-huge": lambda: np.append(rng.integers(0, 40, n - 1).astype(np.uint64), np.uint64((1 << 64) - 1)),
             "all-bits": lambda: rng.integers(0, 1 << 64, n, dtype=np.uint64)}[values]()
        p = np.zeros(n, argus.INTERVAL_DTYPE)
        p["region"], p["inclusive"] = r, v
        parts.append(p)
    smp = np.concatenate(parts)
    smp = smp[rng.permutation(len(smp))]
    idx = np.arange(len(sizes)).astype(np.uint64)
    _, want, _ = oracle.join_samples(ref, idx, smp)
    d_ref, d_smp, d_idx = _dev(ref), _dev(smp), torch.from_numpy(idx.view(np.int64).copy()).to(DEV)
    d_off = torch.tensor([[0, len(smp)]], dtype=torch.int64, device=DEV)
    for out, st in (argus.argus_join_samples(d_ref, d_idx, d_smp), argus.argus_join_samples_hashed(d_ref, d_idx, d_smp),
                    argus.argus_join_samples_grouped(d_ref, d_idx, d_smp, d_off, 1)):
        assert int(argus.argus_status_fetch(st)["code"]) == 0
        assert out.cpu().numpy()[: len(sizes) * 64].view(argus.JOIN_DTYPE).tobytes() == want.tobytes()


@pytest.mark.parametrize("n", [1, 255, 256, 257, 2047, 2048, 2049, 4097])
def test_scan_lengths(n):
    """Samples around the numbers that a block asks for at a time: the last ones count, those past the end of a range do not."""
    rng = np.random.default_rng(n)
    ref = np.zeros(3, argus.INTERVAL_DTYPE)
    ref["region"], ref["stream"] = [0, 1, 0], [0, 0, 1]
    smp = np.zeros(2 * n + 3, argus.INTERVAL_DTYPE)
    smp["region"], smp["inclusive"] = rng.integers(0, 2, len(smp)), rng.integers(1, 1 << 40, len(smp))
    smp["region"][n - 1], smp["stream"][n:] = 0, 1
    idx = np.arange(3, dtype=np.uint64)
    _, want, _ = oracle.join_samples(ref, idx, smp)
    d_ref, d_smp, d_idx = _dev(ref), _dev(smp), torch.from_numpy(idx.view(np.int64).copy()).to(DEV)
    d_off = torch.tensor([[0, n, len(smp)]], dtype=torch.int64, device=DEV)
    for out, st in (argus.argus_join_samples(d_ref, d_idx, d_smp), argus.argus_join_samples_grouped(d_ref, d_idx, d_smp, d_off, 2)):
        assert int(argus.argus_status_fetch(st)["code"]) == 0
        assert out.cpu().numpy()[: 3 * 64].view(argus.JOIN_DTYPE).tobytes() == want.tobytes()
