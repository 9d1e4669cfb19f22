"""The pass over the digests: 128, 256 or 512 threads a stream by the streams' average length, with and without copies
of the hot regions' cells, on both sides of each line; wide intervals, carries, flags and ambiguity records among them."""
import numpy as np
import pytest

import paper_2609_12299_b200 as argus
from paper_2609_12299_b200 import tracegen as tg
from test_gpu_parity import _synthesize_matches

pytestmark = pytest.mark.gpu


def _stream(rng, n, shares, wide):
    region = rng.choice(5, size=n, p=shares).astype(np.uint32)
    dur = np.where(rng.random(n) < 0.5, rng.integers(1 << 21, 1 << 23, n), rng.integers(0, 300, n))
    dur = np.where(rng.random(n) < wide, rng.integers(1 << 23, 1 << 36, n), dur).astype(np.uint64)
    ev = np.zeros(2 * n, argus.EVENT_DTYPE)
    ev["ts"][0::2] = (1 << 33) + np.concatenate([[0], np.cumsum(dur + np.uint64(3))[:-1]]).astype(np.uint64)[:n]
    ev["ts"][1::2] = ev["ts"][0::2] + dur
    ev["tag"][0::2], ev["tag"][1::2] = region << 1, (region << 1) | 1
    ev["ctx"][0::2] = ev["ctx"][1::2] = np.arange(n, dtype=np.uint32)
    ev["ctx"][1::2] += rng.random(n) < 0.01          # flagged
    return ev[rng.random(2 * n) >= 0.002] if wide else ev  # lost markers: ambiguity records


@pytest.mark.parametrize("wide", [0.0, 0.01, 1.0])
@pytest.mark.parametrize("length", [1, 511, 512, 1023, 1024, 2047, 8191, 8192, 8225])
def test_stream_lengths(length, wide):
    rng = np.random.default_rng(length)
    spec = tg.TraceSpec(tg.GEMM, 2, 1)  # only for warps_per_cta, cta_sm and pairs
    shares = [[0.2] * 5, [0.9, 0.05, 0.05, 0, 0], [0, 0, 0, 0, 1.0], [0.3, 0.3, 0.2, 0.1, 0.1]]
    streams = [_stream(rng, length, shares[s % 4], wide) for s in range(spec.num_streams)]
    if length > 40:  # the same average with an empty stream, a short one and a long one
        streams[3] = _stream(rng, 2 * length - 31, shares[1], wide)
        streams[4] = _stream(rng, 31, shares[0], wide)
        streams[5], streams[6] = streams[5][:0], _stream(rng, 2 * length, shares[2], wide)
    offs = np.cumsum([0] + [len(e) for e in streams]).astype(np.uint64)
    _synthesize_matches(spec, np.concatenate(streams), offs)
