"""Kernels whose shared memory depends on the number of regions or rows, at sizes that together with the kernel's static arrays just pass the
48 KB which every kernel gets: calls are accepted whatever was called before, so each path runs in a process of its own, its smallest size first."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def synthesize(length, regions):
    from types import SimpleNamespace

    import numpy as np

    import helpers
    from paper_2609_12299_b200 import tracegen as tg
    from test_gpu_parity import _synthesize_matches
    spec = tg.TraceSpec(tg.GEMM, 1, 1)
    S, rng = spec.num_streams, np.random.default_rng(length)
    for R in regions:
        ev = np.zeros(2 * S * length, helpers.EVENT)
        region = rng.integers(0, R, S * length).astype(np.uint32)
        region[:3] = R - 1
        ev["tag"][0::2], ev["tag"][1::2] = region << 1, (region << 1) | 1
        ev["ts"] = (1 << 40) + np.cumsum(rng.integers(0, 90, len(ev)))
        offs = (np.arange(S + 1) * 2 * length).astype(np.uint64)
        case = SimpleNamespace(num_regions=R, warps_per_cta=spec.warps_per_cta, cta_sm=spec.cta_sm, num_sms=spec.num_sms,
                               overlap_pairs=np.array([[0, R - 1]], np.uint32))
        _synthesize_matches(case, ev, offs)


def attribute(rows):
    import numpy as np
    import torch

    from test_gpu_map import check_attribution
    rng = np.random.default_rng(3)
    for r in rows:
        counts = rng.integers(0, 50, (r, 70)).astype(np.uint64)
        check_attribution(torch.from_numpy(counts.view(np.int64)).to("cuda:0"), counts, rng.random(70))


# blocks of 512, 256 and 128 threads of the pass over the digests; the attribution of counts
@pytest.mark.parametrize("call", ["synthesize(8200, range(314, 323))", "synthesize(1500, range(346, 354))", "synthesize(40, range(346, 354))",
                                  "attribute(range(174, 195))"])
def test_sizes_in_a_fresh_process(call):
    r = subprocess.run([sys.executable, "-c", f"import test_gpu_shared_memory_limits as t; t.{call}"], cwd=HERE, capture_output=True, text=True, timeout=300,
                       env={**os.environ, "PYTHONPATH": os.pathsep.join([HERE, os.path.dirname(HERE), os.environ.get("PYTHONPATH", "")])})
    assert r.returncode == 0, r.stderr[-3000:]
