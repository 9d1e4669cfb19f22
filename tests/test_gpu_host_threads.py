"""Host threads that call the same operation with different numbers of regions or rows, and so with different needs of shared
memory, each with its own stream and buffers: no call is refused, and the results are those of a call alone."""
import ctypes
import threading

import numpy as np
import pytest
import torch

import paper_2609_12299_b200 as argus
from paper_2609_12299_b200 import tracegen as tg
from paper_2609_12299_b200.binding import _ScopeStruct

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
CALLS = 2000


def _new(n):
    return torch.empty(int(n), dtype=torch.uint8, device=DEV)


def _attribute(rows, lib):
    P = 64
    g = torch.Generator(device=DEV).manual_seed(rows)
    counts = torch.randint(0, 50, (rows, P), dtype=torch.int64, device=DEV, generator=g)
    metric = torch.rand(P, dtype=torch.float64, device=DEV, generator=g)
    out, need = [_new(rows * 8), _new(P * 8), _new(rows * P * 8)], lib.argus_attribute_workspace_bytes(rows, P)
    ws = _new(need)
    args = (counts.data_ptr(), rows, P, metric.data_ptr(), *[t.data_ptr() for t in out], ws.data_ptr(), need)
    return (lambda stream: lib.argus_attribute(*args, stream)), out, (counts, metric, ws)


def _trace(ctas, iters):
    spec = tg.config(1).scaled(ctas, iters)
    ev, offs = tg.generate_host(spec)
    dev = [torch.from_numpy(np.ascontiguousarray(a).view(np.uint8).reshape(-1).copy()).to(DEV) for a in (ev, offs, spec.cta_sm, spec.overlap_pairs)]
    return spec, len(ev), dev


def _synthesize(regions, iters, lib):
    spec, n, dev = _trace(1, iters)
    S, W, M, K = spec.num_streams, spec.warps_per_cta, spec.num_sms, len(spec.overlap_pairs)
    need = lib.argus_synthesize_workspace_bytes(n, S, regions, 64, K, M, n)
    iv, io, am, ao, st, ws, cta = _new(n * 24), _new((S + 1) * 8), _new(64 * 32), _new((S + 1) * 8), _new(64), _new(need), _new(S * regions * 576)
    out = [_new(S * regions * 576), _new(regions * 576), _new(K * M * 32)]
    args = (dev[0].data_ptr(), n, dev[1].data_ptr(), S, regions, iv.data_ptr(), n // 2, io.data_ptr(), am.data_ptr(), 64, ao.data_ptr(), W,
            dev[2].data_ptr(), M, out[0].data_ptr(), cta.data_ptr(), None, out[1].data_ptr(), dev[3].data_ptr(), K, out[2].data_ptr(), n,
            st.data_ptr(), ws.data_ptr(), need)
    return (lambda stream: lib.argus_synthesize(*args, stream)), out, (dev, iv, io, am, ao, st, ws, cta)


def _iterations(regions, lib):
    spec, _, dev = _trace(1, 30)
    S = spec.num_streams
    p = argus.argus_pair_intervals(dev[0], dev[1].view(torch.int64), regions)
    scope = _ScopeStruct(3, 9, 2**64 - 1, None, None)
    need = lib.argus_aggregate_workspace_bytes(0, S, regions)
    st, ws = _new(64), _new(need)
    out = [_new(regions * 576), _new(7 * regions * 576)]
    args = (p.intervals.data_ptr(), p.interval_offsets.data_ptr(), None, None, S, spec.warps_per_cta, dev[2].data_ptr(), spec.num_sms, regions,
            ctypes.addressof(scope), None, None, None, out[0].data_ptr(), None, out[1].data_ptr(), st.data_ptr(), ws.data_ptr(), need)
    return (lambda stream: lib.argus_aggregate_scoped(*args, stream)), out, (dev, p, scope, st, ws)


# shared memory of the two: 102 and 51 KB, 89 and 49, 67 and 52 (512 threads), 55 and 51 (128 threads)
@pytest.mark.parametrize("what,one,other", [(_attribute, (400,), (200,)), (_iterations, (400,), (220,)), (_synthesize, (400, 1300), (280, 1300)),
                                            (_synthesize, (400, 30), (370, 30))])
def test_threads(what, one, other):
    lib = argus.load_library()
    jobs = [what(*a, lib) for a in (one, other, one, other)]
    for call, _, _ in jobs:
        assert call(torch.cuda.current_stream().cuda_stream) == 0
    torch.cuda.synchronize()
    want = [[t.clone() for t in out] for _, out, _ in jobs]
    refused = []

    def work(call):
        stream = torch.cuda.Stream()
        for i in range(CALLS):
            rc = call(stream.cuda_stream)
            if rc:
                refused.append((i, rc))
        stream.synchronize()

    threads = [threading.Thread(target=work, args=(call,)) for call, _, _ in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not refused, (len(refused), refused[:4])
    assert all(torch.equal(a, b) for (_, out, _), w in zip(jobs, want) for a, b in zip(out, w))
