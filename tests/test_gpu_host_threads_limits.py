"""Host threads as in test_gpu_host_threads, where both calls of a pair need more shared memory than a kernel gets without asking, which is checked: the
passes over the digests with blocks of 512, 256 and 128 threads, and argus_aggregate's pass over the records with blocks of 256, 192 and 128."""
import ctypes

import pytest
import torch

import paper_2609_12299_b200 as argus
import test_gpu_host_threads as base

pytestmark = pytest.mark.gpu


def _aggregate(regions, lib):
    spec, _, dev = base._trace(2, 300)
    S = spec.num_streams
    p = argus.argus_pair_intervals(dev[0], dev[1].view(torch.int64), regions)
    need = lib.argus_aggregate_workspace_bytes(0, S, regions)
    st, ws = base._new(64), base._new(need)
    out = [base._new(S * regions * 576), base._new(regions * 576)]
    args = (p.intervals.data_ptr(), p.interval_offsets.data_ptr(), None, None, S, spec.warps_per_cta, dev[2].data_ptr(), spec.num_sms, regions,
            out[0].data_ptr(), None, None, out[1].data_ptr(), st.data_ptr(), ws.data_ptr(), need)
    return (lambda stream: lib.argus_aggregate(*args, stream)), out, (dev, p, st, ws)


@pytest.mark.parametrize("what,one,other", [
    (base._synthesize, (400, 1300), (340, 1300)), (base._synthesize, (400, 300), (370, 300)), (base._synthesize, (400, 30), (370, 30)),
    (_aggregate, (400,), (200,)), (_aggregate, (330,), (300,)), (_aggregate, (365,), (335,)),  # 24 streams: 256, 192 and 128 threads
])
def test_both_calls_ask(what, one, other):
    lib = argus.load_library()
    lib.argus_testing_limit_requests.restype = ctypes.c_ulonglong
    for args in (one, other):
        call, _, keep = what(*args, lib)
        stream = torch.cuda.current_stream().cuda_stream
        assert call(stream) == 0
        before = lib.argus_testing_limit_requests()
        assert call(stream) == 0
        assert lib.argus_testing_limit_requests() == before + 1
        torch.cuda.synchronize()
    base.test_threads(what, one, other)
