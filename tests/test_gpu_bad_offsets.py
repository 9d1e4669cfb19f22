"""Offsets that decrease: the lengths of the streams add up to more than there are events. Such a call reports ARGUS_ERR_BAD_OFFSETS and
touches nothing behind the workspace that it asked for, nor behind its outputs."""
import numpy as np
import pytest
import torch

import paper_2609_12299_b200 as argus

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
GUARD, MARK = 8 << 20, 0xA5
BAD_OFFSETS = 7


def _guarded(n):
    t = torch.full((int(n) + GUARD,), MARK, dtype=torch.uint8, device=DEV)
    assert t.data_ptr() % 256 == 0
    return t


def _untouched(t, n):
    return bool((t[int(n):] == MARK).all())


def _input(n, streams, length):
    """n markers, begin and end in turn; streams that are, in turn, the first `length` of them and an impossible one."""
    ev = np.zeros(n, argus.EVENT_DTYPE)
    ev["ts"] = np.arange(n, dtype=np.uint64) * np.uint64(3)
    ev["tag"] = np.arange(n, dtype=np.uint32) & 1
    offs = np.array([0, length] * (streams // 2) + [0], np.int64)
    return torch.from_numpy(ev.view(np.uint8).reshape(-1).copy()).to(DEV), torch.from_numpy(offs).to(DEV)


# the larger one: few long streams, whose segments outnumber what fits so many events
@pytest.mark.parametrize("n,streams,length", [(1000, 4, 1000), (1 << 21, 200, 30_000)])
def test_pairing(n, streams, length):
    ev, off = _input(n, streams, length)
    lib = argus.load_library()
    icap = streams * length
    need = lib.argus_pair_workspace_bytes(n, streams, n)
    ws, iv, am, st = _guarded(need), _guarded(icap * 48), _guarded(n * 32), _guarded(64)
    io, ao = _guarded((streams + 1) * 8), _guarded((streams + 1) * 8)
    rc = lib.argus_pair_intervals(ev.data_ptr(), n, off.data_ptr(), streams, 1, iv.data_ptr(), icap, io.data_ptr(), am.data_ptr(), n,
                                  ao.data_ptr(), st.data_ptr(), ws.data_ptr(), need, torch.cuda.current_stream().cuda_stream)
    assert rc == 0 and int(argus.argus_status_fetch(st)["code"]) == BAD_OFFSETS
    assert all(_untouched(t, k) for t, k in ((ws, need), (iv, icap * 48), (am, n * 32), (st, 64), (io, (streams + 1) * 8), (ao, (streams + 1) * 8)))


@pytest.mark.parametrize("num_pairs", [0, 1])
@pytest.mark.parametrize("n,streams,length", [(1000, 4, 1000), (1 << 20, 80, 30_000), (1 << 21, 200, 30_000)])
def test_synthesize(n, streams, length, num_pairs):
    """Room for more intervals than so many events can hold: the digests beside them stop where their array does."""
    ev, off = _input(n, streams, length)
    lib = argus.load_library()
    icap, sms, spans = streams * length, 2, n
    cta_sm, pairs = torch.zeros(streams, dtype=torch.int32, device=DEV), torch.zeros(2, dtype=torch.int32, device=DEV)
    need = lib.argus_synthesize_workspace_bytes(n, streams, 1, n, num_pairs, sms, spans)
    ws, iv, am, st = _guarded(need), _guarded(icap * 48), _guarded(n * 32), _guarded(64)
    io, ao = _guarded((streams + 1) * 8), _guarded((streams + 1) * 8)
    tabs, ov = [_guarded(k * 576) for k in (streams, streams, sms, 1)], _guarded(sms * 32)
    rc = lib.argus_synthesize(ev.data_ptr(), n, off.data_ptr(), streams, 1, iv.data_ptr(), icap, io.data_ptr(), am.data_ptr(), n, ao.data_ptr(), 1,
                              cta_sm.data_ptr(), sms, *[t.data_ptr() for t in tabs], pairs.data_ptr(), num_pairs, ov.data_ptr(), spans,
                              st.data_ptr(), ws.data_ptr(), need, torch.cuda.current_stream().cuda_stream)
    assert rc == 0 and int(argus.argus_status_fetch(st)["code"]) == BAD_OFFSETS
    assert all(_untouched(t, k) for t, k in ((ws, need), (iv, icap * 48), (am, n * 32), (st, 64), (io, (streams + 1) * 8), (ao, (streams + 1) * 8)))
    assert all(_untouched(t, k * 576) for t, k in zip(tabs, (streams, streams, sms, 1))) and _untouched(ov, sms * 32)
