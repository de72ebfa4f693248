"""Calls on a stream that is not torch's current one: what the binding
allocates, fills or copies on the current stream is ordered before the call,
and what the call still uses after its return is kept from other uses."""
import numpy as np
import pytest

import gen

pytestmark = pytest.mark.gpu

BUSY = 20_000_000  # clock cycles (about 10 ms) one stream is kept busy


@pytest.fixture(scope="module")
def gb():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1610_03007_gb300 as g
    g.load()
    return g


def u32(x):
    return x.cpu().numpy().view(np.uint32)


def test_bwt_and_trace_while_the_current_stream_is_busy(gb, orc):
    import torch
    t = gen.text("zipf_repeats", 31, 60001)
    d = torch.from_numpy(np.repeat(t, 2)).cuda()[::2]  # made contiguous by the call
    sa = torch.from_numpy(orc.pd_sa(t)[0].view(np.int32)).cuda()
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    torch.cuda._sleep(BUSY)
    bwt, primary = gb.sa_bwt(d, sa, stream=s)
    want, want_primary = orc.bwt(t, u32(sa))
    assert primary == want_primary
    assert np.array_equal(bwt.cpu().numpy(), want)
    torch.cuda._sleep(BUSY)
    _, _, st, trace = gb.sa_build_ex(d, paper_names=True, h0_chars=2, trace_cap=32, stream=s)
    _, _, rounds, names = orc.pd_sa(t, h0=2, trace_cap=32)
    assert st["rounds"] == rounds + 1
    assert np.array_equal(u32(trace[:st["rounds"]]), np.asarray(names[:st["rounds"]], dtype=np.uint32))


def test_lcp_buffers_outlive_the_call(gb, orc):
    import torch
    t = gen.text("zipf_repeats", 32, 70001)
    want = orc.lcp(t, orc.pd_sa(t)[0])
    d = torch.from_numpy(t).cuda()
    sa = gb.sa_build(d)
    s = torch.cuda.Stream()
    size = gb.load().sa_lcp_workspace_bytes(t.size)
    torch.cuda.synchronize()
    for _ in range(3):
        with torch.cuda.stream(s):
            torch.cuda._sleep(BUSY)
        lcp = gb.sa_lcp(d, sa, stream=s)
        torch.empty(size, dtype=torch.uint8, device="cuda").fill_(0x5A)
        s.synchronize()
        assert np.array_equal(u32(lcp), want)
