"""A build's results are complete when the call returns (include/gbsa.h), with
every output the options add: nothing of it is left on the stream, so the
workspace may be used again at once on another one."""
import numpy as np
import pytest

import gen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1610_03007_gb300 as g
    g.load()
    return g


def u32(x):
    return x.cpu().numpy().view(np.uint32)


@pytest.mark.parametrize("recipe,n,kw", [("dna", 1, {"isa": True}), ("dna", 1 << 24, {"isa": True}),
                                         ("zipf_repeats", 1 << 22, {"isa": True}), ("dna", (1 << 25) + 3, {"isa": True}),
                                         ("dna", (1 << 25) + 3, {"isa": True, "bucket_min": 1 << 20}),
                                         ("dna", 70001, {"isa": True, "trace_cap": 2}),
                                         ("dna", 1 << 24, {"trace_cap": 1})])
def test_nothing_left_on_the_stream(gb, orc, recipe, n, kw):
    import torch
    t = gen.text(recipe, 21, n)
    d = torch.from_numpy(t).cuda()
    s = torch.cuda.Stream()
    ws = torch.empty(gb.workspace_bytes(n), dtype=torch.uint8, device="cuda")
    gb.sa_build_ex(d, workspace=ws, stream=s, **kw)  # first launches set the kernels up
    torch.cuda.synchronize()
    for _ in range(3):
        sa, isa, _, _ = gb.sa_build_ex(d, workspace=ws, stream=s, **kw)
        assert s.query()
        ws.fill_(0x5A)  # on the current stream, which does not wait for s
    torch.cuda.synchronize()
    assert orc.check_sa(t, u32(sa)) == (0, -1)
    if isa is not None:
        inverse = np.empty(n, np.uint32)
        inverse[u32(sa)] = np.arange(n, dtype=np.uint32)
        assert np.array_equal(u32(isa), inverse)
