"""Texts that end in a run of their smallest character (csrc/k_local.cu): its code
is the padding's, so the run's tail suffixes have the run's own key. Exact
against the oracle around the sizes of a bin and of a tile, in batches of such
texts; and no slower than a run of another character."""
import time

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


def ending_in(kind, n, run, symbol=min):
    t = gen.text(kind, 50 + run % 7, n)
    t[n - run:] = symbol(t)
    return t


@pytest.mark.parametrize("run", [1, 31, 32, 33, 63, 64, 65, 95, 600, 2559, 2560, 2900, 3073])
@pytest.mark.parametrize("kind", ["dna", "zipf", "bytes"])
def test_runs(gb, orc, kind, run):
    import torch
    t = ending_in(kind, 9001, run)
    want_sa, want_isa, _, _ = orc.pd_sa(t)
    d = torch.from_numpy(t).cuda()
    for kw in ({}, {"h0_chars": 20}, {"paper_names": True}):
        sa, isa, _, _ = gb.sa_build_ex(d, isa=True, **kw)
        assert np.array_equal(u32(sa), want_sa), kw
        assert np.array_equal(u32(isa), want_isa), kw


@pytest.mark.parametrize("h0", [0, 3, 33])
def test_batch(gb, orc, h0):
    import torch
    texts = [np.full(k, 66, np.uint8) for k in (1, 40, 63, 64, 65, 700, 2000, 2900, 3500)]
    texts += [ending_in("dna", 2000 + k, 40 + 100 * k) for k in range(12)] + [np.empty(0, np.uint8)]
    off = np.concatenate([[0], np.cumsum([x.size for x in texts])]).astype(np.uint64)
    got = u32(gb.sa_build_batched(torch.from_numpy(np.concatenate(texts)).cuda(), off, h0_chars=h0))
    for k, x in enumerate(texts):
        if x.size:
            assert np.array_equal(got[int(off[k]):int(off[k + 1])], orc.pd_sa(x)[0]), k


@pytest.mark.parametrize("kind", ["dna", "zipf"])
def test_as_fast_as_another_character(gb, kind):
    """2500 of the smallest byte at the end of 2^20 characters against 2500 of the
    largest: compared all against all the former took twice as long."""
    import torch
    best = []
    for symbol in (min, max):
        d = torch.from_numpy(ending_in(kind, 1 << 20, 2500, symbol)).cuda()
        times = []
        for _ in range(25):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            gb.sa_build(d)
            torch.cuda.synchronize()
            times.append(time.perf_counter() - t0)
        best.append(min(times))
    assert best[0] < 1.4 * best[1]
