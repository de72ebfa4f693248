"""The refine's pivot path (csrc/k_refine.cu) at its edges, against the oracle;
exact SA and ISA: copies of a block with few, many and very many
substitutions per copy (none, some and most tiles take it; lists up to and
past their limit), group sizes below and above the limits of every tile shape,
the paper's names, and a batch."""
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


@pytest.fixture(scope="module")
def orc():
    import oracle
    return oracle.get()


def u32(x):
    return x.cpu().numpy().view(np.uint32)


def copies(size, count, rate, seed):
    rng = np.random.default_rng(seed)
    t = np.tile(gen.text("zipf", seed, size), count)
    m = rng.random(t.size) < rate
    t[m] = rng.integers(1, 255, int(m.sum()))
    return t.astype(np.uint8)


@pytest.mark.parametrize("shape", [1, 2, 3, 4])
@pytest.mark.parametrize("size,count,rate", [(97, 250, 0.0), (97, 250, 0.001), (211, 383, 0.004), (211, 385, 0.02),
                                             (53, 511, 0.1), (53, 514, 0.005), (31, 2050, 0.01)])
def test_copies(gb, orc, shape, size, count, rate):
    import torch
    t = copies(size, count, rate, size + count)
    want_sa, want_isa, _, _ = orc.pd_sa(t)
    sa, isa, _, _ = gb.sa_build_ex(torch.from_numpy(t).cuda(), isa=True, refine_shape=shape, h0_chars=4)
    assert np.array_equal(u32(sa), want_sa)
    assert np.array_equal(u32(isa), want_isa)


def test_paper_names(gb, orc):
    import torch
    t = copies(101, 200, 0.004, 5)
    _, _, st, trace = gb.sa_build_ex(torch.from_numpy(t).cuda(), paper_names=True, h0_chars=2, trace_cap=32,
                                     refine_shape=2)
    _, _, rounds, names = orc.pd_sa(t, h0=2, trace_cap=32)
    assert st["rounds"] == rounds + 1
    assert np.array_equal(u32(trace[:st["rounds"]]), np.asarray(names[:st["rounds"]], dtype=np.uint32))


def test_batch(gb, orc):
    import torch
    texts = [copies(40 + 7 * k, 150, 0.01, 60 + k) for k in range(12)]
    off = np.concatenate([[0], np.cumsum([x.size for x in texts])]).astype(np.uint64)
    got = u32(gb.sa_build_batched(torch.from_numpy(np.concatenate(texts)).cuda(), off, h0_chars=3))
    for k, x in enumerate(texts):
        assert np.array_equal(got[int(off[k]):int(off[k + 1])], orc.pd_sa(x)[0]), k
