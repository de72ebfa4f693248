"""The direct form of sa_lcp (csrc/k_lcp.cu) and its hand-overs, against the
oracle; exact: texts around the 16-byte windows and the end of the text,
neighbours that agree in just under and over 16, 64 and 4096 characters
(listed pairs, and pairs that send a long text to the permuted form), texts
just below and above the size from which that form is an option, and an
unaligned text."""
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


def check(gb, orc, t, off=0):
    import torch
    t = np.ascontiguousarray(t)
    sa = orc.pd_sa(t)[0]
    d = torch.zeros(t.size + off, dtype=torch.uint8, device="cuda")[off:]
    d.copy_(torch.from_numpy(t))
    got = gb.sa_lcp(d, torch.from_numpy(sa.view(np.int32).copy()).cuda()).cpu().numpy().view(np.uint32)
    assert np.array_equal(got, orc.lcp(t, sa))


@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 31, 33, 1000, 65536, 65537, (1 << 20) + 3])
def test_short_prefixes(gb, orc, n):
    check(gb, orc, gen.text("dna", n, n))


@pytest.mark.parametrize("n", [60000, 70001, (1 << 20) + 5])
@pytest.mark.parametrize("size", [15, 17, 63, 64, 65, 300, 4095, 4200])
def test_one_repeat(gb, orc, n, size):
    t = gen.text("bytes", 5 * n + size, n)
    t[n // 2:n // 2 + size] = t[100:100 + size]
    t[n - size // 2:] = t[n // 3:n // 3 + size // 2]  # and one that ends with the text
    check(gb, orc, t)


@pytest.mark.parametrize("recipe", ["zipf_repeats", "markov"])
def test_repetitive(gb, orc, recipe):
    check(gb, orc, gen.text(recipe, 3, 200003))
    check(gb, orc, np.full(20001, 7, np.uint8))


@pytest.mark.parametrize("off", [1, 4, 8])
def test_unaligned(gb, orc, off):
    check(gb, orc, gen.text("dna", 9, 100001), off)
