"""The filtered ISA (csrc/k_isa.cu) where its plans have more offsets or coarser
granules: growth factors 3 and 4, batches with empty texts, and a text long
enough that a granule holds more than one position; repeats longer than one
plan covers (2^17) in all of them, no ISA output (which turns the filter off), at
most a quarter of the suffixes active. A missed entry would misplace suffixes:
the oracle's checker on every SA."""
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


def with_copies(recipe, seed, n, copies):
    """(source, target, length) segments copied inside a text."""
    t = gen.text(recipe, seed, n)
    for src, dst, size in copies:
        t[dst:dst + size] = t[src:src + size].copy()
    return t


@pytest.mark.parametrize("multiplier", [2, 3, 4])
@pytest.mark.parametrize("recipe,h0", [("dna", 0), ("dna", 16), ("zipf", 0)])
def test_growth_factors(gb, orc, multiplier, recipe, h0):
    import torch
    n = (1 << 22) + 77
    t = with_copies(recipe, 80 + multiplier, n, [(1000, n - 300001, 300001), (400001, 2000003, 150001)])
    sa, _, st, _ = gb.sa_build_ex(torch.from_numpy(t).cuda(), multiplier=multiplier, h0_chars=h0)
    assert st["rounds"] > 5 and st["active"][1] <= n // 4
    assert orc.check_sa(t, u32(sa)) == (0, -1)


@pytest.mark.parametrize("multiplier", [2, 4])
def test_batch(gb, orc, multiplier):
    import torch
    texts = [np.empty(0, np.uint8), with_copies("dna", 90, 1800001, [(777, 1500000, 200001)]), np.empty(0, np.uint8),
             gen.text("dna", 91, 900007), with_copies("dna", 92, 1700003, [(5, 1400000, 170003)]),
             np.full(3, 65, np.uint8), np.empty(0, np.uint8)]
    off = np.concatenate([[0], np.cumsum([x.size for x in texts])]).astype(np.uint64)
    assert int(off[-1]) > 1 << 22
    sa, st = gb.sa_build_batched(torch.from_numpy(np.concatenate(texts)).cuda(), off, stats=True, multiplier=multiplier)
    assert st["rounds"] > 5 and st["active"][1] <= int(off[-1]) // 4
    got = u32(sa)
    for k, x in enumerate(texts):
        if x.size:
            assert orc.check_sa(x, np.ascontiguousarray(got[int(off[k]):int(off[k + 1])])) == (0, -1), k


@pytest.mark.parametrize("multiplier", [2, 3])
def test_granules_of_two_positions(gb, orc, multiplier):
    import torch
    n = (1 << 26) + 12345
    t = with_copies("dna", 95, n, [(12347, 40000001, 400003), (9000001, 60000000, 270001), (1, n - 200003, 200003)])
    sa, _, st, _ = gb.sa_build_ex(torch.from_numpy(t).cuda(), multiplier=multiplier)
    assert st["rounds"] > 5 and st["active"][1] <= n // 4
    assert orc.check_sa(t, u32(sa)) == (0, -1)
