"""Round 0 by buckets of equal top bits (csrc/k_local.cu) and the filtered ISA
entries (csrc/k_isa.cu) at their edges, against the oracle; exact.

Texts whose buckets end around a tile's window (2560 positions) and its last
slot (3072), whose bins hold runs of equal keys, runs beside a tail suffix,
two keys that agree for many bits, buckets too large for a tile (alone or
among small ones), and batches of such texts; and a text long enough
(2^22) that only the needed ISA entries are written, with repeats longer than
one plan of offsets covers."""
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


def two_blocks():
    """286 copies of a 70-character block that differ in one late character:
    keys that agree in their first 60 bits."""
    block = np.random.default_rng(1).integers(0, 2, 70).astype(np.uint8)
    pick = np.random.default_rng(2).integers(0, 2, 286)
    out = np.tile(block, 286)
    out[60::70] = pick
    return out


TEXTS = {
    "dna 2": lambda: gen.text("dna", 1, 2), "dna 2559": lambda: gen.text("dna", 2, 2559),
    "dna 2560": lambda: gen.text("dna", 3, 2560), "dna 2561": lambda: gen.text("dna", 4, 2561),
    "dna 3072": lambda: gen.text("dna", 5, 3072), "dna 3073": lambda: gen.text("dna", 6, 3073),
    "dna 65537": lambda: gen.text("dna", 7, 65537), "zipf 100003": lambda: gen.text("zipf", 8, 100003),
    "bytes 300007": lambda: gen.text("bytes", 9, 300007), "run": lambda: np.full(7001, 97, np.uint8),
    "binary": lambda: np.random.default_rng(3).integers(0, 2, 50001).astype(np.uint8),
    "repeats": lambda: gen.text("zipf_repeats", 10, 70001), "two blocks": two_blocks,
    "run in bytes": lambda: np.concatenate([gen.text("bytes", 11, 4000), np.full(3500, 7, np.uint8),
                                            gen.text("bytes", 12, 4000), np.full(900, 7, np.uint8)]),
    "short runs": lambda: np.concatenate([np.r_[np.full(40, 5, np.uint8), gen.text("bytes", 20 + k, 30)]
                                          for k in range(200)]),
}


@pytest.mark.parametrize("name", list(TEXTS))
def test_edges(gb, orc, name):
    import torch
    t = np.ascontiguousarray(TEXTS[name]())
    want_sa, want_isa, _, _ = orc.pd_sa(t)
    d = torch.from_numpy(t).cuda()
    sa, isa, _, _ = gb.sa_build_ex(d, isa=True)
    assert np.array_equal(u32(sa), want_sa)
    assert np.array_equal(u32(isa), want_isa)
    assert np.array_equal(u32(gb.sa_build(d)), want_sa)


def test_batch(gb, orc):
    import torch
    texts = [np.ascontiguousarray(f()) for f in TEXTS.values()] + [np.empty(0, np.uint8)] * 3
    off = np.concatenate([[0], np.cumsum([x.size for x in texts])]).astype(np.uint64)
    got = u32(gb.sa_build_batched(torch.from_numpy(np.concatenate(texts)).cuda(), off))
    for k, x in enumerate(texts):
        if x.size:
            assert np.array_equal(got[int(off[k]):int(off[k + 1])], orc.pd_sa(x)[0]), k


@pytest.mark.parametrize("h0,copy", [(0, 400000), (12, 3000)])
def test_needed_entries(gb, orc, h0, copy):
    import torch
    n = (1 << 22) + 77
    t = gen.text("dna", 13, n)
    t[n - copy:] = t[1000:1000 + copy]
    sa, _, st, _ = gb.sa_build_ex(torch.from_numpy(t).cuda(), h0_chars=h0)
    assert st["rounds"] > 5
    assert orc.check_sa(t, u32(sa)) == (0, -1)


@pytest.mark.parametrize("count,size", [(3, 3000), (4, 90001), (20, 200003)])
def test_batch_of_unlike_texts(gb, orc, count, size):
    """Texts of four letters beside texts of many: more top digits are sorted
    than the counts of the whole batch ask for."""
    import torch
    texts = [gen.text("zipf" if k % 2 else "dna", 40 + k, size - 7 * k) for k in range(count)]
    off = np.concatenate([[0], np.cumsum([x.size for x in texts])]).astype(np.uint64)
    got = u32(gb.sa_build_batched(torch.from_numpy(np.concatenate(texts)).cuda(), off))
    for k, x in enumerate(texts):
        assert np.array_equal(got[int(off[k]):int(off[k + 1])], orc.pd_sa(x)[0]), k
