"""The position order of the groups after round 0 (csrc/k_reorder.cu) at the
edges of its tiles: groups of two to tens of thousands of members (spanning
several 2048-item tiles, or a thousand to a tile), texts that end inside and
at the edge of a 224-position line, and batches whose many empty texts need
more lines of marks than characters. Against the oracle; exact."""
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


def text(kind, n):
    if kind == "pairs":  # two copies of one random text: groups of two
        t = gen.text("bytes", 3, n // 2 + 1)
        return np.concatenate([t, t])[:n].copy()
    if kind == "ab":
        return np.tile(np.frombuffer(b"ab", dtype=np.uint8), n // 2 + 1)[:n].copy()
    if kind == "binary":  # a few huge groups under short keys
        return np.random.default_rng(n).integers(0, 2, n).astype(np.uint8)
    return gen.text(kind, 17, n)


@pytest.mark.parametrize("kind,h0", [("pairs", 0), ("ab", 0), ("binary", 3), ("dna", 2), ("zipf_repeats", 0)])
@pytest.mark.parametrize("n", [2, 223, 224, 225, 2048, 4097, 8192, 60001])
def test_position_order(gb, orc, kind, h0, n):
    import torch
    t = text(kind, n)
    want_sa, want_isa, _, _ = orc.pd_sa(t)
    sa, isa, _, _ = gb.sa_build_ex(torch.from_numpy(t).cuda(), isa=True, group_order=1, h0_chars=h0)
    assert np.array_equal(u32(sa), want_sa)
    assert np.array_equal(u32(isa), want_isa)


def test_more_lines_than_characters(gb, orc):
    import torch
    texts = [np.empty(0, np.uint8)] * 3000 + [np.frombuffer(b"abababab", dtype=np.uint8)] * 3
    flat = np.concatenate(texts)
    off = np.concatenate([[0], np.cumsum([x.size for x in texts])]).astype(np.uint64)
    got = u32(gb.sa_build_batched(torch.from_numpy(flat).cuda(), off, group_order=1, h0_chars=1))
    want = orc.pd_sa(np.frombuffer(b"abababab", dtype=np.uint8).copy())[0]
    assert np.array_equal(got, np.tile(want, 3))
