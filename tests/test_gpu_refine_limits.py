"""Which groups the refine takes in its tiles (csrc/launch.h, REFINE_SHAPE): where
many suffixes are in groups above the shape's own limit, groups of up to half
a tile, so that no round after round 0 sorts them globally. Exact SA and
ISA against the oracle."""
import numpy as np
import pytest

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


def copies(count, seed, size=61, rate=0.002):
    """A block of distinct characters: no group has more than `count` members."""
    rng = np.random.default_rng(seed)
    t = np.tile(rng.permutation(size).astype(np.uint8) + 1, count)
    m = rng.random(t.size) < rate
    t[m] = rng.integers(100, 255, int(m.sum()))
    return t


@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("shape,count,in_tiles", [(1, 385, True), (1, 512, True), (1, 513, False),
                                                  (2, 513, True), (2, 1024, True), (2, 1025, False), (2, 2049, False),
                                                  (3, 2048, True), (3, 2049, False), (4, 512, True), (4, 513, False)])
def test_limits(gb, orc, shape, count, in_tiles, order):
    import torch
    t = copies(count, 7 * count + shape, rate=0.002 if in_tiles else 0)
    want_sa, want_isa, _, _ = orc.pd_sa(t)
    d = torch.from_numpy(t).cuda()
    for kw in ({}, {"multiplier": 3}, {"device_rounds": 1}):
        sa, isa, st, _ = gb.sa_build_ex(d, isa=True, refine_shape=shape, group_order=order, **kw)
        assert np.array_equal(u32(sa), want_sa), kw
        assert np.array_equal(u32(isa), want_isa), kw
        assert st["rounds"] > 1
        if in_tiles or kw == {}:
            assert (max(st["passes"][1:]) == 0) == in_tiles, (kw, st["passes"])


@pytest.mark.parametrize("size,in_tiles", [(2, False), (40, True)])
def test_share_beside_smaller_groups(gb, orc, size, in_tiles):
    """Groups of 800 beside groups of 300: sorted globally where they are few,
    in tiles where they are many."""
    import torch
    t = np.concatenate([copies(800, 3, size=size, rate=0), copies(300, 4, size=140, rate=0) + 60])
    want_sa, want_isa, _, _ = orc.pd_sa(t)
    sa, isa, st, _ = gb.sa_build_ex(torch.from_numpy(t).cuda(), isa=True, refine_shape=2)
    assert np.array_equal(u32(sa), want_sa)
    assert np.array_equal(u32(isa), want_isa)
    assert st["rounds"] > 1
    assert (max(st["passes"][1:]) == 0) == in_tiles


def test_batch(gb, orc):
    import torch
    texts = [copies(500 + 90 * k, 60 + k, size=20 + k) for k in range(6)] + [np.empty(0, np.uint8)]
    off = np.concatenate([[0], np.cumsum([x.size for x in texts])]).astype(np.uint64)
    got = u32(gb.sa_build_batched(torch.from_numpy(np.concatenate(texts)).cuda(), off, refine_shape=2))
    for k, x in enumerate(texts):
        if x.size:
            assert np.array_equal(got[int(off[k]):int(off[k + 1])], orc.pd_sa(x)[0]), k
