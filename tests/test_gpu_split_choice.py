"""How many top digits round 0 sorts before its tiles (Build::choose_split): what
repeats make of the buckets is measured on a sample of the text's prefixes
(KeySample), which the character counts do not show. The SA is exact either way
(the oracle's checker); the radix passes of round 0 tell the choice."""
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


def copies(n, count, seed):
    """`count` copies of a block of Zipf bytes, 0.1% of them replaced."""
    rng = np.random.default_rng(seed)
    t = np.tile(gen.text("zipf", seed, -(-n // count)), count)[:n]
    at = rng.integers(0, n, n // 1000)
    t[at] = t[rng.integers(0, n, at.size)]
    return t


N = (1 << 24) + 77  # the shortest texts that are sampled, and a few more


@pytest.mark.parametrize("make,split", [(lambda: gen.text("zipf", 3, N), True), (lambda: gen.text("bytes", 4, N), True),
                                        (lambda: copies(N, 100, 5), True), (lambda: copies(N, 4000, 6), False),
                                        (lambda: copies(N, 20000, 7), False)],
                         ids=["zipf", "bytes", "100 copies", "4000 copies", "20000 copies"])
def test_copies_are_not_split_in_vain(gb, orc, make, split):
    """Groups of equal keys too large for any tile: all eight digits at once
    instead of the top ones, then the rest of nearly every key again (which
    makes more passes than eight, or fewer where hardly any key is left)."""
    import torch
    t = make()
    sa, _, st, _ = gb.sa_build_ex(torch.from_numpy(t).cuda())
    assert orc.check_sa(t, u32(sa)) == (0, -1)
    assert (st["passes"][0] == 8) == (not split), st["passes"]


@pytest.mark.parametrize("symbols,offset", [(4, 0), (5, 1), (9, 5), (255, 0), (255, 7)])
def test_sampled_alphabets_and_alignments(gb, orc, symbols, offset):
    import torch
    t = np.random.default_rng(symbols).integers(0, symbols, N).astype(np.uint8)
    d = torch.empty(N + 16, dtype=torch.uint8, device="cuda")[offset:offset + N]
    d.copy_(torch.from_numpy(t))
    assert orc.check_sa(t, u32(gb.sa_build(d))) == (0, -1)
