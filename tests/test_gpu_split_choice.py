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


N = (1 << 22) + 77  # the shortest texts that are sampled, and a few more


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


def test_batches_are_measured(gb, orc):
    """Texts of four letters beside texts of many need more digits than either
    the batch's counts or a batch of like texts."""
    import torch
    size, count, passes = 60001, 24, {}
    for kinds in (("zipf", "zipf"), ("protein", "protein"), ("zipf", "dna")):
        rng = np.random.default_rng(9)
        texts = [rng.integers(0, 20, size - 11 * k).astype(np.uint8) if kinds[k % 2] == "protein" else
                 gen.text(kinds[k % 2], 70 + k, size - 11 * k) for k in range(count)]
        off = np.concatenate([[0], np.cumsum([x.size for x in texts])]).astype(np.uint64)
        sa, st = gb.sa_build_batched(torch.from_numpy(np.concatenate(texts)).cuda(), off, stats=True)
        got = u32(sa)
        for k, x in enumerate(texts):
            assert np.array_equal(got[int(off[k]):int(off[k + 1])], orc.pd_sa(x)[0]), k
        passes[kinds[1]] = st["passes"][0]
    assert passes["protein"] < passes["zipf"] < passes["dna"]


@pytest.mark.parametrize("count,size", [(2, 3), (2, 5000), (700, 90), (3571, 40), (3572, 40), (9000, 7)])
def test_sampled_batches(gb, orc, count, size):
    """Batches whose offsets the sample holds in shared memory, and larger ones."""
    import torch
    rng = np.random.default_rng(count)
    texts = [rng.integers(0, 40, int(rng.integers(0, size + 1))).astype(np.uint8) for _ in range(count)]
    texts[0] = np.arange(3, dtype=np.uint8)
    off = np.concatenate([[0], np.cumsum([x.size for x in texts])]).astype(np.uint64)
    got = u32(gb.sa_build_batched(torch.from_numpy(np.concatenate(texts)).cuda(), off))
    for k in range(0, count, 1 + count // 300):
        if texts[k].size:
            assert np.array_equal(got[int(off[k]):int(off[k + 1])], orc.pd_sa(texts[k])[0]), k
