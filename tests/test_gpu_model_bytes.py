"""The byte model of the classification counts the groups that there are, not
the buffer's capacity (a build with few ties would show a rate far above the
memory's)."""
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


@pytest.mark.parametrize("recipe,n,kw", [("dna", 1 << 20, {}), ("markov", 1 << 20, {}), ("zipf", 300001, {"h0_chars": 2}),
                                         ("zipf_repeats", 1 << 20, {"group_order": 1}),
                                         ("markov", 1 << 20, {"refine_shape": 3, "h0_chars": 8})])
def test_classification(gb, recipe, n, kw):
    import torch
    st = gb.sa_build_ex(torch.from_numpy(gen.text(recipe, 11, n)).cuda(), profile=True, **kw)[2]
    got = st["kernels"]["classify"]["bytes"] if "classify" in st["kernels"] else 0
    # At most 36 bytes per group and 4 per tile of at least 256 items, once a
    # round and twice more after round 0.
    groups, items = sum(st["groups"]) + 2 * st["groups"][0], sum(st["active"][1:]) + 2 * n
    assert got <= 36 * groups + 4 * (items // 256 + st["rounds"] + 3)
    assert got >= 4 * sum(st["groups"])


def test_batch_of_few_ties(gb):
    import torch
    texts = [gen.text("dna", k, 20000 + k) for k in range(40)]
    off = np.concatenate([[0], np.cumsum([x.size for x in texts])]).astype(np.uint64)
    _, st = gb.sa_build_batched(torch.from_numpy(np.concatenate(texts)).cuda(), off, stats=True, profile=True)
    if "classify" in st["kernels"]:
        assert st["kernels"]["classify"]["bytes"] <= 36 * 3 * sum(st["groups"]) + 4 * (int(off[-1]) // 64 + 8)
