"""The workloads whose speed this repository is measured on.

Each case is work that a user has the library do through its public entry
points: suffix arrays of one text (resident on the GPU, or end to end from
host memory), of batches of texts, with the optional inverse, and the BWT and
LCP arrays built from a suffix array. Texts are synthetic, made on the GPU
from a seed; their sizes and alphabets follow the repository's configurations
(uniform DNA, Zipf bytes, a repeated Zipf block with substitutions, order-3
Markov DNA with copied segments, log-uniform batches and requests), with
protein-like and prose-like texts beside them.
"""
import math

import numpy as np
import torch

import paper_1610_03007_gb300 as gbsa

DEV = "cuda"
CHUNK = 1 << 26  # characters generated at a time


def listed():
    return [
        # The smallest requests a server sees: launches and latency only.
        {"name": "dna_12k", "call": "build", "text": "dna", "n": 12345},
        # A typical small serving request, host buffer to host buffer.
        {"name": "request_zipf_100k", "call": "host", "text": "zipf", "n": 100003},
        # A bacterial-size chunk of DNA (configuration 1).
        {"name": "dna_1m", "call": "build", "text": "dna", "n": 1 << 20},
        # A collection of prose, 7 bits per character, phrases that recur.
        {"name": "words_8m", "call": "build", "text": "words", "n": 8000003},
        # A protein database, 5 bits per character, with the inverse too.
        {"name": "protein_16m_isa", "call": "build_isa", "text": "protein", "n": 1 << 24},
        # Bytes of a skewed distribution, 8 bits per character.
        {"name": "zipf_32m", "call": "build", "text": "zipf", "n": 33554467},
        # A chromosome-size DNA text, the largest serving request.
        {"name": "dna_64m", "call": "build", "text": "dna", "n": 1 << 26},
        # Versions of one document (configuration 2): many rounds of large groups.
        {"name": "repeats_256m", "call": "build", "text": "repeats", "n": 1 << 28, "base": 1 << 20},
        # A genome with duplicated segments (configuration 3 at half size).
        {"name": "markov_1g", "call": "build", "text": "markov", "n": 1 << 30},
        # Queued small requests built as one batch from host memory.
        {"name": "batch_host_48", "call": "batch_host", "text": "mixed", "count": 48, "lo": 10 << 10, "hi": 256 << 10},
        # Contigs of an assembly (configuration 4 at a quarter of its count).
        {"name": "batch_dna_1024", "call": "batch", "text": "dna", "count": 1024, "lo": 1 << 10, "hi": 4 << 20},
        # The index arrays that follow a suffix array: BWT and LCP.
        {"name": "bwt_lcp_words_48m", "call": "bwt_lcp", "text": "words", "n": 48000001},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["build", "build", "build", "build", "build_isa", "host", "repeats", "markov",
                       "batch", "batch_host", "bwt_lcp"])
    kind = rng.choice(["dna", "zipf", "words", "protein", "bytes", "binary"])
    if call == "repeats":
        base = _log_uniform(rng, 1 << 14, 1 << 20)
        return {"call": "build", "text": "repeats", "n": base * rng.randint(16, 256) + rng.randint(0, 99), "base": base}
    if call == "markov":
        return {"call": "build", "text": "markov", "n": _log_uniform(rng, 1 << 20, 1 << 29)}
    if call == "batch":
        return {"call": "batch", "text": rng.choice(["dna", "zipf", "protein"]), "count": rng.randint(16, 512),
                "lo": 1 << 10, "hi": _log_uniform(rng, 64 << 10, 4 << 20)}
    if call == "batch_host":
        return {"call": "batch_host", "text": "mixed", "count": rng.randint(2, 48), "lo": 10 << 10, "hi": 256 << 10}
    if call == "host":
        return {"call": "host", "text": kind, "n": _log_uniform(rng, 10 << 10, 16 << 20)}
    if call == "bwt_lcp":
        return {"call": "bwt_lcp", "text": kind, "n": _log_uniform(rng, 10 << 10, 1 << 26)}
    return {"call": call, "text": kind, "n": _log_uniform(rng, 10 << 10, 1 << 27)}


# ---- texts -------------------------------------------------------------------


def _from_weights(weights, symbols, n, g):
    """n i.i.d. symbols with the given weights."""
    w = torch.as_tensor(weights, dtype=torch.float64)
    cdf = (w.cumsum(0) / w.sum()).to(torch.float32).to(DEV)
    sym = torch.as_tensor(list(symbols), dtype=torch.uint8, device=DEV)
    out = torch.empty(n, dtype=torch.uint8, device=DEV)
    for a in range(0, n, CHUNK):
        b = min(n, a + CHUNK)
        k = torch.searchsorted(cdf, torch.rand(b - a, device=DEV, generator=g), right=True, out_int32=True)
        out[a:b] = sym[k.clamp_(max=len(w) - 1)]
    return out


def _zipf(n, g, top=255, s=1.1):
    return _from_weights([r ** -s for r in range(1, top + 1)], range(1, top + 1), n, g)


def _dna(n, g):
    return _from_weights([1.0] * 4, b"ACGT", n, g)


def _protein(n, g):
    # Amino-acid letters with roughly their frequencies in protein databases.
    freq = {"A": 8.3, "C": 1.4, "D": 5.5, "E": 6.7, "F": 3.9, "G": 7.1, "H": 2.3, "I": 5.9, "K": 5.8, "L": 9.7,
            "M": 2.4, "N": 4.1, "P": 4.7, "Q": 3.9, "R": 5.5, "S": 6.6, "T": 5.3, "V": 6.9, "W": 1.1, "Y": 2.9}
    return _from_weights(list(freq.values()), "".join(freq).encode(), n, g)


def _words(n, g):
    """Words of a 30000-word vocabulary with Zipf frequencies, one space or
    punctuation mark after each: prose-like, about 75 distinct bytes."""
    vocab, longest = 30000, 12
    letters = b"etaoinshrdlcumwfgypbvkjxqz" + b"ETAOINSHRDLCUMWFGYPBVKJXQZ" + b"0123456789"
    weights = [1.0 / (r + 2) for r in range(26)] + [0.02 / (r + 2) for r in range(26)] + [0.003] * 10
    table = _from_weights(weights, letters, vocab * longest, g).view(vocab, longest)
    length = torch.randint(1, longest, (vocab,), device=DEV, generator=g)
    cdf = torch.arange(1, vocab + 1, device=DEV, dtype=torch.float64).pow(-1.0).cumsum(0)
    cdf = (cdf / cdf[-1]).to(torch.float32)
    seps = torch.tensor(list(b"          ,,.;:?!-\n\n"), dtype=torch.uint8, device=DEV)
    out = torch.empty(n, dtype=torch.uint8, device=DEV)
    at = 0
    while at < n:
        count = min(n - at, CHUNK // 4) // 2 + 1
        w = torch.searchsorted(cdf, torch.rand(count, device=DEV, generator=g)).clamp_(max=vocab - 1)
        sep = seps[torch.randint(0, len(seps), (count,), device=DEV, generator=g)]
        size = length[w] + 1
        end = size.cumsum(0)
        which = torch.repeat_interleave(torch.arange(count, device=DEV), size)
        off = torch.arange(which.numel(), device=DEV) - (end - size)[which]
        part = torch.where(off == length[w][which], sep[which], table[w[which], off.clamp_(max=longest - 1)])
        take = min(n - at, part.numel())
        out[at:at + take] = part[:take]
        at += take
    return out


def _repeats(n, base, g):
    """A Zipf block repeated to n characters, every copy with 0.1% of its
    characters replaced by others."""
    block = _zipf(base, g)
    out = block.repeat(-(-n // base))[:n].clone()
    for a in range(0, n, CHUNK):
        part = out[a:a + CHUNK]
        at = (torch.rand(part.numel(), device=DEV, generator=g) < 0.001).nonzero().view(-1)
        step = torch.randint(1, 255, (at.numel(),), device=DEV, generator=g)
        part[at] = ((part[at].long() - 1 + step) % 255 + 1).to(torch.uint8)
    return out


def _markov(n, g):
    """Order-3 Markov DNA (64 random rows), then segments of 1 to 100 KiB
    copied to random places until they cover 5% of the text."""
    chains = max(1, min(1 << 18, n >> 10))
    steps = -(-n // chains)
    row = -torch.rand(64, 4, device=DEV, generator=g).clamp_(min=1e-7).log()
    cum = (row / row.sum(1, keepdim=True)).cumsum(1)[:, :3].contiguous()
    state = torch.randint(0, 64, (chains,), device=DEV, generator=g)
    codes = torch.empty(steps, chains, dtype=torch.uint8, device=DEV)
    for t in range(steps):
        u = torch.rand(chains, 1, device=DEV, generator=g)
        c = (u > cum[state]).sum(1)
        codes[t] = c
        state = (state * 4 + c) & 63
    text = torch.tensor(list(b"ACGT"), dtype=torch.uint8, device=DEV)[codes.t().reshape(-1)[:n].int()]
    del codes
    source, covered = text.clone(), 0
    r = torch.randint(0, 1 << 62, (3, n // 20480 + 64), device=DEV, generator=g).cpu().numpy()
    for k in range(r.shape[1]):
        size = min(1024 + int(r[0, k] % (99 * 1024 + 1)), n // 4)
        src, dst = int(r[1, k] % (n - size + 1)), int(r[2, k] % (n - size + 1))
        text[dst:dst + size] = source[src:src + size]
        covered += size
        if covered >= n // 20:
            break
    return text


def _text(case, kind, n, g):
    if kind == "dna":
        return _dna(n, g)
    if kind == "zipf":
        return _zipf(n, g)
    if kind == "protein":
        return _protein(n, g)
    if kind == "words":
        return _words(n, g)
    if kind == "bytes":
        return torch.randint(0, 256, (n,), dtype=torch.uint8, device=DEV, generator=g)
    if kind == "binary":
        return torch.randint(0, 2, (n,), dtype=torch.uint8, device=DEV, generator=g)
    if kind == "repeats":
        return _repeats(n, case["base"], g)
    if kind == "markov":
        return _markov(n, g)
    raise ValueError(kind)


def _lengths(case):
    """Log-uniform lengths of a batch: the quantiles of the distribution in a
    shuffled order, the same for every seed."""
    count = case["count"]
    q = (np.arange(count) + 0.5) / count
    v = np.exp(np.log(case["lo"]) + q * (np.log(case["hi"]) - np.log(case["lo"])))
    return np.random.RandomState(case["count"]).permutation(v.astype(np.int64))


def _inputs(case, seed):
    """The texts of a case: one tensor, or (flat tensor, offsets)."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    if "count" not in case:
        return _text(case, case["text"], case["n"], g), None
    lengths = _lengths(case)
    offsets = np.zeros(case["count"] + 1, dtype=np.uint64)
    np.cumsum(lengths, out=offsets[1:])
    if case["text"] == "mixed":  # half the requests are DNA, half Zipf bytes
        parts = [(_dna if k % 2 else _zipf)(int(n), g) for k, n in enumerate(lengths)]
        return torch.cat(parts), offsets
    return _text(case, case["text"], int(offsets[-1]), g), offsets


def _pinned(x):
    return torch.empty(x.shape, dtype=x.dtype, pin_memory=True).copy_(x)


# ---- prepare, run, work --------------------------------------------------------


def prepare(case, seed):
    text, offsets = _inputs(case, seed)
    call = case["call"]
    state = {"call": call, "text": text, "offsets": offsets}
    if call == "host":  # a server's pinned request and result buffers
        state["text"] = _pinned(text.cpu()).numpy()
        state["out"] = torch.empty(case["n"], dtype=torch.int32, pin_memory=True).numpy().view(np.uint32)
    elif call == "batch_host":
        flat = _pinned(text.cpu()).numpy()
        out = torch.empty(flat.size, dtype=torch.int32, pin_memory=True).numpy().view(np.uint32)
        at = [int(o) for o in offsets]
        state["text"] = [flat[a:b] for a, b in zip(at, at[1:])]
        state["out"] = [out[a:b] for a, b in zip(at, at[1:])]
    elif call == "bwt_lcp":
        state["sa"] = gbsa.sa_build(text)
    return state


def run(state):
    call, text = state["call"], state["text"]
    if call == "build":
        return gbsa.sa_build(text)
    if call == "build_isa":
        sa, isa, _, _ = gbsa.sa_build_ex(text, isa=True)
        return {"sa": sa, "isa": isa}
    if call == "host":
        return gbsa.sa_build_host(text, sa_out=state["out"])
    if call == "batch":
        return gbsa.sa_build_batched(text, state["offsets"])
    if call == "batch_host":
        return gbsa.sa_build_batched_host(text, outs=state["out"])
    if call == "bwt_lcp":
        bwt, primary = gbsa.sa_bwt(text, state["sa"])
        return {"bwt": bwt, "primary": primary, "lcp": gbsa.sa_lcp(text, state["sa"])}
    raise ValueError(call)


def work(case):
    """Every input character read once and every output written once."""
    n = case["n"] if "n" in case else int(_lengths(case).sum())
    per = {"build": 5, "host": 5, "batch": 5, "batch_host": 5, "build_isa": 9, "bwt_lcp": 10}[case["call"]]
    return {"bytes": per * n, "flops": 0}


# ---- the same results in plain torch -------------------------------------------

EXACT_MAX = 1 << 28  # larger texts would take too long


def _naming(key):
    """(order, rank by position, number of distinct keys)."""
    key, order = torch.sort(key)
    rank = torch.zeros_like(key)
    rank[1:] = (key[1:] != key[:-1]).long().cumsum(0)
    distinct = int(rank[-1]) + 1
    out = torch.empty_like(rank)
    out[order] = rank
    return order, out, distinct


def _suffix_array(text, levels=None):
    """Prefix doubling on 64-bit keys from single characters on; `levels`
    collects (h, ranks of the h-character prefixes)."""
    n = text.numel()
    h = 1
    order, rank, distinct = _naming(text.long())
    while True:
        if levels is not None:
            levels.append((h, rank.int()))
        if distinct == n:
            return order.int()
        key = rank * (n + 1)
        if h < n:
            key[:n - h] += rank[h:] + 1
        order, rank, distinct = _naming(key)
        h *= 2


def _lcp(sa, levels):
    """Longest common prefix of neighbours in sa, from the largest h down."""
    n = sa.numel()
    a, b = sa[:-1].long(), sa[1:].long()
    got = torch.zeros(n - 1, dtype=torch.long, device=sa.device)
    for h, rank in reversed(levels):
        x, y = a + got, b + got
        inside = (x + h <= n) & (y + h <= n)
        same = inside & (rank[x.clamp(max=n - 1)] == rank[y.clamp(max=n - 1)])
        got += h * same.long()
    return torch.cat([got.new_zeros(1), got]).int()


def exact(case, seed):
    text, offsets = _inputs(case, seed)
    if text.numel() > EXACT_MAX and offsets is None:
        return None
    if offsets is not None:
        at = [int(o) for o in offsets]
        parts = [_suffix_array(text[a:b]) for a, b in zip(at, at[1:])]
        return [p.cpu().numpy() for p in parts] if case["call"] == "batch_host" else torch.cat(parts)
    call = case["call"]
    if call != "bwt_lcp":
        sa = _suffix_array(text)
        if call == "host":
            return sa.cpu().numpy()
        if call == "build_isa":
            isa = torch.empty_like(sa)
            isa[sa.long()] = torch.arange(text.numel(), dtype=torch.int32, device=DEV)
            return {"sa": sa, "isa": isa}
        return sa
    levels = []
    sa = _suffix_array(text, levels)
    first = int((sa == 0).nonzero()[0])
    rows = torch.cat([text[-1:], text[(sa.long() - 1).clamp(min=0)]])
    rows[first + 1] = 0
    return {"bwt": rows, "primary": first + 1, "lcp": _lcp(sa, levels)}
