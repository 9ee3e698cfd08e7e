"""Performance cases of the block-tree library: what a program that uses it has it do.

Four kinds of work go through the public binding (``paper_2512_23314_gb300.bt``):

* ``build``   one text to its tree and the tree to its canonical serialization
              in a caller's pinned buffer (an indexing job: build, store, free);
* ``batch``   many documents built in one call, then rank queries on every tree
              (a collection being indexed and served);
* ``query``   device-resident batches of access, rank and select queries on a
              tree that is already there;
* ``points``  single access, rank and select calls from the host;
* ``prefix``  the Karp-Rabin prefix fingerprints of a text.

Texts have the shapes of the repetitive collections the library is for: versions
of a Zipf text with edit runs, copies of a genome with substitutions, indels and
N runs.  They are generated on the GPU from the seed.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2512_23314_gb300 import bt

ACGT = (65, 67, 71, 84)
MIB = 1 << 20


def listed():
    return [
        # A program that asks for one character, one count, one position at a time.
        dict(name="points_dna_1MiB", kind="points", text="dna_sub", n=MIB, copies=16, tau=2, leaf=16, m=4),
        # One web request's worth of queries on a document's tree: launch and latency.
        dict(name="query_1k_text_16MiB", kind="query", text="text", n=16 * MIB, copies=16, tau=4, leaf=32,
             leaf_counts=False, m=1000),
        # Bulk queries on the 256 MiB versioned text's tree, every kind.
        dict(name="query_4M_text_256MiB", kind="query", text="text", n=256 * MIB, copies=64, tau=4, leaf=32,
             leaf_counts=False, m=1 << 22),
        # The space-efficient counters on a genome collection, at an odd count of queries.
        dict(name="query_space_dna_64MiB", kind="query", text="dna", n=64 * MIB, copies=32, tau=4, leaf=64,
             leaf_counts=True, m=1_000_003),
        # Fingerprints alone, for a program with its own matching; a ragged end.
        dict(name="prefix_256MiB_77", kind="prefix", text="text", n=256 * MIB + 77, copies=64),
        # The smallest index: one short document from host memory.
        dict(name="build_text_4KiB", kind="build", text="text", n=4096, copies=4, tau=4, leaf=32, host=True,
             prune=True, two_phase=False),
        # A small DNA collection: deep binary tree with short leaves.
        dict(name="build_dna_1MiB", kind="build", text="dna_sub", n=MIB, copies=16, tau=2, leaf=16, host=False,
             prune=True, two_phase=False),
        # A document of a service's upload, pinned host memory, odd length, wide nodes.
        dict(name="build_text_20MB_odd", kind="build", text="text", n=20_000_003, copies=16, tau=8, leaf=32,
             host=True, prune=True, two_phase=False),
        # The versioned text of the headline benchmark.
        dict(name="build_text_256MiB", kind="build", text="text", n=256 * MIB, copies=64, tau=4, leaf=32,
             host=False, prune=True, two_phase=False),
        # The genome collection, the longest text, with the option its programs set.
        dict(name="build_dna_2GiB", kind="build", text="dna", n=2048 * MIB, copies=64, tau=4, leaf=64, host=False,
             prune=True, two_phase=True),
        # A micro-batch of the serving loop: a few dozen short documents.
        dict(name="batch_64_docs_1MiB", kind="batch", docs=64, min_len=1 << 10, max_len=MIB, leaf=32, m=2000),
        # A collection of documents of uneven length, built in one call.
        dict(name="batch_1024_docs_4MiB", kind="batch", docs=1024, min_len=4 << 10, max_len=4 * MIB, leaf=32,
             m=2000),
    ]


def _logint(rng, lo, hi):
    return int(min(hi, max(lo, math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    kind = rng.choice(["build", "build", "build", "batch", "query", "query", "points", "prefix"])
    text = rng.choice(["text", "text", "dna", "dna_sub"])
    copies = rng.choice([8, 16, 32, 64])
    tau = rng.choice([2, 3, 4, 4, 8])
    leaf = rng.choice([16, 32, 32, 64, 24, 33])
    if kind == "build":
        return dict(kind=kind, text=text, n=_logint(rng, 1 << 10, 256 * MIB), copies=copies, tau=tau, leaf=leaf,
                    host=rng.random() < 0.5, prune=rng.random() < 0.8,
                    two_phase=text == "dna" and rng.random() < 0.5)
    if kind == "batch":
        lo = rng.choice([1 << 10, 4 << 10])
        return dict(kind=kind, docs=_logint(rng, 8, 1024), min_len=lo, max_len=_logint(rng, 64 << 10, 4 * MIB),
                    leaf=rng.choice([16, 32, 64]), m=2000)
    if kind == "query":
        return dict(kind=kind, text=text, n=_logint(rng, 64 << 10, 256 * MIB), copies=copies, tau=tau, leaf=leaf,
                    leaf_counts=rng.random() < 0.3, m=_logint(rng, 100, 1 << 22))
    if kind == "points":
        return dict(kind=kind, text=text, n=_logint(rng, 4 << 10, 64 * MIB), copies=copies, tau=tau, leaf=leaf,
                    m=rng.randint(1, 8))
    return dict(kind=kind, text=text, n=_logint(rng, 1 << 10, 512 * MIB), copies=copies)


# ---------------------------------------------------------------------------
# Texts.
# ---------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _zipf(g, sigma):
    """One symbol per entry of `sigma` (its alphabet size): rank k with
    probability about 1/k; printable bytes when the alphabet fits."""
    u = torch.rand(sigma.shape, generator=g, device="cuda")
    s = sigma.to(torch.float32)
    k = torch.exp(u * torch.log(s + 1)).floor_().clamp_(min=1).minimum(s) - 1
    return (k + torch.where(sigma <= 96, 32.0, 0.0)).to(torch.uint8)


def _edit(g, t, fresh, rate, max_run, keep_kinds=(0, 1, 2)):
    """`t` with round(rate len) edit runs of U[1, max_run] symbols at uniform
    places: 0 substitute, 1 insert, 2 delete.  `fresh(idx)` draws a symbol
    for each source position in idx.  Returns the new text and, for every old
    position (and the end), the new position it moved to."""
    n = t.numel()
    m = int(round(rate * n))
    pos = torch.randint(0, n, (m,), generator=g, device="cuda")
    kind = torch.tensor(keep_kinds, device="cuda")[torch.randint(0, len(keep_kinds), (m,), generator=g, device="cuda")]
    run = torch.randint(1, max_run + 1, (m,), generator=g, device="cuda")
    end = (pos + run).clamp(max=n)

    def covered(which):
        d = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
        one = (kind == which).to(torch.int32)
        d.index_add_(0, pos, one)
        d.index_add_(0, end, -one)
        return d.cumsum(0)[:n] > 0

    sub, gone = covered(0), covered(2)
    more = torch.zeros(n, dtype=torch.int64, device="cuda")
    more.index_add_(0, pos, run * (kind == 1))
    reps = more + (~gone).to(torch.int64)
    start = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(reps, 0, out=start[1:])
    idx = torch.repeat_interleave(reps)
    new = sub[idx] | (torch.arange(idx.numel(), device="cuda") - start[idx] < more[idx])
    return torch.where(new, fresh(idx), t[idx]), start


def make_text(kind, n, copies, seed):
    """`n` bytes on the GPU: `copies` versions or copies of a base of n / copies."""
    g = _gen(seed)
    base_n = max(256, -(-n // copies))
    out = torch.empty(n, dtype=torch.uint8, device="cuda")
    filled = 0
    if kind == "text":
        v = _zipf(g, torch.full((base_n,), 96, dtype=torch.int32, device="cuda"))
    else:
        acgt = torch.tensor(ACGT, dtype=torch.uint8, device="cuda")
        genome = torch.randint(0, 4, (base_n,), generator=g, device="cuda", dtype=torch.uint8)
    while filled < n:
        if kind == "text":
            c = v
            v, _ = _edit(g, v, lambda i: _zipf(g, torch.full(i.shape, 96, dtype=torch.int32, device="cuda")), 5e-4, 32)
        else:
            hit = torch.rand(base_n, generator=g, device="cuda") < 1e-3
            shift = torch.randint(1, 4, (base_n,), generator=g, device="cuda", dtype=torch.uint8)
            c = acgt[((genome + hit * shift) & 3).to(torch.int32)]
            if kind == "dna":
                c, _ = _edit(g, c, lambda i: acgt[torch.randint(0, 4, i.shape, generator=g, device="cuda")], 1e-4, 50,
                             (1, 2))
                c, _ = _edit(g, c, lambda i: torch.full_like(i, 78, dtype=torch.uint8), 1e-6, 20, (0,))
        take = min(c.numel(), n - filled)
        out[filled:filled + take] = c[:take]
        filled += take
    return out


def _doc_params(case):
    """Lengths, alphabet sizes and arities of a batch's documents: the
    collection's shape is the case's, its content the seed's."""
    r = random.Random(case["docs"] * 1_000_003 + case["max_len"])
    n = [_logint(r, case["min_len"], case["max_len"]) for _ in range(case["docs"])]
    return n, [r.randint(4, 128) for _ in n], [r.choice((2, 4, 8)) for _ in n]


def make_docs(case, seed):
    """The documents in one pinned host buffer, each 16 or more versions of its base."""
    g = _gen(seed)
    lens, sigmas, _ = _doc_params(case)
    base = [max(min(1024, n), n // 16) for n in lens]
    bounds = torch.tensor(np.concatenate([[0], np.cumsum(base)]), device="cuda")
    sig = torch.repeat_interleave(torch.tensor(sigmas, dtype=torch.int32, device="cuda"),
                                  torch.tensor(base, device="cuda"))
    v = _zipf(g, sig)
    at = np.concatenate([[0], np.cumsum(lens)])
    buf = torch.empty(int(at[-1]), dtype=torch.uint8, pin_memory=True)
    out = buf.numpy()
    fill = [0] * len(lens)
    while True:
        host, b = v.cpu().numpy(), bounds.tolist()
        for d, n in enumerate(lens):
            take = min(b[d + 1] - b[d], n - fill[d])
            if take > 0:
                o = int(at[d]) + fill[d]
                out[o:o + take] = host[b[d]:b[d] + take]
                fill[d] += take
        if all(f >= n for f, n in zip(fill, lens)):
            return buf, at
        grown = []

        def fresh(i):
            grown.append(sig[i])
            return _zipf(g, grown[0])

        v, start = _edit(g, v, fresh, 5e-4, 32)
        sig = grown[0]
        bounds = start[bounds]


# ---------------------------------------------------------------------------
# Queries.
# ---------------------------------------------------------------------------
def _query_args(text, m, seed):
    """Positions anywhere, symbols as they occur, occurrences that exist."""
    g = _gen(seed)
    n = text.numel()
    acc = torch.randint(0, n, (m,), generator=g, device="cuda")
    c = text[torch.randint(0, n, (m,), generator=g, device="cuda")].to(torch.int64)
    rank = torch.stack([c, torch.randint(0, n + 1, (m,), generator=g, device="cuda")], 1).contiguous()
    count = sum(torch.bincount(p.to(torch.int32), minlength=256) for p in text.split(1 << 26))
    c = text[torch.randint(0, n, (m,), generator=g, device="cuda")].to(torch.int64)
    j = (torch.rand(m, generator=g, device="cuda", dtype=torch.float64) * count[c]).to(torch.int64).minimum(
        count[c] - 1) + 1
    return acc, rank, torch.stack([c, j], 1).contiguous()


def _answers(text, acc, rank, sel):
    """The same by plain counting."""
    r, s = torch.zeros_like(rank[:, 0]), torch.zeros_like(sel[:, 0])
    for c in torch.unique(torch.cat([rank[:, 0], sel[:, 0]])).tolist():
        where = torch.nonzero(text == c).reshape(-1)
        a, b = rank[:, 0] == c, sel[:, 0] == c
        r[a] = torch.searchsorted(where, rank[a, 1].contiguous())
        s[b] = where[sel[b, 1] - 1]
    return text[acc].to(torch.int64), r, s


# ---------------------------------------------------------------------------
# The five functions.
# ---------------------------------------------------------------------------
def _export_cap(n, leaf):
    """Bytes that hold any tree's serialization (a block of the text costs at
    most 16 bytes or its own text, marks a few bits); the longest texts' many
    copies need less than a quarter."""
    return n * 5 // 16 if n > 256 * MIB else n * max(1, -(-16 // leaf)) + n // 4 + (64 << 10)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        buf, at = make_docs(case, seed)
        lens, sigmas, taus = _doc_params(case)
        r = np.random.default_rng(seed)
        m, host = case["m"], buf.numpy()
        args = np.empty((len(lens), m, 2), np.int64)
        for d, n in enumerate(lens):
            args[d, :, 0] = host[at[d] + r.integers(0, n, m)]
            args[d, :, 1] = r.integers(0, n + 1, m)
        return dict(kind=kind, buf=buf, texts=[buf[at[d]:at[d + 1]] for d in range(len(lens))], n=lens, sigma=sigmas,
                    tau=taus, leaf=[case["leaf"]] * len(lens), args=torch.from_numpy(args).cuda(),
                    out=torch.empty((len(lens), m), dtype=torch.int64, device="cuda"))
    text = make_text(case["text"], case["n"], case["copies"], seed)
    if kind == "prefix":
        return dict(kind=kind, text=text, out=torch.empty(case["n"] // 32 + 1, dtype=torch.int64, device="cuda"))
    sigma = 96 if case["text"] == "text" else 5
    if kind == "build":
        if case["host"]:
            text = text.cpu().pin_memory()
        return dict(kind=kind, text=text, sigma=sigma, tau=case["tau"], leaf=case["leaf"],
                    opts=bt.BuildOptions(prune=case["prune"], two_phase=case["two_phase"]),
                    out=torch.zeros(_export_cap(case["n"], case["leaf"]), dtype=torch.uint8, pin_memory=True))
    tree = bt.Tree(text, sigma, case["tau"], case["leaf"],
                   bt.BuildOptions(leaf_counts=case.get("leaf_counts", False)))
    args = _query_args(text, case["m"], seed + 1)
    if kind == "points":
        return dict(kind=kind, tree=tree, args=[a.tolist() for a in args])
    return dict(kind=kind, tree=tree, args=args,
                out=[torch.empty(case["m"], dtype=torch.int64, device="cuda") for _ in args])


def run(state):
    kind = state["kind"]
    if kind == "build":
        tree = bt.Tree(state["text"], state["sigma"], state["tau"], state["leaf"], state["opts"])
        size = bt.bt_export_into(tree.handle, state["out"])
        tree.close()
        return {"size": size, "blob": state["out"]}
    if kind == "batch":
        trees = bt.bt_build_batch(state["texts"], state["n"], state["sigma"], state["tau"], state["leaf"])
        m = state["out"].shape[1]
        stream = torch.cuda.current_stream()
        for t, a, o in zip(trees, state["args"], state["out"]):
            bt.bt_query_batch(t, bt.BT_Q_RANK, a, m, o, stream)
        stream.synchronize()  # the answers, before the trees go
        for t in trees:
            bt.bt_free(t)
        return state["out"]
    if kind == "query":
        stream = torch.cuda.current_stream()
        for q, a, o in zip((bt.BT_Q_ACCESS, bt.BT_Q_RANK, bt.BT_Q_SELECT), state["args"], state["out"]):
            state["tree"].query_batch(q, a, o, stream)
        return state["out"]
    if kind == "points":
        tree, (acc, rank, sel) = state["tree"], state["args"]
        return [np.array([tree.access(i) for i in acc], np.int64),
                np.array([tree.rank(c, i) for c, i in rank], np.int64),
                np.array([tree.select(c, j) for c, j in sel], np.int64)]
    bt.bt_prefix_fingerprints(state["text"], state["text"].numel(), 0, 0, 32, state["out"],
                              torch.cuda.current_stream())
    return state["out"]


def work(case):
    kind = case["kind"]
    if kind == "batch":  # the texts once, the arguments and answers
        return {"bytes": sum(_doc_params(case)[0]) + case["docs"] * case["m"] * 24, "flops": 0}
    if kind == "prefix":
        return {"bytes": case["n"] + (case["n"] // 32 + 1) * 8, "flops": 0}
    if kind == "build":  # the text once and the serialization, about a quarter of it
        return {"bytes": case["n"] + case["n"] // 4, "flops": 0}
    return {"bytes": case["m"] * (16 + 24 + 24), "flops": 0}  # arguments and answers


def exact(case, seed):
    """Query answers by plain counting; trees and fingerprints have no counterpart outside the library."""
    if case["kind"] in ("query", "points"):
        text = make_text(case["text"], case["n"], case["copies"], seed)
        return list(_answers(text, *_query_args(text, case["m"], seed + 1)))
    return None
