"""The level pass by first occurrences (blocks of 27 bytes or more) against the oracle.

Sizes at its edges: block lengths around the shortest that always holds a
selected gram, short last blocks of every kind (no gram, a gram or none, always
one), text lengths around the list's words and segments, unaligned texts, texts
that settle nothing early (periodic, runs, one byte), and a modulus that makes
fingerprint matches of open keys false.
"""
import random

import numpy as np
import pytest
import torch

import oracle
from paper_2512_23314_gb300 import bt, workloads

pytestmark = pytest.mark.gpu


def check(text, tau, leaf, shift=0, **kw):
    pad = np.concatenate([np.zeros(shift, np.uint8), text])
    t = bt.Tree(torch.from_numpy(pad).cuda()[shift:], 256, tau, leaf, bt.BuildOptions(**kw))
    assert t.export() == oracle.build(text, tau, leaf, prune=kw.get("prune", True)).export(), (len(text), tau, leaf, kw)
    return t


def texts(n, seed):
    rng = np.random.default_rng(seed)
    yield workloads.text_versions(n=n, base_len=max(256, n // 12), sigma=40, edit_rate=5e-3, seed=seed)
    yield workloads.dna_genome(n=n, genome_len=max(300, n // 9), snp_rate=1e-2, indel_rate=2e-3, seed=seed)
    unit = rng.integers(97, 100, 1 + seed % 61, dtype=np.uint8)
    yield np.resize(unit, n)
    runs = np.repeat(rng.integers(97, 99, n, dtype=np.uint8), rng.integers(1, 90, n))[:n]
    yield np.ascontiguousarray(runs)


@pytest.mark.parametrize("leaf", [26, 27, 28, 31, 32, 33, 48, 64])
@pytest.mark.parametrize("tau", [2, 3, 5])
def test_block_lengths_and_tails(leaf, tau):
    for i, r in enumerate((0, 1, 3, 4, 15, 16, 20, 26, 27, leaf - 1)):
        n = 40 * leaf + r % leaf
        for text in texts(n, 100 * leaf + 10 * tau + i):
            check(text, tau, leaf, prune=bool(i & 1))


@pytest.mark.parametrize("n", [1, 15, 16, 17, 31, 47, 48, 1023, 1024, 1025, 1038, 1039, 1040, 2048 + 16, 8192 * 3 + 15,
                               65536 + 16, 65536 * 2 + 1])
def test_list_edges(n):
    for i, text in enumerate(texts(n, n)):
        check(text, 4, 32, shift=(0, 1, 16, 7)[i])


def test_false_matches_of_open_keys():
    total = 0
    for i in range(12):
        for text in texts(3000 + 517 * i, 7 * i + 1):
            t = check(text, 2 + i % 3, 27 + i, modulus=331, seed=i, prune=bool(i % 2))
            total += sum(s["collisions"] for s in t.stats())
    assert total > 0


def test_shared_cells_and_repeats():
    """Texts whose grams come again in other surroundings: strings cut and pasted at every shift."""
    rng = random.Random(3)
    base = workloads.random_bytes(2000, 4, 5).tobytes()
    for leaf in (27, 32, 64):
        out = bytearray()
        while len(out) < 60_000:
            a = rng.randrange(len(base) - 40)
            out += base[a:a + rng.randrange(20, 400)]
        text = np.frombuffer(bytes(out), np.uint8).copy()
        check(text, 2, leaf)
        check(text, 4, leaf, prune=False, two_phase=True)


@pytest.mark.parametrize("n", [28 << 20, (33 << 20) + 77])
def test_lists_in_two_parts(n):
    """More than 2^22 list entries: distances of repeats, of grams that are new after the leading part, of both; the
    tree is that of the scan of every window."""
    half = workloads.random_bytes(n // 2, 256, 1)
    for text in (workloads.random_bytes(n, 256, n % 97), np.concatenate([half, half[::-1], half])[:n],
                 workloads.dna_genome(n=n, genome_len=n // 3, snp_rate=1e-2, indel_rate=1e-3, seed=2)):
        d = torch.from_numpy(np.ascontiguousarray(text)).cuda()
        blob = bt.Tree(d, 256, 4, 64).export()
        assert blob == bt.Tree(d, 256, 4, 64, bt.BuildOptions(dense_scan=True)).export()
