"""Texts made of few grams: the search of a level's open keys goes by their first
grams, or by every window, where too many keys share their newest gram.  The trees are
the oracle's (or those of the scan of every window throughout), on the grid, in one
CTA and in clusters, and the windows the search tests stay below the positions."""
import numpy as np
import pytest
import torch

import oracle
from paper_2512_23314_gb300 import bt, workloads

pytestmark = pytest.mark.gpu


def words(n, count, mean, seed):
    """`count` words of about `mean` bytes in random order."""
    r = np.random.default_rng(seed)
    ws = [r.integers(33, 127, int(r.integers(mean // 2, mean * 3 // 2 + 1)), dtype=np.uint8) for _ in range(count)]
    width = max(map(len, ws))
    table, lens = np.zeros((count, width), np.uint8), np.array([len(w) for w in ws])
    for i, w in enumerate(ws):
        table[i, :len(w)] = w
    ids = r.integers(0, count, int(n / lens.mean() * 1.1) + 50)
    text = table[ids][np.arange(width)[None] < lens[ids][:, None]]
    return np.ascontiguousarray(text[:n])


def kinds(n, seed):
    yield words(n, 2, 40, seed)
    yield words(n, 10, 40, seed)
    yield words(n, 4, 300, seed)
    yield workloads.random_bytes(n, 2, seed)
    half = workloads.text_versions(n=n // 2, base_len=n // 20, sigma=90, edit_rate=1e-3, seed=seed)
    yield np.concatenate([half, words(n - len(half), 3, 50, seed)])   # ordinary in its first sixteenth
    yield np.concatenate([words(n - len(half), 3, 50, seed), half])   # and the other way round


@pytest.mark.parametrize("n", [30_000, 200_003, (1 << 20) + 21])
@pytest.mark.parametrize("tau,leaf", [(2, 27), (4, 32)])
def test_against_the_oracle(n, tau, leaf):
    for i, text in enumerate(kinds(n, n % 100 + leaf)):
        d = torch.from_numpy(text).cuda()
        ref = oracle.build(text, tau, leaf, prune=bool(i & 1)).export()
        assert bt.Tree(d, 256, tau, leaf, bt.BuildOptions(prune=bool(i & 1))).export() == ref, i


@pytest.mark.parametrize("n", [(9 << 20) + 77, 12 << 20])
def test_lists_in_two_parts(n):
    """Around the length from which a sample of the list decides (2^21 entries)."""
    for i, text in enumerate(kinds(n, n % 1000)):
        d = torch.from_numpy(text).cuda()
        t = bt.Tree(d, 256, 4, 32)
        assert t.export() == bt.Tree(d, 256, 4, 32, bt.BuildOptions(dense_scan=True)).export(), i


@pytest.mark.parametrize("docs", [3, 20])
@pytest.mark.parametrize("modulus", [0, 65521])
def test_batches(docs, modulus):
    """Clusters (few long documents) and one CTA each (batch_ctas); lists of one part and of two."""
    if modulus and docs > 3:
        pytest.skip("the exact search of many documents takes minutes")
    sizes = (700_001, 150_000) if not modulus else (40_000, 20_001)
    texts = [t for s in range((docs + 5) // 6) for t in kinds(sizes[s & 1] + s, s)][:docs]
    for ctas in (0, 40):
        opts = bt.BuildOptions(modulus=modulus, batch_ctas=ctas).to_c()
        hs = bt.bt_build_batch(texts, [len(t) for t in texts], [256] * docs, [2] * docs, [32] * docs, opts=opts[0])
        try:
            for i, (h, t) in enumerate(zip(hs, texts)):
                one = bt.Tree(torch.from_numpy(t).cuda(), 256, 2, 32, bt.BuildOptions(batch_workers=True))
                assert bt.bt_export(h) == one.export(), (i, ctas)
        finally:
            for h in hs:
                bt.bt_free(h)


@pytest.mark.parametrize("n", [(2 << 20) + 5, (8 << 20) + 3, 40 << 20])
def test_bounds_of_the_search(n):
    """Around the least bound (2^21 steps) and above it, with lists of one part and (40 MiB) of two."""
    for i, text in enumerate(kinds(n, n % 999)):
        d = torch.from_numpy(text).cuda()
        dense = bt.Tree(d, 256, 4, 32, bt.BuildOptions(dense_scan=True)).export()
        assert bt.Tree(d, 256, 4, 32).export() == dense, i


def test_windows_of_short_texts():
    """A short text's search is not given up: its steps are cheaper than a second way (two-letter runs of 256 KiB
    were given up and took twice as long).  Levels given up go by every window and test few (7 in all), this
    search tests over a million on 7 levels."""
    n = 256 << 10
    r = np.random.default_rng(7)
    text = np.repeat(r.integers(97, 99, n // 20, dtype=np.uint8), r.integers(1, 90, n // 20))[:n].copy()
    t = bt.Tree(torch.from_numpy(text).cuda(), 256, 4, 32)
    assert sum(s["candidates"] for s in t.stats()) > n


def test_windows_per_position():
    """A level of K keys that go by few newest grams proposes up to K windows at every occurrence of one: 4.6 per text
    position on random bits.  A search is given up at n / 16 steps of work, and 32 windows take 7, so that sample,
    comparison and rest test at most (1/64 + 1/256 + 1/16) 32/7 n windows, and what 4864 warps do between two reports
    (256 steps, three times): 0.64 n for 64 MiB."""
    n = 64 << 20
    for text in (workloads.random_bytes(n, 2, 1), words(n, 10, 40, 2)):
        t = bt.Tree(torch.from_numpy(text).cuda(), 256, 4, 32)
        worst = max(s["candidates"] for s in t.stats())
        assert worst < 0.7 * n, worst / n


def test_without_room_for_the_scan_of_every_window():
    """The scan takes 8 bytes per position: without them the search goes on."""
    n = 8 << 20
    d = torch.from_numpy(workloads.random_bytes(n, 2, 9)).cuda()
    ref = bt.Tree(d, 256, 2, 128).export()
    bt.bt_test_alloc_limit(8 * n - 1)
    try:
        assert bt.Tree(d, 256, 2, 128).export() == ref
    finally:
        bt.bt_test_alloc_limit(0)
