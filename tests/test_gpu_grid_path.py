"""The single-text kernels on short texts.

A text of at most 16 KiB is built by one CTA unless a flag asks for the path of
longer texts; `batch_workers` does.  The sizes at which those kernels can go
wrong are cheapest there: block lengths around the shortest that always holds a
selected gram, short last blocks of every kind, the list's words and segments,
explicit block sizes, and a modulus that makes fingerprint matches false, which
is what the exact search of a level is for.
"""
import random

import numpy as np
import pytest

import oracle
from paper_2512_23314_gb300 import bt, workloads
from tests.test_gpu_first_occurrence import check, texts
from tests.test_gpu_parity import _far_anchor_text, _runs_text
from tests.test_oracle import _random_text

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("leaf", [16, 25, 26, 27, 28, 31, 32, 33, 48, 64])
@pytest.mark.parametrize("tau", [2, 3, 5])
def test_block_lengths_and_tails(leaf, tau):
    for i, r in enumerate((0, 1, 3, 4, 15, 16, 20, 26, 27, leaf - 1)):
        n = 40 * leaf + r % leaf
        for text in texts(n, 100 * leaf + 10 * tau + i):
            check(text, tau, leaf, prune=bool(i & 1), batch_workers=True)


@pytest.mark.parametrize("n", [1, 15, 16, 17, 31, 47, 48, 1023, 1024, 1025, 1038, 1039, 1040, 2048 + 16])
def test_list_edges(n):
    for i, text in enumerate(texts(n, n)):
        check(text, 4, 32, shift=(0, 1, 16, 7)[i], batch_workers=True)


def collisions(t, lo, hi):
    return sum(s["collisions"] for s in t.stats() if lo <= s["b"] < hi)


def test_false_matches():
    """Levels of blocks of 27 bytes or more (the search by first occurrences) and of shorter ones (the anchored scan):
    both meet false matches and resolve them exactly."""
    long_blocks = short_blocks = 0
    for i in range(10):
        for text in texts(3000 + 517 * i, 7 * i + 1):
            for leaf in (27 + i, 7 + i):
                t = check(text, 2 + i % 3, leaf, modulus=331, seed=i, prune=bool(i % 2), batch_workers=True)
                long_blocks += collisions(t, 27, 1 << 40)
                short_blocks += collisions(t, 0, 27)
    assert long_blocks > 0 and short_blocks > 0


@pytest.mark.parametrize("n", [16385, 40_001])
def test_false_matches_beyond_one_launch(n):
    total = 0
    for i, text in enumerate(texts(n, n)):
        total += collisions(check(text, 2 + i, 32, modulus=65521, seed=i), 27, 1 << 40)
        check(text, 3, 9, modulus=65521, seed=i)
    assert total > 0


def test_random_texts_and_explicit_sizes():
    rng = random.Random(11)
    for i in range(120):
        n = rng.randrange(1, 3000)
        text = np.frombuffer(bytes(_random_text(rng, n, rng.choice([1, 2, 3, 26]))), np.uint8)
        check(text, rng.choice([2, 3, 4]), rng.choice([1, 3, 8, 40, 100]), batch_workers=True,
              two_phase=bool(i & 1), tiny_queue=bool(i & 2))
    for sizes in ((1 << 12, 64), (4000, 400, 40, 4), (96, 32), (54, 27), (3000,)):
        text = workloads.text_versions(n=9999, base_len=700, sigma=9, edit_rate=5e-3, seed=len(sizes))
        for prune in (True, False):
            t = bt.Tree(text, 256, 2, sizes[-1], bt.BuildOptions(level_sizes=sizes, prune=prune, batch_workers=True))
            one = bt.Tree(text, 256, 2, sizes[-1], bt.BuildOptions(level_sizes=sizes, prune=prune))
            assert t.export() == one.export() == oracle.build(text, 2, sizes[-1], prune=prune, level_sizes=list(sizes)).export(), sizes


def test_long_runs():
    for text, tau, leaf in ((_runs_text(50_000, 1), 2, 8), (_runs_text(120_001, 2, b"abc", 500), 4, 27),
                            (_far_anchor_text(60_000, 5), 2, 128), (_far_anchor_text(50_001, 6), 4, 24)):
        check(text, tau, leaf)
        check(text, tau, leaf, prune=False, two_phase=True, tiny_queue=True)
