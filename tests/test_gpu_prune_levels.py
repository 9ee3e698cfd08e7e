"""Pruning trees whose levels do not grow downwards: a long level over few
children (few distinct short blocks) is pruned by the whole grid like any other
long level, and gives the oracle's tree."""
import time

import numpy as np
import pytest
import torch

import oracle
from paper_2512_23314_gb300 import bt, workloads

pytestmark = pytest.mark.gpu


def records(n, width, values, seed=7):
    r = np.random.default_rng(seed)
    words = r.integers(33, 127, (values, width), dtype=np.uint8)
    return np.ascontiguousarray(words[r.integers(0, values, n // width + 1)].reshape(-1)[:n])


@pytest.mark.parametrize("text,tau,leaf", [
    (records(4 << 20, 64, 4), 4, 32),           # 2048, 8192, 32768 and a few hundred blocks
    (records(2 << 20, 32, 12), 2, 16),          # 32768 over about 30000 over a few hundred
    (workloads.random_bytes(300_001, 2, 5), 2, 2),
])
@pytest.mark.parametrize("rounds", [0, 2])
def test_long_level_over_few_children(text, tau, leaf, rounds):
    t = bt.Tree(torch.from_numpy(text).cuda(), 256, tau, leaf, bt.BuildOptions(max_rounds=rounds))
    blocks = [s["nblocks"] for s in t.stats()]
    assert any(a > 2 * b and b <= 16384 for a, b in zip(blocks, blocks[1:])), blocks
    assert t.export() == oracle.build(text, tau, leaf).export()


def test_pruning_a_long_level_over_few_children_takes_the_grid():
    """16 MiB of random bits as bytes, blocks of 2 bytes at the bottom: levels of 2 M and 4 M blocks above a few
    hundred.  Pruning is a tenth of this build with the grid, and as long as the rest with one CTA."""
    d = torch.from_numpy(workloads.random_bytes(16 << 20, 2, 3)).cuda()

    def best(prune):
        times = []
        for _ in range(6):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            t = bt.Tree(d, 256, 2, 2, bt.BuildOptions(prune=prune))
            times.append(time.perf_counter() - t0)
            t.close()
        return min(times)

    plain, pruned = best(False), best(True)
    assert pruned < 1.5 * plain, (plain, pruned)
