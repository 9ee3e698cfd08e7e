"""Rank and select without stored leaf counters at leaf lengths that leave the
blocks' leaf text at every alignment: every occurrence against naive counts."""
import numpy as np
import pytest
import torch

from paper_2512_23314_gb300 import bt, workloads
from tests.test_gpu_query_layout import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("leaf", [1, 3, 13, 15, 16, 17, 24, 31, 33, 47, 63, 64, 65, 79, 80, 81, 127, 200, 1000])
@pytest.mark.parametrize("tau", [2, 4])
def test_every_alignment(leaf, tau):
    n = 60 * leaf + leaf // 2 + 5
    for T in (workloads.text_versions(n=n, base_len=max(64, n // 9), sigma=5, edit_rate=5e-3, seed=leaf),
              workloads.random_bytes(n, 2, leaf), np.full(n, 9, np.uint8)):
        for counts in (True, False):
            t = bt.Tree(torch.from_numpy(T).cuda(), 256, tau, leaf, bt.BuildOptions(leaf_counts=counts))
            check(t.handle, T)
            t.close()


def test_batched_trees():
    """The leaf text of a batched tree starts anywhere in its pool."""
    docs = [workloads.random_bytes(700 + 13 * i, 4, i) for i in range(24)]
    hs = bt.bt_build_batch(docs, [len(T) for T in docs], [256] * 24, [2] * 24, [17 + i for i in range(24)])
    for h, T in zip(hs, docs):
        check(h, T)
        bt.bt_free(h)
