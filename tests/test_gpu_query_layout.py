"""Queries on the record and counter layout: arities read in groups of four or
one by one, counters of one, two and four bytes, trees whose base level is the
first, the last or in between, alphabets up to 256 symbols, single and batched
builds.  Every position and every occurrence against naive counts."""
import numpy as np
import pytest
import torch

from paper_2512_23314_gb300 import bt, workloads

pytestmark = pytest.mark.gpu


def ask(handle, kind, args):
    out = torch.empty(len(args), dtype=torch.int64, device="cuda")
    bt.bt_query_batch(handle, kind, torch.from_numpy(np.ascontiguousarray(args, np.int64)).cuda(), len(args), out)
    return out.cpu().numpy()


def check(handle, T):
    n = len(T)
    assert np.array_equal(ask(handle, bt.BT_Q_ACCESS, np.arange(n)), T)
    rng = np.random.default_rng(n)
    for c in np.unique(T)[:: max(1, len(np.unique(T)) // 12)]:
        where = np.flatnonzero(T == c)
        i = np.unique(np.concatenate([rng.integers(0, n + 1, 3000), [0, n, n - 1, where[0], where[-1] + 1]]))
        assert np.array_equal(ask(handle, bt.BT_Q_RANK, np.stack([np.full(len(i), c), i], 1)),
                              np.searchsorted(where, i, side="left")), c
        j = np.arange(1, len(where) + 1)
        assert np.array_equal(ask(handle, bt.BT_Q_SELECT, np.stack([np.full(len(j), c), j], 1)), where), c
    assert (ask(handle, bt.BT_Q_RANK, [[c, n + 1], [300, 0]]) == -1).all()
    assert (ask(handle, bt.BT_Q_SELECT, [[c, 0], [c, len(where) + 1]]) == -1).all()


def texts(sigma):
    yield workloads.text_versions(n=70_001, base_len=3000, sigma=sigma, seed=sigma)
    yield workloads.random_bytes(20_003, sigma, 3)          # every level has all its blocks
    yield np.resize(workloads.random_bytes(7, sigma, 1), 300_017)   # pointers from the first level on, long blocks
    yield np.full(1000, 7, np.uint8)


@pytest.mark.parametrize("tau", [2, 3, 4, 5, 8, 16])
@pytest.mark.parametrize("sigma", [2, 96, 256])
def test_single_tree(tau, sigma):
    for k, T in enumerate(texts(sigma)):
        for kw in ({"prune": bool(k & 1)}, {"leaf_counts": True}):
            t = bt.Tree(torch.from_numpy(T).cuda(), 256, tau, (32, 20, 16, 64)[k], bt.BuildOptions(**kw))
            check(t.handle, T)
            t.close()


@pytest.mark.parametrize("tau", [2, 3, 4, 8])
def test_batched_trees(tau):
    docs = [T for sigma in (2, 96, 256) for T in texts(sigma)] + [np.full(1, 9, np.uint8), np.arange(40, dtype=np.uint8)]
    hs = bt.bt_build_batch(docs, [len(T) for T in docs], [256] * len(docs), [tau] * len(docs), [32] * len(docs))
    for h, T in zip(hs, docs):
        check(h, T)
        bt.bt_free(h)
