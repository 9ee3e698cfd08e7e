"""One text by one CTA, a batch's documents by clusters of CTAs, and the levels pruned in one launch.

The three share the device code of the batched kernel; each is compared with the
oracle or with the single-text path at the sizes where the choice turns.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2512_23314_gb300 import bt, workloads

pytestmark = pytest.mark.gpu


def kinds(n, seed):
    yield workloads.text_versions(n=n, base_len=max(64, n // 12), sigma=60, edit_rate=5e-3, seed=seed)
    yield workloads.dna_genome(n=n, genome_len=max(100, n // 9), snp_rate=1e-2, indel_rate=2e-3, seed=seed)
    yield workloads.random_bytes(n, 256, seed)
    yield np.full(n, 97, np.uint8)


def answers(t, n, seed):
    rng = np.random.default_rng(seed)
    m = 300
    i, c = rng.integers(0, n, m), rng.integers(0, 256, m)
    got = []
    for kind, args in ((bt.BT_Q_ACCESS, i), (bt.BT_Q_RANK, np.stack([c, i + 1], 1).ravel()),
                       (bt.BT_Q_SELECT, np.stack([c, i // 8 + 1], 1).ravel())):
        out = torch.zeros(m, dtype=torch.int64, device="cuda")
        bt.bt_query_batch(t.handle, kind, torch.from_numpy(args.astype(np.int64)).cuda(), m, out)
        torch.cuda.synchronize()
        got.append(out.cpu().numpy())
    return got


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 500, 4096, 16383, 16384, 16385])
@pytest.mark.parametrize("tau,leaf", [(2, 1), (4, 16), (3, 27), (8, 64)])
def test_one_launch(n, tau, leaf):
    for k, text in enumerate(kinds(n, n + tau)):
        for prune in (True, False):
            d = torch.from_numpy(np.concatenate([text[:1], text])).cuda()[1:]  # (an odd address)
            one = bt.Tree(d, 256, tau, leaf, bt.BuildOptions(prune=prune))
            many = bt.Tree(d, 256, tau, leaf, bt.BuildOptions(prune=prune, batch_workers=True))
            blob = one.export()
            assert blob == many.export(), (n, k, prune)
            if k < 2:
                assert blob == oracle.build(text, tau, leaf, prune=prune).export()
            for a, b in zip(answers(one, n, k), answers(many, n, k)):
                assert np.array_equal(a, b), (n, k, prune)


@pytest.mark.parametrize("ndocs", [1, 3, 9, 38, 77])
@pytest.mark.parametrize("tau,leaf,modulus", [(2, 32, 0), (4, 16, 0), (5, 40, 331), (3, 7, 331)])
def test_clusters(ndocs, tau, leaf, modulus):
    if ndocs > 9 and (modulus or leaf != 32):
        pytest.skip("the widths of the clusters are covered by one option")
    size = (128 << 10) + (200 << 10) // ndocs
    if modulus:
        size = 128 << 10
    texts = [t for s in range((ndocs + 2) // 3)
             for t in list(kinds(size + 517 * s, s))[:2] + [np.full(size + 3, 98, np.uint8)]][:ndocs]
    opts = bt.BuildOptions(modulus=modulus, seed=5).to_c()
    dev = [torch.from_numpy(t).cuda() for t in texts]
    handles = bt.bt_build_batch(dev, [len(t) for t in texts], [256] * ndocs, [tau] * ndocs, [leaf] * ndocs, opts=opts[0])
    try:
        for i, (h, d) in enumerate(zip(handles, dev)):
            one = bt.Tree(d, 256, tau, leaf, bt.BuildOptions(seed=5, batch_workers=True))
            assert bt.bt_export(h) == one.export(), i
    finally:
        for h in handles:
            bt.bt_free(h)


@pytest.mark.parametrize("blocks", [16383, 16384, 16385, 33000])
def test_levels_pruned_in_one_launch(blocks):
    for leaf, tau in ((8, 2), (32, 4)):
        n = blocks * leaf - 3
        for text in list(kinds(n, blocks))[:2] + [workloads.random_bytes(n, 4, 1)]:
            for rounds in (0, 2):
                t = bt.Tree(torch.from_numpy(text).cuda(), 256, tau, leaf, bt.BuildOptions(max_rounds=rounds, batch_workers=True))
                assert t.export() == oracle.build(text, tau, leaf).export(), (n, leaf, rounds)
