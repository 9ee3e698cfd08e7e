"""Batches at the edges of the batched kernel's launch shapes (four, two or one
CTA per SM, narrow CTAs for few short documents): every document's tree is the
one a single build gives."""
import numpy as np
import pytest
import torch

from paper_2512_23314_gb300 import bt, workloads

pytestmark = pytest.mark.gpu

K = 1 << 10


def docs_of(count, size, seed):
    """Versions, DNA copies, random bits (every key stays open: the largest tables), random bytes (256 symbols)."""
    for i in range(count):
        n = max(1, size - 37 * (i % 11))
        s = seed + i % 8
        yield (workloads.text_versions(n=n, base_len=max(64, n // 12), sigma=96, edit_rate=5e-3, seed=s) if i % 4 == 0 else
               workloads.dna_genome(n=n, genome_len=max(100, n // 9), snp_rate=1e-2, indel_rate=2e-3, seed=s) if i % 4 == 1 else
               workloads.random_bytes(n, 2, s) if i % 4 == 2 else workloads.random_bytes(n, 256, s))


@pytest.mark.parametrize("count,size,longest,threads,per_sm", [
    (8, 100, 0, 512, 1), (20, 8 * K, 0, 512, 1), (20, 8 * K + 400, 0, 1024, 1),
    (170, 3 * K, 0, 256, 4), (160, 40 * K, 0, 1024, 1), (160, 30 * K, 128 * K, 256, 4), (160, 20 * K, 128 * K + 1, 1024, 1),
    (330, 40 * K, 0, 512, 2), (330, 40 * K, 513 * K, 1024, 1),
])
@pytest.mark.parametrize("tau,leaf", [(4, 32), (2, 9)])
def test_shapes(count, size, longest, threads, per_sm, tau, leaf):
    docs = list(docs_of(count, size, size % 1000))
    if longest:
        docs[1] = workloads.dna_genome(n=longest, genome_len=longest // 9, seed=1)
    hs = bt.bt_build_batch(docs, [len(t) for t in docs], [256] * count, [tau] * count, [leaf] * count)
    report = bt.bt_batch_report()
    try:
        if torch.cuda.get_device_properties(0).multi_processor_count == 152:
            assert (report["threads"], report["ctas_per_sm"]) == (threads, per_sm)
        for i in list(range(0, count, max(1, count // 12))) + [1, count - 1]:
            one = bt.Tree(docs[i], 256, tau, leaf, bt.BuildOptions(batch_workers=True))
            assert bt.bt_export(hs[i]) == one.export(), i
        m = 64
        for i in (0, 2, 3, count - 1):  # counters
            t, n = docs[i], len(docs[i])
            at = np.random.default_rng(i).integers(0, n, m)
            args = np.stack([t[at].astype(np.int64), at], 1)
            out = torch.empty(m, dtype=torch.int64, device="cuda")
            bt.bt_query_batch(hs[i], bt.BT_Q_RANK, torch.from_numpy(args).cuda(), m, out)
            assert out.tolist() == [int((t[:p] == c).sum()) for c, p in args.tolist()], i
    finally:
        for h in hs:
            bt.bt_free(h)
