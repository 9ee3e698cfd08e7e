"""The prefix-fingerprint kernels at the edges of their tiles (1024 chunks of
32 bytes; four chunks a thread), with unaligned texts and both moduli, every
value against Horner's rule in Python integers."""
import numpy as np
import pytest
import torch

import oracle
from paper_2512_23314_gb300 import bt, workloads

pytestmark = pytest.mark.gpu

TILE = 32 * 1024


@pytest.mark.parametrize("n", [32, 127, 128, 32 * 1023, TILE - 1, TILE, TILE + 31, TILE + 32, 3 * TILE, 3 * TILE + 97])
@pytest.mark.parametrize("shift,q,noalloc", [(0, 0, False), (0, 0, True), (5, 0, False), (16, 331, False)])
def test_every_prefix(n, shift, q, noalloc):
    text = workloads.random_bytes(n + shift, 256, n)
    d = torch.from_numpy(text).cuda()[shift:]
    out = torch.full((n // 32 + 1,), -1, dtype=torch.int64, device="cuda")
    f = bt.bt_prefix_fingerprints_noalloc if noalloc else bt.bt_prefix_fingerprints
    f(d, n, 3, q, 32, out)
    B, Q, h, want = oracle.base(3, q), q or (1 << 61) - 1, 0, [0]
    for i, c in enumerate(text[shift:].tolist(), 1):
        h = (h * B + c + 1) % Q
        if i % 32 == 0:
            want.append(h)
    assert out.cpu().numpy().tolist() == want
