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


@pytest.mark.parametrize("n", [2 * TILE - 33, 2 * TILE - 1, 2 * TILE, 2 * TILE + 32, 6 * TILE + 31, 8 * TILE, 2 * TILE * 511 + 5,
                               2 * TILE * 513, 2 * TILE * 8200 + 77])
@pytest.mark.parametrize("q", [0, 331])
def test_steps_of_large_tiles(n, q):
    """Tiles of 2048 chunks, up to more of them than the threads that add them up: each value from the one before, at
    every edge of a tile and of a thread's chunks nearby and at random."""
    text = workloads.random_bytes(n, 256, n % 1000)
    out = torch.full((n // 32 + 2,), -1, dtype=torch.int64, device="cuda")
    bt.bt_prefix_fingerprints(torch.from_numpy(text).cuda(), n, 7, q, 32, out[1:])  # (an odd place)
    h, B, Q = out.cpu().numpy()[1:], oracle.base(7, q), q or (1 << 61) - 1
    last = n // 32
    js = np.random.default_rng(n).integers(0, last, 500).tolist()
    js += [t + d for t in range(0, last, 2048) for d in (-2, -1, 0, 7, 8)][-4000:] + [last - 1]
    assert h[0] == 0
    for j in js:
        if 0 <= j < last:
            x = int(h[j])
            for c in text[32 * j:32 * j + 32].tolist():
                x = (x * B + c + 1) % Q
            assert x == h[j + 1], j
