"""Softmax regression on a cluster of 8 CTAs per worker: the shapes where its
split of a step can go wrong (class groups and their padding, rows per lane,
column and row splits, ranks without columns or without rows, unaligned
rows), each against the oracle's steps.  The bound is the repository's for
fp32 paths: a handful of steps of fp32 sums over at most 1500 products (unit
roundoff 6e-8, sums in another order) stays well below 1e-5 of the largest
parameter."""
import numpy as np
import pytest
import torch

import synth
from tests.test_zz_no_alloc import call, check, oracle_steps

pytestmark = pytest.mark.gpu

# (D, C, B, n, tau): classes per group 4, 5, 7, 8; one and two rows per lane
SHAPES = [
    (1, 2, 1, 5, 3),          # seven ranks without columns, seven without rows
    (3, 3, 7, 9, 4),          # a column slice shorter than 4, the shard wraps inside a batch
    (31, 5, 32, 100, 3),      # ragged columns, one row per lane
    (64, 9, 33, 100, 3),      # second row block of one row
    (784, 10, 32, 200, 3),
    (785, 10, 32, 200, 3),    # rows not 16-byte aligned
    (333, 26, 100, 300, 3),
    (100, 17, 64, 200, 3),
    (60, 25, 65, 200, 3),
    (40, 32, 256, 300, 2),    # the most classes
    (1500, 13, 10, 100, 3),
    (64, 10, 512, 700, 2),    # the largest batch
    (60, 32, 512, 700, 2),    # the exchange buffers do not fit: one CTA
]


@pytest.mark.parametrize("D,C,B,n,tau", SHAPES, ids=["x".join(map(str, s[:3])) for s in SHAPES])
def test_cluster_steps_match_oracle(cuda_device, D, C, B, n, tau):
    rng = np.random.default_rng(D * 1000 + C * 10 + B)
    X = rng.standard_normal((n, D)).astype(np.float32)
    y = rng.integers(0, C, n).astype(np.int32)
    flat = np.concatenate([rng.uniform(-1, 1, C * D) / np.sqrt(D), rng.uniform(-0.1, 0.1, C)]).astype(np.float32)
    dev = cuda_device
    p, out, loss = torch.from_numpy(flat).to(dev), torch.empty(C * D + C, device=dev), torch.empty(1, device=dev)
    xd, yd = torch.from_numpy(X).to(dev), torch.from_numpy(y).to(dev)
    cursor = n - 1
    call(p, out, xd, yd, n, cursor, tau, D, C, B, 0.05, loss)
    ref, ref_loss = oracle_steps(flat, X, y, cursor, tau, D, C, B, 0.05)
    check(out.cpu().numpy(), loss.item(), ref, ref_loss, C, D)
    again = torch.empty_like(out)
    call(p, again, xd, yd, n, cursor, tau, D, C, B, 0.05, loss)
    torch.testing.assert_close(again, out, rtol=0, atol=0)   # fixed summation order
