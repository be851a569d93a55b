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

import paper_2102_08550_gb300 as P
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


def _shared_shard(D, C, B, n=300):
    rng = np.random.default_rng(D * 1000 + C * 10 + B)
    X = rng.standard_normal((n, D)).astype(np.float32)
    y = rng.integers(0, C, n).astype(np.int32)
    flat = np.concatenate([rng.uniform(-1, 1, C * D) / np.sqrt(D), rng.uniform(-0.1, 0.1, C)]).astype(np.float32)
    return X, y, flat


def _context(D, C, B, W, X, y, flat, dev, tau):
    xd, yd = torch.from_numpy(X).to(dev), torch.from_numpy(y).to(dev)
    ctx = P.OscarsContext(num_workers=W, dims=[D, C], batch=B, lr=0.05, bf16=False, shards=[(xd, yd)] * W, M=8,
                          init_params=torch.from_numpy(flat).to(dev), t_ticks=[1] * W,
                          stream=torch.cuda.current_stream().cuda_stream)
    ctx.set_local_steps(tau)
    return ctx


# 512, 256 and 128 threads a CTA, and more workers than any of them runs at once
@pytest.mark.parametrize("D,C,B", [(784, 10, 8), (333, 26, 100), (60, 25, 65), (16, 2, 1), (40, 32, 33)])
@pytest.mark.parametrize("W", [3, 17, 40, 150])
def test_cluster_round_workers_share_sms(cuda_device, D, C, B, W):
    X, y, flat = _shared_shard(D, C, B)
    tau = [1 + k % 3 for k in range(W)]
    ctx = _context(D, C, B, W, X, y, flat, cuda_device, tau)
    _, losses = ctx.local_steps()
    got = torch.empty(W, flat.size, device=cuda_device)
    for k in range(W):
        ctx.read_replica(k, got[k])
    torch.cuda.synchronize()
    ctx.close()
    for t in range(1, 4):
        ref, ref_loss = oracle_steps(flat, X, y, 0, t, D, C, B, 0.05)
        check(got[t - 1].cpu().numpy(), losses[t - 1], ref, ref_loss, C, D)
        for k in range(t - 1, W, 3):
            assert torch.equal(got[k], got[t - 1]) and losses[k] == losses[t - 1]


@pytest.mark.parametrize("D,C,B", [(784, 10, 8), (64, 10, 64), (1500, 3, 16)])
def test_thirty_workers_take_one_wave(cuda_device, D, C, B):
    """30 workers run side by side: far less than the two waves (2.0 to 2.4
    times one worker's round) of one CTA an SM; 1.1 to 1.5 when they share SMs."""
    X, y, flat = _shared_shard(D, C, B)

    def us(W):
        ctx = _context(D, C, B, W, X, y, flat, cuda_device, [8] * W)
        best = float("inf")
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(10):
                ctx.local_steps(want_loss=False)
                ctx.push_merge()
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) * 100)
        ctx.close()
        return best

    assert us(30) < 1.8 * us(1)


@pytest.mark.parametrize("D,C,B,steps", [(4, 3, 5, 1), (784, 10, 32, 3), (60, 32, 512, 1)])   # the cluster kernel, and one CTA
def test_infinite_loss_stays_infinite(cuda_device, D, C, B, steps):
    """A label whose logit is minus infinity has an infinite loss (and a finite gradient); so has the step and the
    round.  NaN is for undefined values and for a wait that ran out."""
    dev = cuda_device
    p = torch.zeros(C * D + C, device=dev)
    p[0] = -1e38
    x, y = torch.zeros(2 * B, D, device=dev), torch.ones(2 * B, dtype=torch.int32, device=dev)
    x[1, 0], y[1] = 100.0, 0          # logits (-inf, 0, ...), label 0
    out, loss = torch.empty_like(p), torch.empty(1, device=dev)
    call(p, out, x, y, 2 * B, 0, steps, D, C, B, 0.05, loss)
    assert loss.item() == float("inf")
    assert torch.isfinite(out).all()
    ctx = P.OscarsContext(num_workers=2, dims=[D, C], batch=B, lr=0.05, bf16=False, shards=[(x, y)] * 2, M=8,
                          init_params=p, t_ticks=[1, 1], stream=torch.cuda.current_stream().cuda_stream)
    ctx.set_local_steps([steps] * 2)
    _, losses = ctx.local_steps()
    ctx.close()
    assert losses == [float("inf")] * 2
