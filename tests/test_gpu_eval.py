"""The evaluation loss at the edges of its launches, against the oracle: fewer
samples than a tile, a ragged last tile, more samples than one pass holds,
deep and two-layer MLPs, up to 32 classes, unaligned samples; softmax
regression with every class group and ragged inputs; images that do not fill
a lane and more lanes than workers.  An evaluation between rounds leaves the
training as it was.

Bounds: 1e-5 for the fp32 path (sums of at most 1000 fp32 products); 1e-4 for
the bf16 ones (operands rounded alike on both sides; a hidden activation on a
rounding boundary moves by 2^-8 of itself, one of hundreds in a logit of one of
at least 32 samples)."""
import numpy as np
import pytest
import torch

import paper_2102_08550_gb300 as P
import synth
from oracle import bf16 as obf16
from oracle import conv as oconv
from oracle import model as omodel

pytestmark = pytest.mark.gpu


def _set(D, C, n, seed):
    rng = np.random.default_rng(seed)
    return rng.standard_normal((n, D)).astype(np.float32), rng.integers(0, C, n).astype(np.int32)


def _ctx(dims, B, W, dev, bf16=True, flat=None):
    x, y = torch.zeros(B, dims[0], device=dev), torch.zeros(B, dtype=torch.int32, device=dev)
    return P.OscarsContext(num_workers=W, dims=dims, batch=B, shards=[(x, y)] * W, bf16=bf16, M=2, init_params=flat,
                           t_ticks=[1] * W, stream=torch.cuda.current_stream().cuda_stream)


def _eval(ctx, X, y, dev, shift=0):
    buf = torch.zeros(X.size + shift, device=dev)
    buf[shift:] = torch.from_numpy(X.reshape(-1)).to(dev)
    xt = buf[shift:].view(X.shape)
    return ctx.eval_loss(xt, torch.from_numpy(y).to(dev))


@pytest.mark.parametrize("dims,B,n,shift", [
    ([64, 128, 10], 32, 32, 0), ([72, 128, 10], 32, 224, 0), ([784, 512, 10], 64, 16384 + 192, 0),
    ([40, 256, 128, 2], 64, 320, 0), ([200, 128, 384, 128, 32], 32, 96, 1), ([8, 640, 17], 256, 512, 3),
], ids=lambda v: "-".join(map(str, v)) if isinstance(v, list) else str(v))
def test_eval_mlp(cuda_device, dims, B, n, shift):
    rng = np.random.default_rng(n)
    layers = [(rng.uniform(-1, 1, (o, i)).astype(np.float32) / np.sqrt(i), rng.uniform(-0.1, 0.1, o).astype(np.float32))
              for i, o in zip(dims[:-1], dims[1:])]
    layers = [(a.astype(np.float32), b.astype(np.float32)) for a, b in layers]
    ctx = _ctx(dims, B, 3, cuda_device, flat=torch.from_numpy(synth.flatten_layers(layers)).to(cuda_device))
    X, y = _set(dims[0], dims[-1], n, n + 1)
    ref = omodel.loss_of(layers, X, y, obf16.round_bf16)
    for _ in range(2):
        got = _eval(ctx, X, y, cuda_device, shift)
        assert abs(got - ref) <= 1e-4 * abs(ref), (got, ref)
    ctx.close()


@pytest.mark.parametrize("D,C,n", [(1, 2, 1), (33, 4, 3), (784, 10, 500), (100, 13, 65), (95, 20, 64), (64, 32, 2000),
                                   (1000, 8, 4097)])
def test_eval_softreg(cuda_device, D, C, n):
    rng = np.random.default_rng(D)
    layers = [(rng.uniform(-1, 1, (C, D)).astype(np.float32), rng.uniform(-0.1, 0.1, C).astype(np.float32))]
    ctx = _ctx([D, C], 4, 2, cuda_device, bf16=False, flat=torch.from_numpy(synth.flatten_layers(layers)).to(cuda_device))
    X, y = _set(D, C, n, n)
    ref = omodel.loss_of(layers, X, y, obf16.identity)
    got = _eval(ctx, X, y, cuda_device)
    assert abs(got - ref) <= 1e-5 * abs(ref), (got, ref)
    ctx.close()


@pytest.mark.parametrize("n,W", [(1, 2), (17, 2), (100, 3), (7, 1), (33, 2), (48, 1)])   # a lane alone, whole or not, and others
def test_eval_cnn(cuda_device, n, W):
    B, dev = 16, cuda_device
    w = synth.ConvWorkload("cnn-eval", W, [32 * 32 * 3, 10], B, 0.05, B, 4, 1, clip=3.0, blocks=1, in_ch=3)
    m = oconv.CNN(32, 32, 3, 64, 1, 10)
    p0 = synth.init_cnn_np(w)
    x, y = torch.zeros(B, 3072, device=dev), torch.zeros(B, dtype=torch.int32, device=dev)
    ctx = P.OscarsContext(num_workers=W, dims=w.cnn_dims, model=P.MODEL_CNN, blocks=1, batch=B, shards=[(x, y)] * W, M=2,
                          init_params=torch.from_numpy(m.flatten(p0)).to(dev), t_ticks=[1] * W,
                          stream=torch.cuda.current_stream().cuda_stream)
    Xe, ye = synth.eval_np(w, n=n)
    ref = m.loss_of(p0, Xe, ye, obf16.round_bf16)
    got = _eval(ctx, Xe, ye, dev)
    assert abs(got - ref) <= 1e-4 * abs(ref), (got, ref)
    ctx.close()


@pytest.mark.parametrize("dims,flags", [([64, 128, 10], 0), ([64, 128, 128, 10], 0), ([64, 128, 10], P.FLAG_NO_GRAPH)])
def test_eval_between_rounds_changes_nothing(cuda_device, dims, flags):
    w = synth.TrainWorkload("eval-between", 3, dims, 32, 0.05, 200, 4, 3)
    dev = cuda_device
    shards = [synth.shard_t(w, k, dev, n=200) for k in range(3)]
    flat = torch.from_numpy(synth.flatten_layers(synth.init_layers_np(w))).to(dev)
    X, y = synth.eval_np(w, n=256)
    out = []
    for evaluate in (False, True):
        ctx = P.OscarsContext(num_workers=3, dims=dims, batch=32, shards=shards, M=4, init_params=flat, t_ticks=[3, 4, 5],
                              stream=torch.cuda.current_stream().cuda_stream, flags=flags)
        losses = []
        for _ in range(3):
            _, loss = ctx.local_steps()
            if evaluate:
                _eval(ctx, X, y, dev)
            ctx.push_merge()
            losses.append(loss)
        m = torch.empty(ctx.P, device=dev)
        ctx.pull(m)
        torch.cuda.synchronize()
        out.append((losses, m.cpu()))
        ctx.close()
    assert out[0][0] == out[1][0]
    torch.testing.assert_close(out[0][1], out[1][1], rtol=0, atol=0)


def test_eval_on_a_nearly_full_device(cuda_device):
    """A layer of 16384 outputs: two buffers of 16384 samples want 1.1 GB.  With 400 MB left the evaluation takes
    fewer samples a pass, and gives the same loss (sums of the same 32-sample partials)."""
    dims, B, n, dev = [64, 16384, 128, 10], 32, 16384 + 96, cuda_device
    rng = np.random.default_rng(3)
    flat = torch.from_numpy(synth.flatten_layers(
        [(rng.uniform(-1, 1, (o, i)).astype(np.float32) / np.float32(np.sqrt(i)), np.zeros(o, np.float32))
         for i, o in zip(dims[:-1], dims[1:])])).to(dev)
    X, y = _set(dims[0], dims[-1], n, 5)
    x, yd = torch.from_numpy(X).to(dev), torch.from_numpy(y).to(dev)
    ctx = _ctx(dims, B, 1, dev, flat=flat)
    want = ctx.eval_loss(x, yd)
    ctx.close()
    ctx = _ctx(dims, B, 1, dev, flat=flat)
    ctx.eval_loss(x[:B], yd[:B])
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    hold = torch.empty(max(free - 400 * 2 ** 20, 1), dtype=torch.uint8, device=dev)
    try:
        first = ctx.eval_loss(x, yd)
        again = ctx.eval_loss(x, yd)
    finally:
        del hold
        torch.cuda.empty_cache()
    later = ctx.eval_loss(x[:n - 96], yd[:n - 96])
    ctx.close()
    assert first == again and abs(first - want) <= 1e-6 * abs(want), (first, again, want)
    assert abs(later - want) <= 0.05 * abs(want)
