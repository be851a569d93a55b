"""MLPs with more hidden layers than one weight-gradient launch takes (four):
the second launch requests its first master block while the first one runs.
One local step on integer inputs against the oracle (the first layer's forward
is exact in any summation order; bound as in the other exact-input cases), and
several rounds bit for bit against the same context while profiling, where no
kernel starts before the one ahead of it has ended."""
import numpy as np
import pytest
import torch

import paper_2102_08550_gb300 as P
import synth
from oracle import run as orun
from tests.gpu_util import LOSS_RTOL, PARAM_RTOL, per_tensor_errors

pytestmark = pytest.mark.gpu

DIMS = [[64, 128, 128, 256, 128, 128, 10], [72, 128, 256, 128, 128, 128, 128, 128, 128, 128, 17]]   # 2 and 3 launches


def _inputs(dims, B, W, n):
    rng = np.random.default_rng(sum(dims) + B)
    layers = [((rng.integers(-4, 5, (o, i)) * 2.0 ** -5).astype(np.float32), np.zeros(o, np.float32))
              for i, o in zip(dims[:-1], dims[1:])]
    shards = [(rng.integers(-3, 4, (n, dims[0])).astype(np.float32), rng.integers(0, dims[-1], n).astype(np.int32))
              for _ in range(W)]
    return layers, shards


def _rounds(dims, B, W, layers, shards, tau, rounds, dev, flags):
    ctx = P.OscarsContext(num_workers=W, dims=dims, batch=B, lr=0.05, M=8, t_ticks=[1] * W, flags=flags,
                          shards=[(torch.from_numpy(x).to(dev), torch.from_numpy(y).to(dev)) for x, y in shards],
                          init_params=torch.from_numpy(synth.flatten_layers(layers)).to(dev),
                          stream=torch.cuda.current_stream().cuda_stream)
    ctx.set_local_steps(tau)
    losses = []
    for _ in range(rounds):
        losses.append(ctx.local_steps()[1])
        ctx.push_merge()
    out = torch.empty(ctx.P, device=dev)
    ctx.pull(out)
    torch.cuda.synchronize()
    assert P.oscars_check_padding(ctx.handle) == 0
    ctx.close()
    return losses, out.cpu().numpy()


@pytest.mark.parametrize("dims", DIMS, ids=len)
@pytest.mark.parametrize("B", [32, 64, 128])
def test_deep_mlp_one_step(cuda_device, dims, B):
    W = 3
    layers, shards = _inputs(dims, B, W, 2 * B)
    losses, got = _rounds(dims, B, W, layers, shards, [1] * W, 1, cuda_device, 0)
    _, recs = orun.run(dims, layers, shards, t_iter=np.ones(W, np.int64), M=2, rounds=1, batch=B, lr=0.05, bf16=True,
                       tau_override=[1] * W)
    np.testing.assert_allclose(losses[0], recs[0].worker_loss, rtol=LOSS_RTOL)
    assert np.max(per_tensor_errors(got, recs[0].x_g, dims)) <= PARAM_RTOL


@pytest.mark.parametrize("dims", DIMS, ids=len)
@pytest.mark.parametrize("B,W,flags", [(32, 1, 0), (64, 5, 0), (128, 20, 0), (64, 5, P.FLAG_NO_GRAPH)])
def test_deep_mlp_overlapped_launches(cuda_device, dims, B, W, flags):
    layers, shards = _inputs(dims, B, W, 300)
    tau = [1 + (3 * k) % 5 for k in range(W)]
    a = _rounds(dims, B, W, layers, shards, tau, 4, cuda_device, flags)
    b = _rounds(dims, B, W, layers, shards, tau, 4, cuda_device, flags | P.FLAG_PROFILE)
    assert a[0] == b[0] and np.isfinite(a[0]).all()
    np.testing.assert_array_equal(a[1], b[1])
