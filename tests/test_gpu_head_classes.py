"""The tensor-core last layer at its edges: 2 to 32 classes (padded to 16 or
32 columns), one and two feature halves per CTA, one CTA and a cluster, every
batch it takes, against the oracle for one local step per worker on integer
inputs (the first layer's forward is exact in any summation order), so that
the merged model must match to 1e-5 per tensor, as in the other exact-input
cases."""
import numpy as np
import pytest
import torch

import paper_2102_08550_gb300 as P
import synth
from oracle import run as orun
from tests.gpu_util import LOSS_RTOL, PARAM_RTOL, per_tensor_errors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,B", [
    ([64, 128, 2], 32), ([64, 256, 9], 64), ([64, 640, 10], 128), ([72, 128, 11], 128), ([64, 1024, 16], 64),
    ([64, 384, 17], 32), ([136, 256, 31], 128), ([64, 768, 32], 64), ([64, 128, 128, 17], 64), ([64, 128, 128, 24], 32),
], ids=lambda v: "-".join(map(str, v)) if isinstance(v, list) else str(v))
def test_head_classes_one_step(cuda_device, dims, B):
    W, C, n, dev = 3, dims[-1], 2 * B, cuda_device
    rng = np.random.default_rng(sum(dims))
    layers = [((rng.integers(-4, 5, (o, i)) * 2.0 ** -7).astype(np.float32), np.zeros(o, np.float32))
              for i, o in zip(dims[:-1], dims[1:])]
    shards = [(rng.integers(-3, 4, (n, dims[0])).astype(np.float32), rng.integers(0, C, n).astype(np.int32))
              for _ in range(W)]
    ctx = P.OscarsContext(num_workers=W, dims=dims, batch=B, lr=0.05, M=2, t_ticks=[1] * W, flags=P.FLAG_PER_LAYER,
                          shards=[(torch.from_numpy(x).to(dev), torch.from_numpy(y).to(dev)) for x, y in shards],
                          init_params=torch.from_numpy(synth.flatten_layers(layers)).to(dev),
                          stream=torch.cuda.current_stream().cuda_stream)
    ctx.set_local_steps([1] * W)
    _, loss = ctx.local_steps()
    ctx.push_merge()
    out = torch.empty(ctx.P, device=dev)
    ctx.pull(out)
    torch.cuda.synchronize()
    assert P.oscars_check_padding(ctx.handle) == 0
    ctx.close()
    _, recs = orun.run(dims, layers, shards, t_iter=np.ones(W, np.int64), M=2, rounds=1, batch=B, lr=0.05, bf16=True,
                       tau_override=[1] * W)
    np.testing.assert_allclose(loss, recs[0].worker_loss, rtol=LOSS_RTOL)
    assert np.max(per_tensor_errors(out.cpu().numpy(), recs[0].x_g, dims)) <= PARAM_RTOL
