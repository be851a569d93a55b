"""Forward and input-gradient products of the per-layer path: clusters of 4
and of 2 CTAs per tile, K-blocks that do not divide evenly among them, a last
K-block that is partly past K, and one worker alone; unsplit with one or two
tiles of 64 samples, and more K-blocks than ring entries; against the oracle for one local step on integer inputs (the first
layer's forward is exact in any summation order).

With 20 workers a logit gradient may round to the other of two bf16
neighbours than the oracle's (they agree to fp32 rounding before): one unit in
the last place is 2^-8 of a value that is at most 3 times the gradients' root
mean square, and a bias that starts at zero is the sum of W B C such terms of
either sign, so the biases are compared to 3 2^-8 / sqrt(W B C) there.  One
sample's mask bit wrong in one feature would move it by 1 / sqrt(W B)."""
import numpy as np
import pytest
import torch

import paper_2102_08550_gb300 as P
import synth
from oracle import run as orun
from tests.gpu_util import LOSS_RTOL, PARAM_RTOL, per_tensor_errors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,B,W", [
    ([1000, 128, 10], 32, 3),         # forward: 16 K-blocks on 4 CTAs, the last 40 wide
    ([1096, 256, 17], 64, 1),         # forward: 18 K-blocks on 4 CTAs (4, 5, 4, 5)
    ([520, 128, 17], 64, 3),          # forward: 9 K-blocks on 2 CTAs, the last 8 wide
    ([64, 128, 512, 10], 32, 2),      # input gradient: 8 K-blocks on 2 CTAs
    ([64, 128, 1024, 16], 64, 2),     # input gradient: 16 K-blocks on 4 CTAs
    ([64, 128, 512, 10], 128, 2),     # input gradient: 8 K-blocks on 2 CTAs, two tiles of 64 samples
    ([64, 256, 128, 10], 128, 2),     # unsplit, fewer K-blocks than ring entries
    ([64, 1024, 1024, 10], 64, 20),   # unsplit, 16 K-blocks: the mask's entry waits for the ring
    ([64, 1024, 1024, 10], 128, 20),
], ids=lambda v: "-".join(map(str, v)) if isinstance(v, list) else str(v))
def test_split_k_one_step(cuda_device, dims, B, W):
    C, n, dev = dims[-1], 2 * B, cuda_device
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
    errs = per_tensor_errors(out.cpu().numpy(), recs[0].x_g, dims)   # weights and biases in turn
    assert np.max(errs[0::2]) <= PARAM_RTOL
    assert np.max(errs[1::2]) <= (PARAM_RTOL if W < 20 else 3 * 2.0 ** -8 / np.sqrt(W * B * C))
