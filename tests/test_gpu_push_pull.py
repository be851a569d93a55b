"""Pushed deltas merged into a padded slot in one launch, and the one-launch
pull, at the layouts where the pieces can go wrong: tensors of odd length
(their canonical offsets leave the 16-byte boundaries of the padded slot),
deltas that share a misalignment or do not, and an unaligned destination.
The merge is a handful of fp32 operations per element: 1e-6 of the largest
value.  The pull copies, so it is exact."""
import numpy as np
import pytest
import torch

import paper_2102_08550_gb300 as P
import synth
from oracle import merge as omerge

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,bf16,W,shifts", [
    ([333, 26], False, 5, [0]), ([333, 26], False, 3, [1]), ([18, 3], False, 2, [0, 2]),
    ([64, 128, 10], True, 4, [0]), ([72, 128, 128, 17], True, 3, [3]), ([64, 128, 10], True, 2, [0, 1]),
    ([72, 128, 128, 128, 128, 17], True, 3, [0]), ([72] + [128] * 14 + [17], True, 2, [1, 0]),   # 10 and 30 tensors
], ids=lambda v: "-".join(map(str, v)) if isinstance(v, list) else str(v))
@pytest.mark.parametrize("dst_shift", [0, 1])
def test_push_deltas_and_pull(cuda_device, dims, bf16, W, shifts, dst_shift):
    rng = np.random.default_rng(sum(dims) + W)
    w = synth.TrainWorkload("push", W, dims, 32, 0.05, 32, 4, 1, bf16=bf16)
    flat = synth.flatten_layers(synth.init_layers_np(w))
    n = flat.size
    d = (rng.standard_normal((W, n)) * 1e-2).astype(np.float32)
    dev = cuda_device
    rows = []
    for k in range(W):
        sh = shifts[k % len(shifts)]
        buf = torch.zeros(n + sh, device=dev)
        buf[sh:] = torch.from_numpy(d[k]).to(dev)
        rows.append(buf[sh:])
    x, y = torch.zeros(32, dims[0], device=dev), torch.zeros(32, dtype=torch.int32, device=dev)
    ctx = P.OscarsContext(num_workers=W, dims=dims, batch=32, shards=[(x, y)] * W, bf16=bf16, M=2,
                          init_params=torch.from_numpy(flat).to(dev), t_ticks=[1] * W,
                          stream=torch.cuda.current_stream().cuda_stream)
    ctx.push_merge(rows)
    ctx.push_merge(rows)
    out = torch.full((n + dst_shift + 1,), 7.0, device=dev)
    ctx.pull(out[dst_shift:dst_shift + n])
    host = torch.empty(n)
    ctx.pull(host)
    torch.cuda.synchronize()
    wk = np.full(W, 1.0 / W, np.float32)
    ref = omerge.merge_deltas(omerge.merge_deltas(flat, list(d), wk), list(d), wk)
    got = out[dst_shift:dst_shift + n].cpu().numpy()
    assert np.abs(got - ref).max() <= 1e-6 * np.abs(ref).max()
    np.testing.assert_array_equal(got, host.numpy())
    assert out[dst_shift + n].item() == 7.0 and (dst_shift == 0 or out[0].item() == 7.0)
    assert P.oscars_check_padding(ctx.handle) == 0
    ctx.close()
