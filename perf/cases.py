"""The work that a program built on this library has it do, as timed cases.

Each case goes through the library's public entry points (the Python binding
``paper_2102_08550_gb300``, one call per C entry point):

* ``round``: one round of the method: local steps of every worker, the
  asynchronous read of the workers' losses, the server merge of the pushed
  replicas, and the pull of the merged model into the caller's buffer;
* ``train``: several rounds in one ``oscars_train`` call, the shards in pinned
  host memory (the training set does not fit the device, or is refilled by a
  loader), then the pull of the final model;
* ``eval``: the loss of the global model on a held-out set (the forward-only
  direction; what a time-to-loss run does between rounds);
* ``push``: the server merge of deltas that remote workers pushed into caller
  buffers, and the pull of the result;
* ``merge``: the same update on plain buffers, without a context;
* ``steps``: the allocation-free local steps of one softmax-regression worker;
* ``gemm``: the bf16 contraction of a dense layer.

Models and sizes are the repository's workloads (softmax regression 784 -> 10
with 4 workers, the 784-512-10 and 3072-1024-1024-10 MLPs, the CIFAR-shaped
residual network, the 25.6 M-parameter merge of 64 workers) and generic odd
ones.  The data is a Gaussian mixture: class means and unit noise.
"""
from __future__ import annotations

import ctypes
import functools
import math
import random

import numpy as np
import torch

import paper_2102_08550_gb300 as lib

DEV = "cuda"


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # one edge worker's eight local steps of softmax regression, for callers
        # that cannot allocate (the smallest call: a serial chain of tiny steps)
        {"name": "steps-softreg-784x10-b32", "kind": "steps", "dims": "784-10", "batch": 32, "tau": 8, "n": 4096},
        # a round of the smallest workload: four workers, speeds 1 1 2 4
        {"name": "round-softreg-784x10-w4", "kind": "round", "model": "softreg", "dims": "784-10", "workers": 4,
         "batch": 32, "M": 8, "speeds": "1 1 2 4", "n": 4096},
        # the same path away from its tuned size: odd input width, more classes
        # and rows than threads expect, a worker count that fills the GPU unevenly
        {"name": "round-softreg-333x26-w12", "kind": "round", "model": "softreg", "dims": "333-26", "workers": 12,
         "batch": 100, "M": 16, "speed_seed": 5, "n": 1500},
        # the headline workload: 16 workers, 784-512-10, batch 64
        {"name": "round-mlp-784-512-10-w16", "kind": "round", "model": "mlp", "dims": "784-512-10", "workers": 16,
         "batch": 64, "M": 16, "speed_seed": 1, "n": 16384},
        # the same model trained from shards in pinned host memory, eight rounds a call
        {"name": "train-host-784-512-10-w16", "kind": "train", "model": "mlp", "dims": "784-512-10", "workers": 16,
         "batch": 64, "M": 16, "speed_seed": 1, "n": 2048, "rounds": 8, "host": True},
        # a small odd MLP: ragged input, three layers, 17 classes, five workers
        {"name": "round-mlp-1000-384-256-17-w5", "kind": "round", "model": "mlp", "dims": "1000-384-256-17",
         "workers": 5, "batch": 32, "M": 16, "speed_seed": 3, "n": 2048},
        # the large MLP workload: CIFAR-sized inputs, 32 workers, batch 128
        {"name": "round-mlp-3072-1024-1024-10-w32", "kind": "round", "model": "mlp", "dims": "3072-1024-1024-10",
         "workers": 32, "batch": 128, "M": 16, "speed_seed": 1, "n": 8192, "clip": 3.0},
        # the convolutional workload: residual network on 32 x 32 x 3 images
        {"name": "round-cnn-c64-w16", "kind": "round", "model": "cnn", "cin": 3, "blocks": 1, "classes": 10,
         "workers": 16, "batch": 32, "M": 16, "speed_seed": 1, "n": 2048, "clip": 3.0},
        # the held-out loss between rounds: 8192 samples
        {"name": "eval-mlp-784-512-10-n8192", "kind": "eval", "model": "mlp", "dims": "784-512-10", "workers": 16,
         "batch": 64, "eval_n": 8192},
        # the server merge of a ResNet-50-sized model pushed by 64 workers
        {"name": "merge-25.6M-w64", "kind": "merge", "P": 25_600_000, "workers": 64, "shift": 0},
        # remote workers push deltas of the headline model
        {"name": "push-784-512-10-w16", "kind": "push", "dims": "784-512-10", "workers": 16, "batch": 64},
        # the first layer of the large MLP over a whole held-out set
        {"name": "gemm-1024x8192x3072", "kind": "gemm", "M": 1024, "N": 8192, "K": 3072},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw_model(rng):
    """A model and its batch, within what oscars_create takes."""
    model = rng.choice(["softreg", "mlp", "mlp", "mlp", "cnn"])
    if model == "softreg":
        classes = rng.randint(2, 32)
        batch = _log_int(rng, 1, 256)
        dim = _log_int(rng, 16, 1500)
        while dim * (classes + batch) + batch * (classes + 4) + 64 > 54000:   # weights and one batch in shared memory
            batch = max(1, batch * 3 // 4)
            dim = max(16, dim * 7 // 8)
        return {"model": model, "dims": "%d-%d" % (dim, classes), "batch": batch}
    if model == "cnn":
        return {"model": model, "cin": rng.choice([1, 3, 3, 4, 7, 16]), "blocks": rng.choice([1, 1, 2]),
                "classes": rng.randint(2, 32), "batch": 16 * rng.randint(1, 4)}
    hidden = [128 * _log_int(rng, 1, 8) for _ in range(rng.choice([1, 1, 2]))]
    classes = rng.choice([10, 10, rng.randint(2, 32)])
    dims = [8 * _log_int(rng, 8, 384)] + hidden + [classes]
    return {"model": model, "dims": "-".join(map(str, dims)), "batch": rng.choice([32, 64, 64, 128, 256])}


def draw(rng):
    """One more case of the same ranges, no more work than the listed network's round."""
    largest = max(_cost(c) for c in listed())
    while True:
        case = _draw(rng)
        if _cost(case) <= largest:
            return case


def _cost(case):
    w = work(case)
    return max(w["bytes"], w["flops"] / 50)


def _draw(rng):
    kind = rng.choice(["steps", "round", "round", "round", "train", "eval", "push", "merge", "gemm"])
    if kind == "steps":
        while True:
            m = _draw_model(rng)
            if m["model"] == "softreg":
                return {"kind": kind, "dims": m["dims"], "batch": min(128, m["batch"]), "tau": _log_int(rng, 1, 32),
                        "n": rng.randint(200, 4096)}
    if kind == "gemm":
        return {"kind": kind, "M": 128 * _log_int(rng, 1, 32), "N": _log_int(rng, 1, 8192), "K": 8 * _log_int(rng, 4, 384)}
    if kind == "merge":
        w = _log_int(rng, 1, 64)
        return {"kind": kind, "P": _log_int(rng, 1000, 25_600_000), "workers": w, "shift": rng.choice([0, 0, 1, 2, 3])}
    if kind == "push":
        while True:
            m = _draw_model(rng)
            if m["model"] == "mlp":
                return {"kind": kind, "dims": m["dims"], "workers": rng.randint(1, 32), "batch": m["batch"]}
    m = _draw_model(rng)
    m["kind"] = kind
    w = rng.randint(2, 32)
    if m["model"] == "cnn":   # no more images a step than the listed network has
        w = max(2, min(16, 512 // (m["batch"] * m["blocks"])))
        w = rng.randint(2, w)
        m["clip"] = 3.0
    m["workers"] = w
    if kind == "eval":
        n = _log_int(rng, 256, 8192 if m["model"] != "cnn" else 1024)
        m["eval_n"] = max(1, n // m["batch"]) * m["batch"] if m["model"] == "mlp" else n
        return m
    m["M"] = rng.choice([4, 8, 16])
    m["speed_seed"] = rng.randint(1, 1000)
    m["n"] = rng.randint(max(m["batch"], 300), 2048 if m["model"] != "cnn" else 600)
    if kind == "train":
        m["rounds"] = 1 if m["model"] == "cnn" else 2 if m["dims"].count("-") == 3 or m["batch"] > 64 else rng.randint(2, 8)
        m["host"] = m["model"] == "mlp" and rng.random() < 0.5
        m["workers"] = min(w, 16)
    return m


# ------------------------------------------------------------------ sizes
def _dims(case):
    return [int(v) for v in case["dims"].split("-")]


def _classes(case):
    return case["classes"] if case.get("model") == "cnn" else _dims(case)[-1]


def _in_dim(case):
    return 32 * 32 * case["cin"] if case.get("model") == "cnn" else _dims(case)[0]


def _shapes(case):
    """Parameter tensors in the canonical order of the flat vector."""
    if case.get("model") == "cnn":
        s = [(64, 3, 3, case["cin"]), (64,)]
        for _ in range(2 * case["blocks"]):
            s += [(64, 3, 3, 64), (64,)]
        return s + [(case["classes"], 64), (case["classes"],)]
    d = _dims(case)
    return [t for i, o in zip(d[:-1], d[1:]) for t in ((o, i), (o,))]


def _num_params(case):
    return sum(int(np.prod(s)) for s in _shapes(case))


def _ticks(case):
    """Iteration times of the workers: fixed speeds or lognormal ones."""
    if "speeds" in case:
        sp = [float(v) for v in case["speeds"].split()]
    elif "speed_seed" in case:
        sp = np.random.default_rng(case["speed_seed"]).lognormal(0.0, 0.5, case["workers"]).tolist()
    else:
        sp = [1.0] * case["workers"]
    return lib.oscars_iteration_ticks(sp)


@functools.lru_cache(maxsize=64)
def _tau(key):
    case = dict(key)
    return lib.oscars_schedule_solve(_ticks(case), case["M"])[2]


def _local_steps(case):
    return _tau(tuple(sorted((k, case[k]) for k in ("speeds", "speed_seed", "workers", "M") if k in case)))


def _flops_per_sample(case):
    """Forward, weight gradient, and the input gradients that are needed."""
    if case.get("model") == "cnn":
        px = 1024
        stem, conv = 2 * px * 64 * 9 * case["cin"], 2 * px * 64 * 9 * 64
        return 2 * stem + 3 * 2 * case["blocks"] * conv + 6 * 64 * case["classes"]
    d = _dims(case)
    return sum(2 * i * o * (2 if l == 0 else 3) for l, (i, o) in enumerate(zip(d[:-1], d[1:])))


def work(case):
    k = case["kind"]
    if k == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 2 * (M + N) * K + 4 * M * N, "flops": 2 * M * N * K}
    if k == "merge":
        return {"bytes": 4 * case["P"] * (case["workers"] + 2), "flops": 2 * case["P"] * case["workers"]}
    P = _num_params(case)
    if k == "push":   # deltas in, the model in and out, the pulled copy
        return {"bytes": 4 * P * (case["workers"] + 3), "flops": 2 * P * case["workers"]}
    row = 4 * _in_dim(case) + 4
    if k == "steps":
        s = case["tau"] * case["batch"]
        return {"bytes": s * row + 8 * P, "flops": s * _flops_per_sample(case)}
    if k == "eval":
        fwd = _flops_per_sample(case) / (2 if case["model"] == "softreg" else 3)
        return {"bytes": case["eval_n"] * row + 4 * P, "flops": case["eval_n"] * fwd}
    # a round reads its mini-batches and the global model once, and writes the
    # replicas, the merged model and the pulled copy once
    samples, rounds = sum(_local_steps(case)) * case["batch"], case.get("rounds", 1)
    by = samples * row + 4 * P * (1 + case["workers"] + 1)
    return {"bytes": rounds * by + 4 * P, "flops": rounds * samples * _flops_per_sample(case)}


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _data(case, g, means, n):
    y = torch.randint(0, means.shape[0], (n,), device=DEV, generator=g)
    x = torch.randn(n, means.shape[1], device=DEV, generator=g)
    x += means[y]
    if case.get("clip"):
        x.clamp_(-case["clip"], case["clip"])
    return x, y.to(torch.int32)


def _init(case, g):
    """W ~ U(+-1/sqrt(fan_in)), biases 0, as one flat vector."""
    parts = []
    for s in _shapes(case):
        n = int(np.prod(s))
        if len(s) == 1:
            parts.append(torch.zeros(n, device=DEV))
        else:
            lim = 1.0 / math.sqrt(n // s[0])
            parts.append((torch.rand(n, device=DEV, generator=g) * 2 - 1) * lim)
    return torch.cat(parts)


def _inputs(case, seed):
    """Shards (or the evaluation set) and the initial model, from the seed alone."""
    g = _gen(seed)
    means = torch.randn(_classes(case), _in_dim(case), device=DEV, generator=g)
    if case["kind"] == "eval":
        return _data(case, g, means, case["eval_n"]), _init(case, g)
    if case["kind"] == "steps":
        return _data(case, g, means, case["n"]), _init(case, g)
    return [_data(case, g, means, case["n"]) for _ in range(case["workers"])], _init(case, g)


def _context(case, shards, init):
    kw = dict(num_workers=case["workers"], batch=case["batch"], lr=0.05, shards=shards, init_params=init,
              t_ticks=_ticks(case), M=case.get("M", 8))
    if case.get("model") == "cnn":
        return lib.OscarsContext(model=lib.MODEL_CNN, dims=[32, 32, case["cin"], 64, case["classes"]],
                                 blocks=case["blocks"], **kw)
    return lib.OscarsContext(dims=_dims(case), bf16=case.get("model", "mlp") == "mlp", **kw)


def _deltas(case, g, P):
    """Pushed deltas of sd 1e-3, `shift` floats past a 16-byte boundary."""
    sh = case.get("shift", 0)
    out = []
    for _ in range(case["workers"]):
        d = torch.randn(P + sh, device=DEV, generator=g)
        d *= 1e-3
        out.append(d[sh:])
    return out


def prepare(case, seed):
    k = case["kind"]
    if k == "gemm":
        g = _gen(seed)
        a = torch.randn(case["M"], case["K"], device=DEV, generator=g).to(torch.bfloat16)
        b = torch.randn(case["N"], case["K"], device=DEV, generator=g).to(torch.bfloat16)
        return {"case": case, "a": a, "b": b, "c": torch.empty(case["M"], case["N"], device=DEV)}
    if k == "merge":
        g = _gen(seed)
        sh = case["shift"]
        xg = torch.rand(case["P"] + sh, device=DEV, generator=g) * 0.1 - 0.05
        d = _deltas(case, g, case["P"])
        w = [1.0 / case["workers"]] * case["workers"]
        return {"case": case, "xg": xg[sh:], "deltas": d, "ptrs": [t.data_ptr() for t in d], "w": w}
    P = _num_params(case)
    if k == "push":
        g = _gen(seed)
        init = _init(case, g)
        d = _deltas(case, g, P)
        # the context needs a shard per worker even when only remote deltas come in
        x, y = torch.zeros(case["batch"], _in_dim(case), device=DEV), torch.zeros(case["batch"], dtype=torch.int32, device=DEV)
        ctx = _context(case, [(x, y)] * case["workers"], init)
        return {"case": case, "ctx": ctx, "deltas": d, "model": torch.empty(P, device=DEV)}
    data, init = _inputs(case, seed)
    if k == "steps":
        return {"case": case, "x": data[0], "y": data[1], "p": init, "out": torch.empty(P, device=DEV),
                "loss": torch.empty(1, device=DEV)}
    if k == "eval":
        x, y = data
        ctx = _context(case, [(x, y)] * case["workers"], init)
        return {"case": case, "ctx": ctx, "x": x, "y": y}
    if case.get("host"):
        data = [(x.cpu().pin_memory(), y.cpu().pin_memory()) for x, y in data]
    return {"case": case, "ctx": _context(case, data, init), "model": torch.empty(P, device=DEV),
            "losses": torch.empty(case["workers"], device=DEV)}


# ------------------------------------------------------------------ one pass
def run(state):
    case = state["case"]
    k = case["kind"]
    if k == "gemm":
        lib.oscars_gemm_bf16_nt(state["a"].data_ptr(), state["b"].data_ptr(), state["c"].data_ptr(), case["M"], case["N"],
                                case["K"])
        return state["c"]
    if k == "merge":
        lib.oscars_merge(state["xg"].data_ptr(), state["ptrs"], state["w"], case["P"])
        return state["xg"]
    if k == "steps":
        d = _dims(case)
        lib.oscars_softreg_steps_noalloc(state["p"].data_ptr(), state["out"].data_ptr(), state["x"].data_ptr(),
                                         state["y"].data_ptr(), case["n"], 0, case["tau"], d[0], d[1], case["batch"], 0.05,
                                         state["loss"].data_ptr())
        return {"params": state["out"], "loss": state["loss"]}
    ctx = state["ctx"]
    if k == "eval":
        return {"loss": ctx.eval_loss(state["x"], state["y"])}
    if k == "push":
        ctx.push_merge(state["deltas"])
        ctx.pull(state["model"])
        return state["model"]
    if k == "train":
        log = ctx.train(case["rounds"])
        ctx.pull(state["model"])
        return {"model": state["model"], "losses": [r["worker_loss"] for r in log]}
    ctx.local_steps(want_loss=False)
    ctx.losses_async(state["losses"])
    ctx.push_merge()
    ctx.pull(state["model"])
    return {"model": state["model"], "losses": state["losses"]}


# ------------------------------------------------------------------ what is right
def tolerance(case):
    """About four times what the path differed by from another correct
    implementation: the 64-bit result for the 32-bit paths, the per-layer
    kernels or the bf16-emulating oracle (three passes) for the bf16 ones,
    where a flipped rounding or ReLU mask travels through the later steps."""
    k = case["kind"]
    if k == "gemm":
        return {"rel": 1.3e-5}       # 3.2e-6: fp32 accumulation of K = 3072 products
    if k in ("merge", "push"):
        return {"rel": 1e-6}         # 2.6e-8 after one merge; the passes add up
    if k == "steps" or case.get("model") == "softreg":
        return {"rel": 1e-5}         # 1e-7 after one round
    if k == "eval":
        return {"rel": 1e-4}         # one forward pass, the mean over all samples
    # model 2.6e-4 (three-layer MLP, batch 32) and losses 4e-5 after two rounds,
    # more for the longer schedules that are drawn
    return {"rel": 2e-3}


def _split(flat, shapes):
    out, off = [], 0
    for s in shapes:
        n = int(np.prod(s))
        out.append(flat[off:off + n].reshape(s))
        off += n
    return out


def _conv(x, w, b):
    """3x3, stride 1, zero padding 1; x [n, 32, 32, c], w [o, 3, 3, c]."""
    n, _, _, c = x.shape
    p = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1))
    cols = torch.stack([p[:, dy:dy + 32, dx:dx + 32] for dy in range(3) for dx in range(3)], dim=3)
    return (cols.reshape(n * 1024, 9 * c) @ w.reshape(w.shape[0], 9 * c).t() + b).reshape(n, 32, 32, -1)


def _logits(case, params, x):
    if case.get("model") == "cnn":
        h = torch.relu(_conv(x.reshape(-1, 32, 32, case["cin"]), params[0], params[1]))
        for i in range(case["blocks"]):
            wa, ba, wb, bb = params[2 + 4 * i:6 + 4 * i]
            h = torch.relu(_conv(torch.relu(_conv(h, wa, ba)), wb, bb) + h)
        return h.mean(dim=(1, 2)) @ params[-2].t() + params[-1]
    for i in range(0, len(params), 2):
        x = x @ params[i].t() + params[i + 1]
        if i + 2 < len(params):
            x = torch.relu(x)
    return x


def _local(case, flat, x, y, cursor, tau):
    """tau SGD steps from `flat` on successive mini-batches; the mean loss."""
    shapes, B = _shapes(case), case["batch"]
    p, total = flat, 0.0
    for s in range(tau):
        rows = (cursor + s * B + torch.arange(B, device=DEV)) % x.shape[0]
        q = p.detach().requires_grad_(True)
        loss = torch.nn.functional.cross_entropy(_logits(case, _split(q, shapes), x[rows].double()), y[rows].long())
        (grad,) = torch.autograd.grad(loss, q)
        p = q.detach() - 0.05 * grad
        total += loss.item()
    return p, total / tau


def exact(case, seed):
    k = case["kind"]
    if k in ("gemm", "merge", "push"):
        s = prepare(case, seed) if k != "push" else None
        if k == "gemm":
            return s["a"].double() @ s["b"].double().t()
        if k == "merge":
            xg = s["xg"].double()
            for d, w in zip(s["deltas"], s["w"]):
                xg += ctypes.c_float(w).value * d.double()
            return xg
        g = _gen(seed)
        xg = _init(case, g).double()
        for d in _deltas(case, g, _num_params(case)):
            xg += d.double() / case["workers"]
        return xg
    data, init = _inputs(case, seed)
    g = init.double()
    if k == "steps":
        p, loss = _local(case, g, data[0], data[1], 0, case["tau"])
        return {"params": p, "loss": torch.tensor([loss], dtype=torch.float64)}
    if k == "eval":
        total = 0.0
        for i in range(0, case["eval_n"], 256):
            z = _logits(case, _split(g, _shapes(case)), data[0][i:i + 256].double())
            total += torch.nn.functional.cross_entropy(z, data[1][i:i + 256].long(), reduction="sum").item()
        return {"loss": total / case["eval_n"]}
    tau, B, means = _local_steps(case), case["batch"], []
    for r in range(case.get("rounds", 1)):
        acc, losses = torch.zeros_like(g), []
        for i, (x, y) in enumerate(data):
            p, loss = _local(case, g, x, y, r * tau[i] * B, tau[i])
            acc += p
            losses.append(loss)
        g = acc / case["workers"]
        means.append(sum(losses) / len(losses))
    if k == "train":
        return {"model": g, "losses": means}
    return {"model": g, "losses": torch.tensor(losses, dtype=torch.float64)}
