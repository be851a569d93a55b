"""Calls from host threads: one that has made no CUDA call before, and several at
once that launch the same kernels with different sizes (the shared-memory limit
belongs to a kernel, not to a launch)."""
import threading

import pytest
import torch

import paper_2102_08550_gb300 as P

pytestmark = pytest.mark.gpu


def _run_together(jobs):
    errors, go = [], threading.Barrier(len(jobs))

    def work(job):
        try:
            go.wait()
            job()
        except Exception as e:   # noqa: BLE001 (the main thread raises it)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    if errors:
        raise errors[0]


def test_product_is_a_threads_first_cuda_call(cuda_device):
    A, B = torch.eye(128, device=cuda_device).to(torch.bfloat16), torch.eye(128, device=cuda_device).to(torch.bfloat16)
    C = torch.empty(128, 128, device=cuda_device)
    torch.cuda.synchronize()
    for _ in range(2):
        C.fill_(7.0)
        torch.cuda.synchronize()
        _run_together([lambda: P.oscars_gemm_bf16_nt(A.data_ptr(), B.data_ptr(), C.data_ptr(), 128, 128, 128)])
        assert torch.equal(C, torch.eye(128, device=cuda_device))


def test_products_of_several_threads(cuda_device):
    """fp32 accumulation of at most 3072 products: 1e-5 of the largest value, as in the other GEMM cases."""
    state = []
    for M, N, K in [(128, 2048, 512), (128, 96, 64), (128, 224, 3072), (128, 32, 8)]:
        g = torch.Generator(device="cuda").manual_seed(M + N + K)
        A = torch.randn(M, K, generator=g, device=cuda_device).to(torch.bfloat16)
        B = torch.randn(N, K, generator=g, device=cuda_device).to(torch.bfloat16)
        state.append((A, B, torch.full((M, N), float("nan"), device=cuda_device), torch.cuda.Stream()))
    torch.cuda.synchronize()

    def job(A, B, C, s):
        def run():
            for _ in range(8000):
                P.oscars_gemm_bf16_nt(A.data_ptr(), B.data_ptr(), C.data_ptr(), A.shape[0], B.shape[0], A.shape[1],
                                      s.cuda_stream)
        return run

    _run_together([job(*s) for s in state])
    for A, B, C, _ in state:
        ref = A.double() @ B.double().T
        assert (C.double() - ref).abs().max().item() <= 1e-5 * ref.abs().max().item() + 1e-6


def test_steps_of_several_threads(cuda_device):
    """Each call repeats what it gives alone, bit for bit."""
    state = []
    for D, C, B in [(784, 10, 32), (500, 9, 100), (333, 10, 8), (60, 32, 256)]:
        g = torch.Generator(device="cuda").manual_seed(D)
        x = torch.randn(300, D, generator=g, device=cuda_device)
        y = torch.randint(0, C, (300,), generator=g, device=cuda_device).to(torch.int32)
        p = torch.randn(C * D + C, generator=g, device=cuda_device) * 0.01
        state.append((D, C, B, x, y, p, torch.empty_like(p), torch.empty(1, device=cuda_device), torch.cuda.Stream()))

    def call(D, C, B, x, y, p, out, loss, s):
        P.oscars_softreg_steps_noalloc(p.data_ptr(), out.data_ptr(), x.data_ptr(), y.data_ptr(), 300, 0, 2, D, C, B, 0.05,
                                       loss.data_ptr(), s.cuda_stream)

    torch.cuda.synchronize()
    for s in state:
        call(*s)
    torch.cuda.synchronize()
    alone = [(s[6].clone(), s[7].clone()) for s in state]
    _run_together([lambda s=s: [call(*s) for _ in range(400)] for s in state])
    for s, (out, loss) in zip(state, alone):
        assert torch.equal(s[6], out) and torch.equal(s[7], loss)
