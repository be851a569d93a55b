"""Calls from host threads: one that has made no CUDA call before."""
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
