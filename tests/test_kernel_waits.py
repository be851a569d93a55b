"""The waits that the kernels' sources have to hold, read from the sources (a
missing one shows only as a fault or a hang, and only now and then, on a GPU).

* A CTA's shared memory may be touched by a peer of its cluster only once that
  CTA is known to run: in every kernel a cluster barrier's wait comes before
  the first remote load, store or arrival."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2102_08550_gb300", "csrc")
# operations of this repository on another CTA's shared memory
REMOTE = ("st_dsmem_f32x4", "st_dsmem_f64", "ld_dsmem_f32", "ld_dsmem_f32x4", "st_async_v4", "bulk_copy_to_peer",
          "mbar_arrive_at", "umma_commit_pair", "tma_load_3d_pair")


def _clean(text):
    text = re.sub(r"//[^\n]*", "", text)
    return re.sub(r"/\*.*?\*/", "", text, flags=re.S)


def _block(text, at):
    """The brace-matched block that opens at or after `at`."""
    i = text.index("{", at)
    depth = 0
    for j in range(i, len(text)):
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return text[i:j + 1]
    raise ValueError("unbalanced braces")


def _functions(text):
    """name -> (is a kernel, body) of the device functions of a cleaned source."""
    out = {}
    for m in re.finditer(r"(__global__ void(?: __launch_bounds__\((?:[^()]|\([^()]*\))*\))?|__device__ __forceinline__ [\w ]+?)\s+"
                         r"(\w+)\(", text):
        body_at = text.index("{", m.end())
        if text.find(";", m.end()) < body_at and ")" in text[m.end():text.find(";", m.end())]:
            continue   # a declaration
        out[m.group(2)] = (m.group(1).startswith("__global__"), _block(text, body_at))
    return out


def _calls(body, names):
    return sorted(m.start() for n in names for m in re.finditer(r"\b%s(?:<[^;(]*>)?\(" % n, body))


def first_remote_access_without_start(text):
    """Kernels of a source whose first access to a peer's shared memory no cluster wait precedes."""
    fns = _functions(_clean(text))
    remote = set(REMOTE)
    helpers = {n for n, (k, b) in fns.items() if not k and n not in remote and _calls(b, remote)}
    bad = []
    for name, (kernel, body) in fns.items():
        if not kernel:
            continue
        touch, wait = _calls(body, remote | helpers), _calls(body, ("cluster_sync", "cluster_wait"))
        if touch and (not wait or wait[0] > touch[0]):
            bad.append(name)
    return bad


def _sources():
    return sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))


def _read(f):
    with open(os.path.join(CSRC, f)) as h:
        return h.read()


@pytest.mark.parametrize("f", _sources())
def test_peers_have_started_before_their_memory_is_touched(f):
    assert first_remote_access_without_start(_read(f)) == []


def test_the_cluster_kernels_are_found():
    found = {f for f in _sources() for k, b in _functions(_clean(_read(f))).values() if k and _calls(b, REMOTE)}
    assert {"fused_round.cu", "gemm_rows.cu", "gemm_tc.cu", "mlp.cu", "softreg.cu"} <= found


def test_a_missing_start_barrier_is_caught():
    kernel = "__global__ void __launch_bounds__(32) k(int* p) {\n %s st_dsmem_f32x4(p, 1, v);\n cluster_sync();\n}\n"
    assert first_remote_access_without_start(kernel % "") == ["k"]
    assert first_remote_access_without_start(kernel % "cluster_arrive(); cluster_wait();") == []
    assert first_remote_access_without_start(kernel % "// cluster_wait();\n") == ["k"]
