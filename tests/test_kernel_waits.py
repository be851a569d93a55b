"""The waits that the kernels' sources have to hold, read from the sources (a
missing one shows only as a fault or a hang, and only now and then, on a GPU).

* A CTA's shared memory may be touched by a peer of its cluster only once that
  CTA is known to run: in every kernel a cluster barrier's wait comes before
  the first remote load, store or arrival.
* A warp that runs a loop together and elects a lane to issue (elect.sync with a
  full mask) must stay together: such a loop is not left on a wait, which may run
  out in some lanes and not in the others.

Beside them, what a launch must not set by its own size."""
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


def _loops(body):
    """(start, end) of the braced for loops of a function body."""
    out = []
    for m in re.finditer(r"\bfor \(", body):
        depth, i = 0, m.end() - 1
        while True:
            depth += {"(": 1, ")": -1}.get(body[i], 0)
            i += 1
            if depth == 0:
                break
        if body[i:].lstrip().startswith("{"):
            at = body.index("{", i)
            out.append((at, at + len(_block(body, at))))
    return out


def lanes_that_leave_alone(text):
    """Kernels with a loop that elects an issuer and ends on a wait that each lane decides for itself."""
    bad = []
    for name, (kernel, body) in _functions(_clean(text)).items():
        if not kernel:
            continue
        loops = _loops(body)
        for m in re.finditer(r"if \([^;{}]*\bmbar_wait\([^;{}]*break;", body):
            lo, hi = max(l for l in loops if l[0] < m.start() < l[1])
            if _calls(body[lo:hi], ("elect_one",)):
                bad.append(name)
        for lo, hi in loops:
            head = body[body.rindex("for (", 0, lo):lo]
            if re.search(r"\bok\b", head) and _calls(body[lo:hi], ("elect_one",)):
                bad.append(name)
    return bad


@pytest.mark.parametrize("f", _sources())
def test_issuing_warps_leave_their_loops_together(f):
    assert lanes_that_leave_alone(_read(f)) == []


def test_a_lane_wise_wait_is_caught():
    kernel = "__global__ void __launch_bounds__(32) k(int* p) {\n for (int i = 0; %si < 4; ++i) {\n %s;\n if (elect_one() && limit > 1) { go(); }\n }\n}\n"
    assert lanes_that_leave_alone(kernel % ("", "if (!(ok = mbar_wait(b, i))) break")) == ["k"]
    assert lanes_that_leave_alone(kernel % ("ok && ", "ok = mbar_wait(b, i)")) == ["k"]
    assert lanes_that_leave_alone(kernel % ("", "mbar_wait_keep(limit, b, i)")) == []


def test_shared_memory_limits_do_not_depend_on_a_launch():
    """The limit on dynamic shared memory is the kernel's, in the whole process: a launch that set it to its
    own size could lower it under another thread's.  It is set in one place, to one value."""
    sets = {f: len(re.findall(r"cudaFuncAttributeMaxDynamicSharedMemorySize", _clean(_read(f))))
            for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".h", ".cuh"))}
    assert {f for f, n in sets.items() if n} == {"internal.h"} and sets["internal.h"] == 1
