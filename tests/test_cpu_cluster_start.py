"""Shared memory of another CTA of a cluster may be touched only once that CTA runs: in every kernel that
is launched on clusters a barrier of the whole cluster comes before the first remote store.  A missing one
shows on the GPU only as a rare race, so the order is read from the source."""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1910_12007_gb300", "csrc")
REMOTE_STORE = re.compile(r"\bput_all\(|st\.shared::cluster")
# the barrier itself, or on clusters only
BARRIER = re.compile(r"^\s*(if \(C > 1\) )?run_sync\(C\);", re.M)


def _kernel_body(text, name):
    """The braces' content of a __global__ function, without comments."""
    text = re.sub(r"//[^\n]*", "", text)
    at = text.index("{", text.index(name, text.index("__global__", text.index(name) - 200)))
    depth = 0
    for k in range(at, len(text)):
        depth += {"{": 1, "}": -1}.get(text[k], 0)
        if depth == 0:
            return text[at:k]
    raise AssertionError("unbalanced braces")


@pytest.mark.parametrize("file,kernel", [("forward.cu", "forward_kernel(FwdArgs"),
                                         ("forward64.cu", "forward64_kernel(FwdArgs")])
def test_cluster_barrier_before_the_first_remote_store(file, kernel):
    with open(os.path.join(SRC, file)) as f:
        body = _kernel_body(f.read(), kernel)
    store = REMOTE_STORE.search(body)
    assert store is not None
    barrier = BARRIER.search(body)
    assert barrier is not None and barrier.start() < store.start()
    # and none after the last barrier: a CTA stays until the others have written to it
    last = [m.start() for m in BARRIER.finditer(body)][-1]
    assert all(m.start() < last for m in REMOTE_STORE.finditer(body))


def test_run_sync_is_a_barrier_of_the_cluster():
    with open(os.path.join(SRC, "forward_args.cuh")) as f:
        text = f.read()
    body = text[text.index("void run_sync(int C)"):]
    assert body.index("barrier.cluster.arrive.release") < body.index("barrier.cluster.wait.acquire")
