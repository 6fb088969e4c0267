"""A block of a cluster may touch another's shared memory only behind a
cluster barrier that follows the kernel's start (until then the other block
need not have started).  Read from the sources: no kernel with cluster
dimensions reaches map_shared_rank, in itself or in the function it calls,
before such a barrier."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2302_09883_gb300", "csrc")


def _body(text, at):
    """The braced block that opens first behind `at`."""
    i = text.index("{", text.index(")", at))
    depth = 0
    for j in range(i, len(text)):
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return text[i:j]
    raise AssertionError("unbalanced braces")


def _code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


@pytest.mark.parametrize("name,kernel,calls", [("patch2d.cuh", "patch_kernel_cluster(PatchArgs", "patch_body"),
                                               ("mlp.cu", "mlp_train_cluster(float*", None)])
def test_a_barrier_comes_before_the_first_remote_access(name, kernel, calls):
    text = _code(name)
    body = _body(text, text.index(kernel))
    if calls:  # what the kernel calls, in its place
        callee = _body(text, re.search(r"void " + calls + r"\(", text).start())
        body = body[:body.index(calls)] + callee
    barrier = re.search(r"\.sync\(\)|\.barrier_wait\(\)", body)
    remote = re.search(r"map_shared_rank", body)
    assert remote is not None and barrier is not None
    assert barrier.start() < remote.start()


def test_every_cluster_kernel_is_covered():
    found = [f for f in sorted(os.listdir(CSRC)) for _ in re.findall(r"__cluster_dims__\(", _code(f))]
    assert found == ["mlp.cu", "patch2d.cuh"]
