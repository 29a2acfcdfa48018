"""What no run of a kernel can show: rules that its source has to keep."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1708_01609_gb300", "csrc")


def _kernels():
    """(file:name, body) of every __global__ function."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\(.*?\)\s*)?(\w+)\(", text,
                             re.S):
            begin = text.index("{", m.end())
            depth, end = 0, begin
            while True:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
                if depth == 0:
                    break
            yield f"{os.path.basename(path)}:{m.group(1)}", text[begin:end]


REMOTE = re.compile(r"\*\s*cluster\.map_shared_rank\(")
REMOTE_KERNELS = [(n, b) for n, b in _kernels() if REMOTE.search(b)]


def test_the_kernels_with_remote_accesses_are_found():
    names = {n.split(":")[1] for n, _ in REMOTE_KERNELS}
    assert {"unit_kernel", "unit_exchange_kernel", "correlate_multi_kernel", "batch_kernel"} <= names


@pytest.mark.parametrize("name,body", REMOTE_KERNELS, ids=[n for n, _ in REMOTE_KERNELS])
def test_cluster_has_started_before_a_remote_access(name, body):
    """Distributed shared memory may be accessed only when every CTA of the
    cluster has started, which a barrier of the cluster shows."""
    before = body[:REMOTE.search(body).start()]
    assert re.search(r"\bcluster_arrive(_relaxed)?\(\)|\bcluster\.sync\(\)", before), name
