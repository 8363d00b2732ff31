"""Cluster kernels touch another CTA's shared memory only after a barrier that every CTA of the
cluster has reached: before it a CTA need not have started, and its shared memory must not be
accessed.  What goes wrong otherwise is a race on the GPU, so the sources are read instead:
in every kernel that maps shared memory of another CTA, the first mapping comes after a
cluster barrier."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1212_0262_gb300", "csrc")
BARRIER = re.compile(r"cluster\.(sync|barrier_wait)\(\)")


def kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for part in text.split("__global__")[1:]:
            body = part[: part.index("\n}")]
            if "map_shared_rank" in body:
                yield pytest.param(body, id=re.search(r"(\w+_kernel)\(", body).group(1))


@pytest.mark.parametrize("body", list(kernels()))
def test_remote_shared_memory_only_after_a_cluster_barrier(body):
    first = BARRIER.search(body)
    assert first and first.start() < body.index("map_shared_rank")


def test_the_cluster_kernels_are_found():
    assert {p.id for p in kernels()} == {"hmf_run_fp64_kernel", "hmf_run_mixed_kernel"}
