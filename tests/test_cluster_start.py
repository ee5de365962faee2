"""A CTA of a cluster may touch another's shared memory only once it is known that the other has started, that is behind a
cluster barrier.  Nothing shows a missing one at run time (the other CTA has practically always started), so the sources are read."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1910_06188_b200", "csrc")
REMOTE = re.compile(r"\b(?:ld|st|red|atom)\.shared::cluster|mbar_arrive_cluster\w*\(")
MET = re.compile(r"cluster_sync_all\(\)|cluster_wait\(\)|barrier\.cluster\.wait")


def _kernels():
    for name in sorted(os.listdir(CSRC)):
        if name.endswith(".cu"):
            with open(os.path.join(CSRC, name)) as f:
                text = re.sub(r"//[^\n]*", "", f.read())
            for part in re.split(r"\b__global__\b", text)[1:]:
                body = part.split("\n}\n", 1)[0]  # a kernel ends at the first brace in the first column
                if REMOTE.search(body):
                    yield pytest.param(body, id=name + ":" + re.search(r"(\w+)\s*\(const", body).group(1))


KERNELS = list(_kernels())


def test_the_kernels_with_remote_accesses_are_found():
    assert len(KERNELS) >= 4


@pytest.mark.parametrize("body", KERNELS)
def test_remote_shared_memory_is_touched_behind_a_cluster_barrier(body):
    met = MET.search(body)
    assert met is not None and met.start() < REMOTE.search(body).start()
