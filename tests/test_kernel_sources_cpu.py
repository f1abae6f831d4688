"""Rules that the kernel sources keep and no run on a GPU can show reliably."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2008_11511_gb300", "csrc")
SOURCES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")))

REMOTE = re.compile(r"(?:st|ld|atom|red)(?:\.\w+)*\.shared::cluster|\bld_cluster\(")
CLUSTER_WAIT = re.compile(r"barrier\.cluster\.wait|\bcluster_sync\(\)")


def kernels(path):
    """(name, body) of the kernels of a source file, comments taken out; a body
    runs to the next kernel."""
    src = re.sub(r"//[^\n]*", "", open(path).read())
    for part in re.split(r"\b__global__\b", src)[1:]:
        yield re.search(r"\b(k_\w+)\s*\(", part).group(1), part


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_peers_shared_memory_is_touched_after_a_cluster_barrier(path):
    """A block of a cluster may touch another's shared memory only once that
    block has started, which only a cluster barrier says: one is waited for
    before the first such access of every kernel, and one follows the last, so
    that no block ends while another still reads from or writes to it."""
    for name, body in kernels(path):
        remote = [m.start() for m in REMOTE.finditer(body)]
        if not remote:
            continue
        waits = [m.start() for m in CLUSTER_WAIT.finditer(body)]
        assert waits and waits[0] < remote[0], name
        assert waits[-1] > remote[-1], name
