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


TICKET = re.compile(r"atomicAdd\((?:ticket|&a\.maxbits\[2\]), 1u\)")


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_last_block_tickets_are_fenced(path):
    """A block that takes a ticket to find out whether it is the last one has a
    fence right before it, behind what the others must see done (or read), and
    the last block one between the ticket and what it does for all."""
    src = re.sub(r"//[^\n]*", "", open(path).read())
    for m in TICKET.finditer(src):
        last_statements = "".join(src[:m.start()].rsplit(";", 2)[1:])
        assert "__threadfence()" in last_statements, src[m.start() - 200:m.end()]
        after = src[m.end():].split("__global__")[0]
        assert "gridDim.x - 1" in after and "__threadfence()" in after, src[m.start():m.end() + 300]
