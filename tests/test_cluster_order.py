"""Ordering of the thread-block-cluster kernels' shared-memory traffic (no GPU).

* The register panel LU exchanges its warps' candidates through shared memory
  with one block barrier per column.  Its events -- every warp's write of its
  candidate, the barrier, every warp's reading of all candidates, the push of
  the warp that holds the winner, the wait for the pushed bytes -- are laid out
  as a graph of what is ordered before what; a slot may be written again only
  after every reading of what it held.
* Another CTA's shared memory may be touched only once that CTA has started: in
  every kernel that writes there, a cluster-wide barrier comes before the first
  remote address.
"""

import itertools
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2503_17535_gb300", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def _unordered_reuse(slots, warps, steps, winners):
    """Writes of a candidate slot that some reading of its previous content
    is not ordered before.  One CTA, one thread per row: a warp's events of a
    column in program order, the barrier of a column after every warp's write,
    the wait's end after the push of that column's winner only."""
    edges = {}

    def order(a, b):
        edges.setdefault(a, []).append(b)

    for j in range(steps):
        for w in range(warps):
            order(("write", w, j), ("barrier", j))
            order(("barrier", j), ("read", w, j))
            order(("read", w, j), ("wait", w, j))
            order(("wait", w, j), ("write", w, j + 1))
            order(("read", winners[j], j), ("wait", w, j))   # its push

    def after(a):
        seen, todo = set(), [a]
        while todo:
            for b in edges.get(todo.pop(), []):
                if b not in seen:
                    seen.add(b)
                    todo.append(b)
        return seen

    bad = []
    for j in range(steps - slots):
        for r in range(warps):
            later = after(("read", r, j))
            bad += [(r, w, j) for w in range(warps) if ("write", w, j + slots) not in later]
    return bad


def test_panel_candidates_are_read_before_they_are_overwritten():
    src = _source("linalg.cu")
    decl = re.search(r"__shared__ uint4 wrec\[(?:(\d+) \* )?16\];", src)
    slots = int(decl.group(1) or 1)
    uses = re.findall(r"(?<!\w)wrec\[([^;=]*?)\](?: =|;)", src[src.index("void step(int jj"):src.index("void run(int jj")])
    assert len(uses) == 2 and (slots == 1 or all(u.startswith("slot * 16 + ") for u in uses))
    assert "const int slot = jj & 1;" in src
    for winners in itertools.product(range(3), repeat=5):
        assert not _unordered_reuse(slots, 3, 5, winners)


BARRIER = re.compile(r"cluster_wait\(\)|cl\.sync\(\)|this_cluster\(\)\.sync\(\)")
STORE = r"map_shared_rank\(|peer_addr\("
# where a kernel first makes such a store: a call of the lambda or member function that does
CALLS = {"k_trsv_cluster": r"solve\(dm,", "k_lu_panel_reg": r"p\.template run<"}


def _kernels(src):
    """(name, body) of every __global__ function."""
    for m in re.finditer(r"__global__ void (?:__launch_bounds__\([^{;]*?\)\s+)?(k_\w+)\(", src):
        start = src.index("{", m.end())
        depth, i = 1, start + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(src[i], 0)
            i += 1
        yield m.group(1), src[start:i]


@pytest.mark.parametrize("name,count", [("gemm_tc.cu", 1), ("linalg.cu", 2), ("trsv.cu", 1), ("hps_kernels.cu", 1)])
def test_cluster_barrier_before_the_first_remote_store(name, count):
    found = 0
    for kernel, body in _kernels(_source(name)):
        remote = re.search(CALLS.get(kernel, STORE), body)
        if remote:
            found += 1
            barrier = BARRIER.search(body)
            assert barrier and barrier.start() < remote.start(), kernel
    assert found == count
