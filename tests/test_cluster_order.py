"""Ordering of the thread-block-cluster kernels' shared-memory traffic (no GPU).

* The register panel LU exchanges its warps' candidates through shared memory
  with one block barrier per column.  Its events -- every warp's write of its
  candidate, the barrier, every warp's reading of all candidates, the push of
  the warp that holds the winner, the wait for the pushed bytes -- are laid out
  as a graph of what is ordered before what; a slot may be written again only
  after every reading of what it held.
"""

import itertools
import os
import re

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
