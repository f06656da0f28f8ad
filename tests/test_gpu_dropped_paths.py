"""Paths that the frontier drops (they cannot begin a prime path) are counted
exactly: totals, levels and the largest level against every simple path, and
the prime paths themselves, on CFGs of several strongly connected components."""
import collections

import pytest

import oracle
from oracle import literal
from paper_2210_16998_gb300 import cfggen as G

from .helpers import wrap_digraph
from .test_gpu_parity import check_cfg


def rings(sizes, chords=(), entries=1, exits=1, tail=0, fan=False, seed=1):
    """entry -> ring -> ring -> ... -> exit: each ring is entered at `entries`
    vertices and left at `exits`; chords (u, v) are added to every ring (mod
    its size), and `tail` acyclic vertices of random arcs follow every ring
    (`fan`: first one vertex of its own behind every exit)."""
    rng = G.SplitMix64(seed)
    arcs, prev, n = [], [0], 1
    for m in sizes:
        ring = list(range(n, n + m))
        n += m
        arcs += [(ring[i], ring[(i + 1) % m]) for i in range(m)] if m > 1 else []
        arcs += [(ring[u % m], ring[v % m]) for u, v in chords if u % m != v % m]
        for i, p in enumerate(prev):
            for e in range(entries):
                arcs.append((p, ring[(i + e * max(1, m // entries)) % m]))
        prev = [ring[(m - 1 - i) % m] for i in range(exits)]
        if fan:
            arcs += [(p, n + i) for i, p in enumerate(prev)]
            prev = list(range(n, n + len(prev)))
            n += len(prev)
        for _ in range(tail):
            arcs += [(p, n) for p in prev if rng.randint(0, 2) or p == prev[-1]]
            prev = prev[-1:] + [n]
            n += 1
    arcs += [(p, n) for p in prev]
    rp, col = G.csr_from_arcs(n + 1, sorted(set(arcs)))
    return G.CFG(n + 1, rp, col, 0, n, f"rings-{len(sizes)}-{n + 1}")


def entered_everywhere(m):
    arcs = [(u, (u + d) % m) for u in range(m) for d in (1, 5) if d == 1 or u % 3 == 0]
    rp, col = G.csr_from_arcs(m, sorted(arcs))
    return wrap_digraph(G.CFG(m, rp, col, 0, m - 1, f"entered-{m}"))


CASES = {
    "n106": lambda: rings([50, 54]),  # (first: tables of 44 KB beside the kernel's own shared memory)
    "one-vertex-components": lambda: rings([1] * 12, tail=1),
    "rings": lambda: rings([3, 2, 4, 3], exits=2),
    "several-entries": lambda: rings([5, 6, 4], entries=3, exits=2, chords=[(0, 2), (3, 1)]),
    "acyclic-tails": lambda: rings([4, 3, 5], chords=[(2, 0)], exits=2, tail=4, seed=5),
    "many-predecessors": lambda: rings([9, 7], entries=2, exits=7, tail=2, seed=9),
    "n256": lambda: rings([60, 70, 123]),
    "word-edges": lambda: rings([31, 32, 31], chords=[(7, 2)]),
    "every-vertex-entered": lambda: entered_everywhere(14),  # more counters than a graph's share
    "exits-beyond-the-ring": lambda: rings([40, 5], exits=35, fan=True),  # longest * targets: more than the shared rows
}


@pytest.mark.gpu
@pytest.mark.parametrize("name", CASES)
def test_dropped_paths_are_counted(name):
    cfg = CASES[name]()
    paths = literal.simple_paths(cfg.n, [list(map(int, cfg.succ(u))) for u in range(cfg.n)])
    levels = collections.Counter(len(p) for p in paths)
    ref = oracle.run_cfg(cfg)
    assert ref.n_simple == len(paths)
    _, stats = check_cfg(cfg, ref=ref)
    assert stats["levels"] == max(levels)
    assert stats["peak_level_nodes"] == max(levels.values())
    check_cfg(cfg, capacity=(cfg.n, cfg.n, 1), ref=ref)  # every buffer grows: the relaunches count once
