"""Graphs above 256 vertices whose paths do not multiply are walked depth-first
(nothing is stored), the others go through the frontier; both equal the oracle."""
import pytest

import oracle
from paper_2210_16998_gb300 import cfggen as G
from paper_2210_16998_gb300 import tpg

from .helpers import assert_paths_equal, ring_with_tail
from .test_gpu_parity import check_cfg


def cfg_of(n, arcs, name):
    rp, col = G.csr_from_arcs(n, sorted(set(arcs)))
    return G.CFG(n, rp, col, 0, n - 1, name)


def line(n):
    return [(i, i + 1) for i in range(n - 1)]


def looped(n, every=10, back=5):
    return cfg_of(n, line(n) + [(e, e - back) for e in range(every, n - 1, every)], f"looped{n}")


def fan(n):  # 32 arcs and more at one vertex, each to a way of its own length 1
    return cfg_of(n, [(0, i) for i in range(1, n - 1)] + [(i, n - 1) for i in range(1, n - 1)], f"fan{n}")


def self_loops(n):
    return cfg_of(n, line(n) + [(i, i) for i in range(1, n - 1, 40)], f"self{n}")


def diamonds(n, k):  # k diamonds behind a line
    arcs = line(n - 3 * k)
    for d in range(k):
        a = n - 3 * k - 1 + 3 * d
        arcs += [(a, a + 1), (a, a + 2), (a + 1, a + 3), (a + 2, a + 3)]
    return cfg_of(n, arcs, f"diamonds{n}-{k}")


CASES = {
    "ring257": (lambda: ring_with_tail(255), True),
    "ring1000": (lambda: ring_with_tail(998), True),
    "line257": (lambda: cfg_of(257, line(257), "line"), True),
    "looped300": (lambda: looped(300), True),
    "looped1023": (lambda: looped(1023, 31, 30), True),
    "self-loops": (lambda: self_loops(290), True),
    "one-diamond": (lambda: diamonds(300, 1), True),
    "fan": (lambda: fan(320), False),
    "diamonds": (lambda: diamonds(280, 8), False),
}


@pytest.mark.gpu
@pytest.mark.parametrize("name", CASES)
def test_wide_graph(name):
    make, thin = CASES[name]
    cfg = make()
    ref, stats = check_cfg(cfg)
    assert (stats["arena_bytes_alloc"] == 0) == thin
    _, frontier = check_cfg(cfg, capacity=(1 << 20, 1 << 16, 1 << 16), ref=ref)  # capacities are the frontier's
    assert frontier["arena_bytes_alloc"] > 0
    for key in ("simple_paths", "levels", "peak_level_nodes", "pp_levels", "prime_paths", "pp_vertices"):
        assert stats[key] == frontier[key], key


@pytest.mark.gpu
def test_wide_batch_and_capture():
    cfgs = [looped(270), G.diamond_chain(1), ring_with_tail(300), self_loops(41)]
    ns, rp, col, ent, ext = G.concat_batch(cfgs)
    with tpg.tpg_load_cfg_batch(ns, rp, col, ent, ext, location=tpg.TPG_RESULT_DEVICE) as h:
        lists = [(tpg.tpg_prime_paths(h), tpg.tpg_test_paths(h))]
        assert tpg.tpg_get_stats(h)["arena_bytes_alloc"] == 0
        tpg.tpg_graph_capture(h)
        lists.append(tpg.tpg_graph_launch(h))
        for pp, tp in lists:
            for got, which in ((pp, "pp"), (tp, "tp")):
                gp, off, vert = got.host_arrays()
                for i, c in enumerate(cfgs):
                    ref = oracle.run_cfg(c)
                    o = off[int(gp[i]):int(gp[i + 1]) + 1]
                    assert_paths_equal(o - o[0], vert[o[0]:o[-1]], getattr(ref, which + "_offsets"),
                                       getattr(ref, which + "_vertices"), f"graph {i} {which}")
                got.free()
