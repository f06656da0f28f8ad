"""Order and duplicates of test paths where they share long tree paths: lengths
around the packed keys' words, both key widths, sub-runs of one to many first
vertices, and the same list from the host-driven, batched and captured paths."""
import pytest

import oracle
from paper_2210_16998_gb300 import cfggen as G
from paper_2210_16998_gb300 import tpg

from .helpers import assert_paths_equal
from .test_gpu_parity import check_cfg


def lead_and_loops(lead, loops, size, skip):
    """entry -> lead vertices -> `loops` loops of `size` vertices, one behind the
    other; a loop can be left at its end or after `skip` vertices, and an arc
    from its second vertex closes a shorter way round."""
    arcs = [(i, i + 1) for i in range(lead)]
    n = lead + 1
    for _ in range(loops):
        first = n - 1
        arcs += [(first + i, first + i + 1) for i in range(size)]
        arcs += [(first + size - 1, first + 1), (first + skip, first + size)]
        if size > 4:
            arcs.append((first + 2, first + size - 1))
        n += size
    arcs.append((n - 1, n))
    rp, col = G.csr_from_arcs(n + 1, sorted(set(arcs)))
    return G.CFG(n + 1, rp, col, 0, n, f"lead{lead}-loops{loops}x{size}")


CASES = [(lead, loops, size, skip) for lead in (1, 5, 6, 7, 8, 9, 16) for loops, size, skip in ((1, 3, 1), (3, 6, 2))]
CASES += [(2, loops, 5, 3) for loops in (6, 7, 8)]  # PPs below and above what one block takes
CASES += [(3, 2, 40, 7), (235, 3, 6, 2), (236, 3, 6, 2), (237, 3, 6, 2), (600, 2, 9, 3), (7, 5, 5, 3)]


@pytest.mark.gpu
@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(map(str, c)))
def test_tp_order(case):
    cfg = lead_and_loops(*case)
    ref, _ = check_cfg(cfg)
    assert ref.num_pp > 1
    assert_same_as_batch(cfg, ref)


def assert_same_as_batch(cfg, ref):
    others = [G.diamond_chain(2), lead_and_loops(6, 2, 5, 2)]
    for cfgs in ([cfg] + others, others + [cfg]):
        at = cfgs.index(cfg)
        ns, rp, col, ent, ext = G.concat_batch(cfgs)
        with tpg.tpg_load_cfg_batch(ns, rp, col, ent, ext, location=tpg.TPG_RESULT_DEVICE) as h:
            tpg.tpg_prime_paths(h).free()
            lists = [tpg.tpg_test_paths(h)]
            for captured in range(2):
                if not captured:
                    tpg.tpg_graph_capture(h)
                pp, tp = tpg.tpg_graph_launch(h)
                pp.free()
                lists.append(tp)
            for tp in lists:
                gp, off, vert = tp.host_arrays()
                o = off[int(gp[at]):int(gp[at + 1]) + 1]
                assert_paths_equal(o - o[0], vert[o[0]:o[-1]], ref.tp_offsets, ref.tp_vertices, "TP")
                tp.free()
