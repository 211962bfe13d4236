"""The core phase (the last rounds, on the subgraph the worklist induces) at the
sizes where its layout changes: worklists around a word, a 128-rank vector, a
warp of rows and the capacity of the cluster, cliques whose colors run past the
window of forbidden colors held on chip, and rows longer than one warp's share
of the adjacency.  Colors, rounds and traces must equal the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2107_00075_gb300 import inputs as gen

pytestmark = pytest.mark.gpu


def check(g, seed, **kw):
    import torch
    import paper_2107_00075_gb300 as pgc
    rp = torch.from_numpy(np.ascontiguousarray(g.row_ptr)).cuda()
    ci = torch.from_numpy(np.ascontiguousarray(g.col_idx)).cuda()
    prof = pgc.Profile(trace_cap=8192)
    r = pgc.pgc_color_d1(rp, ci, seed=seed, profile=prof, **kw)
    want = oracle.color_d1(g.row_ptr, g.col_idx, seed=seed,
                           recolor_degrees=not kw.get("flags", 0) & pgc.PGC_NO_DEGREE_RULE)
    assert (r.rounds, r.num_colors) == (want.rounds, want.num_colors)
    assert np.array_equal(r.colors.cpu().numpy(), want.colors)
    assert np.array_equal(prof.trace_w, want.trace_w)
    assert np.array_equal(prof.trace_s, want.trace_s)


@pytest.mark.parametrize("n", [15, 16, 17, 127, 128, 129, 511, 513, 2047, 4095, 4096, 4097, 6000])
def test_worklist_sizes(n):
    check(gen.er(n, 20.0, seed=n), seed=n)
    check(gen.er(n, 6.0, seed=n + 1), seed=3, flags=1)


@pytest.mark.parametrize("n", [512, 513, 545, 1100])
def test_colors_past_the_window(n):
    """K_n uses n colors; the window on chip holds 512."""
    check(gen.complete(n), seed=n)


def _core_with_hub(leaves, clique):
    """A clique whose first vertex also has many leaves: its row is far longer
    than its part of the core."""
    edges = [(i, j) for i in range(clique) for j in range(i + 1, clique)]
    edges += [(0, clique + i) for i in range(leaves)]
    return gen.from_edge_list(clique + leaves, edges)


@pytest.mark.parametrize("leaves", [3000, 5000, 20000])
def test_long_rows(leaves):
    check(_core_with_hub(leaves, 70), seed=leaves)


@pytest.mark.parametrize("n,hub", [(1 << 17, 1024), (1 << 20, 2048), (1 << 21, 4096)])
@pytest.mark.parametrize("prio", ["DYNAMIC", "SATURATION"])
def test_varying_hubs(n, hub, prio):
    """Round-varying priorities: the length from which a list takes a block grows
    with n; hubs one short of it, at it and past it, joined into a clique."""
    import torch
    import paper_2107_00075_gb300 as pgc
    degrees = [hub - 1, hub, hub + 1, 2 * hub]
    k, edges, at = len(degrees), [], len(degrees)
    for i, d in enumerate(degrees):
        edges += [(i, j) for j in range(i + 1, k)]
        edges += [(i, at + j) for j in range(d - k + 1)]
        at += d - k + 1
    g = gen.from_edge_list(n, edges)
    r = pgc.pgc_color_d1(torch.from_numpy(g.row_ptr).cuda(), torch.from_numpy(g.col_idx).cuda(),
                         seed=5, flags=getattr(pgc, "PGC_PRIORITY_" + prio))
    want = oracle.color_d1_priority(g.row_ptr, g.col_idx, getattr(oracle, "PRIO_" + prio), seed=5)
    assert (r.rounds, r.num_colors) == (want.rounds, want.num_colors)
    assert np.array_equal(r.colors.cpu().numpy(), want.colors)
