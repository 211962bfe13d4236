"""Distance-2 and partial distance-2 coloring over conflict lists, at the sizes
where the build and its choice change: member counts around a power of two (the
hash set doubles) and around the largest set (above it the net rounds color),
vertices with no, one or more than 32 nets, repeated entries, both sides of a
pattern.  Everything must equal the oracle, with and without the degree rule."""
import numpy as np
import pytest

import oracle
from paper_2107_00075_gb300 import inputs as gen
from tests import _graphs

pytestmark = pytest.mark.gpu


def dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def same(r, want, prof=None):
    assert (r.rounds, r.num_colors) == (want.rounds, want.num_colors)
    assert np.array_equal(r.colors.cpu().numpy(), want.colors)
    if prof is not None:
        assert np.array_equal(prof.trace_w, want.trace_w)
        assert np.array_equal(prof.trace_s, want.trace_s)


def check_pd2(b, seed=1):
    import paper_2107_00075_gb300 as pgc
    args = [dev(a) for a in (b.row_ptr, b.col_idx, b.col_ptr, b.row_idx)]
    # cliques of a thousand vertices take as many rounds: once is enough
    for rule in (True, False) if b.n_cols < 1000 or b.n_rows > 100 else (True,):
        for loop in (0, pgc.PGC_HOST_LOOP) if b.n_cols < 1000 else (0,):
            prof = pgc.Profile(trace_cap=8192)
            r = pgc.pgc_color_pd2(b.n_rows, b.n_cols, *args, seed=seed, profile=prof,
                                  flags=loop | (0 if rule else pgc.PGC_NO_DEGREE_RULE))
            same(r, oracle.color_pd2(b.n_rows, b.n_cols, b.row_ptr, b.col_idx, b.col_ptr,
                                     b.row_idx, seed=seed, recolor_degrees=rule), prof)


def check_d2(g, seed=1):
    import paper_2107_00075_gb300 as pgc
    for rule in (True, False) if np.diff(g.row_ptr).max() < 1000 else (True,):
        r = pgc.pgc_color_d2(dev(g.row_ptr), dev(g.col_idx), seed=seed,
                             flags=0 if rule else pgc.PGC_NO_DEGREE_RULE)
        same(r, oracle.color_d2(g.row_ptr, g.col_idx, seed=seed, recolor_degrees=rule))


@pytest.mark.parametrize("m", [1, 2, 62, 63, 64, 65, 1023, 1024, 2047, 2048])
def test_one_full_row(m):
    """Every column has one net of m members, next to columns in short rows."""
    rows = [list(range(m)), [m, m + 1], [m + 1], []]
    check_pd2(_graphs.bipartite_from_rows(rows, m + 4), seed=m)


@pytest.mark.parametrize("leaves", [61, 62, 63, 64, 1022, 1100])
def test_star(leaves):
    """Distance 2 on a star: the leaves form one clique (2 nets per leaf)."""
    check_d2(gen.star(leaves), seed=leaves)


@pytest.mark.parametrize("nets", [31, 32, 33, 64, 65, 200])
def test_columns_in_many_rows(nets):
    """One column in every row, rows of 1 to 9 other columns."""
    rng = np.random.default_rng(nets)
    rows = [[0] + sorted(1 + rng.choice(150, size=1 + i % 9, replace=False))
            for i in range(nets)]
    check_pd2(_graphs.bipartite_from_rows(rows, 160), seed=nets)


def test_repeated_entries():
    rows = [[0, 1, 1, 2], [2, 2, 3], [3, 3], [0, 4, 4, 4, 5]]
    check_pd2(_graphs.bipartite_from_rows(rows, 7))


@pytest.mark.parametrize("n_cols", [1, 31, 257, 3000, 20000])
def test_random_patterns_and_both_sides(n_cols):
    import paper_2107_00075_gb300 as pgc
    b = gen.bipartite(3 * n_cols, n_cols, seed=n_cols)
    check_pd2(b, seed=n_cols)
    args = (b.row_ptr, b.col_idx, b.col_ptr, b.row_idx)
    r = pgc.pgc_color_pd2_bipartite(b.n_rows, b.n_cols, *[dev(a) for a in args], seed=5)
    same(r, oracle.color_pd2_bipartite(b.n_rows, b.n_cols, *args, seed=5))


@pytest.mark.parametrize("shape", [(3, 1, 1), (17, 5, 9), (40, 41, 43)])
@pytest.mark.parametrize("points", [7, 27])
def test_meshes(shape, points):
    check_d2(gen.stencil3d(*shape, points=points), seed=sum(shape))


def test_repeats_after_distinct_members():
    """A warp that saw few repeats among members skips the hash set; the columns
    after such a one share five equal rows with their neighbors here, so their
    lists then hold repeats, which must change nothing."""
    n = 24000
    b = gen.bipartite(3 * n // 4, n // 4, seed=8)
    rows = [(4 * b.col_idx[b.row_ptr[i]:b.row_ptr[i + 1]]).tolist() for i in range(b.n_rows)]
    for q in range(0, n, 4):
        rows += [[q + 1, q + 2, q + 3]] * 5
    check_pd2(_graphs.bipartite_from_rows(rows, n), seed=3)
