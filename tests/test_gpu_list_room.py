"""D2 and PD2 when the conflict lists do not fit: a sample tells that before the
build, a build that runs out of room all the same gives its memory back, and so
does one whose buffers cannot be allocated.  The net rounds then color, with the
oracle's result, in every form of their launch."""
import numpy as np
import pytest

import oracle
from paper_2107_00075_gb300 import inputs as gen
from tests import _graphs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pgc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2107_00075_gb300 as p
    yield p
    p.pgc_test_list_room(0, 0)
    p.pgc_test_fail_alloc(-1)


def dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


_wanted = {}   # id of an input -> the input (which keeps the id its own) and the oracle's result


def wanted(x):
    if id(x) not in _wanted:
        if isinstance(x, gen.Bipartite):
            w = oracle.color_pd2(x.n_rows, x.n_cols, x.row_ptr, x.col_idx, x.col_ptr, x.row_idx,
                                 seed=2)
        else:
            w = oracle.color_d2(x.row_ptr, x.col_idx, seed=2)
        _wanted[id(x)] = x, w
    return _wanted[id(x)][1]


def color(pgc, x, **kw):
    """The coloring and the kernels that the host loop timed."""
    prof = pgc.Profile(trace_cap=8192)
    kw = dict(seed=2, flags=pgc.PGC_HOST_LOOP, profile=prof) | kw
    if isinstance(x, gen.Bipartite):
        r = pgc.pgc_color_pd2(x.n_rows, x.n_cols, *[dev(a) for a in (x.row_ptr, x.col_idx,
                                                                     x.col_ptr, x.row_idx)], **kw)
    else:
        r = pgc.pgc_color_d2(dev(x.row_ptr), dev(x.col_idx), **kw)
    want = wanted(x)
    assert (r.rounds, r.num_colors) == (want.rounds, want.num_colors)
    assert np.array_equal(r.colors.cpu().numpy(), want.colors)
    assert np.array_equal(prof.trace_w, want.trace_w)
    return set(prof.kernel_ms)


MESH = gen.stencil3d(24, 23, 22, points=27)      # 1.3M list entries of 7.3M pairs
PATTERN = gen.bipartite(30000, 10000, seed=6)    # 1.9M pairs, hardly a repeat


@pytest.mark.parametrize("buffer", [1, 1000, 250_000])
@pytest.mark.parametrize("x", [MESH, PATTERN], ids=["mesh", "pattern"])
def test_build_runs_out_of_room(pgc, x, buffer):
    pgc.pgc_test_list_room(0, buffer)
    try:
        for flags in (pgc.PGC_HOST_LOOP, 0):
            names = color(pgc, x, flags=flags)
            assert not flags or ("net_detect" in names and "net_lists" not in names)
    finally:
        pgc.pgc_test_list_room(0, 0)
    assert "net_lists" in color(pgc, x)


def test_abandoned_build_gives_its_memory_back(pgc):
    """The lists' scratch of a million vertices is over 200 MB, that of the net
    rounds below 130."""
    import torch
    g = gen.stencil3d(100, 100, 100, points=27)
    rp, ci = dev(g.row_ptr), dev(g.col_idx)
    out = torch.empty(g.n, dtype=torch.int32, device="cuda")
    pgc.pgc_release()
    free = torch.cuda.mem_get_info()[0]
    pgc.pgc_test_list_room(0, 1_000_000)
    try:
        pgc.pgc_color_d2(rp, ci, colors=out)
    finally:
        pgc.pgc_test_list_room(0, 0)
    assert free - torch.cuda.mem_get_info()[0] < 160 << 20
    pgc.pgc_release()


@pytest.mark.parametrize("x,limit,built,sampled", [
    (MESH, 0, True, False),                # the default limit holds all pairs
    (MESH, 2_000_000, True, True),         # not all pairs, but the lists
    (MESH, 1_000_000, False, True),
    (PATTERN, 10_000_000, True, False),
    (PATTERN, 1_000_000, False, True),
    # the lists are handed out in chunks here (many vertices per warp): 5.0M
    # entries of 8.8M pairs, and what the chunks leave unused
    (gen.stencil3d(61, 60, 59, points=7), 9_000_000, True, True),
], ids=lambda p: None if not isinstance(p, (bool, int)) else str(p))
def test_sample_decides(pgc, x, limit, built, sampled):
    pgc.pgc_test_list_room(limit, 0)
    try:
        names = color(pgc, x)
        assert ("net_lists" in names) == built
        assert ("net_list_sample" in names) == (built and sampled)   # (else the net rounds' times)
        color(pgc, x, flags=0)
    finally:
        pgc.pgc_test_list_room(0, 0)


def test_list_buffers_that_cannot_be_allocated(pgc):
    """Each allocation after the net setup's eight belongs to the lists."""
    fell_back = 0
    for after in range(8, 40):
        pgc.pgc_release()
        pgc.pgc_test_fail_alloc(after)
        try:
            names = color(pgc, MESH)
        finally:
            pgc.pgc_test_fail_alloc(-1)
        if "net_lists" in names:
            break
        fell_back += 1
    assert 10 <= fell_back < 32
    assert "net_lists" in color(pgc, PATTERN)


def _hub_column():
    """A column in 2100 rows of 2, next to rows of 3 to 90 others."""
    rng = np.random.default_rng(5)
    rows = [[0, 1 + i % 700] for i in range(2100)]
    rows += [sorted(1 + rng.choice(700, size=3 * (i + 1), replace=False)) for i in range(30)]
    return _graphs.bipartite_from_rows(rows, 701)


def _tree(children, leaves):
    """A root whose closed two-hop nets have (children + 1) + children * (leaves
    + 2) members."""
    edges = [(0, 1 + i) for i in range(children)]
    edges += [(1 + i, 1 + children + leaves * i + j)
              for i in range(children) for j in range(leaves)]
    return gen.from_edge_list(1 + children * (1 + leaves), edges)


WIDE = [_hub_column(), _tree(40, 60)]


@pytest.mark.parametrize("kw", [{}, {"block": 128, "grid_per_sm": 1}, {"block": 512},
                                {"block": 1024, "grid_per_sm": 1}], ids=str)
@pytest.mark.parametrize("host_loop", [True, False])
def test_net_rounds_in_every_launch_form(pgc, kw, host_loop):
    """A vertex with 2048 or more net members: net rounds from the start."""
    for x in WIDE:
        names = color(pgc, x, flags=pgc.PGC_HOST_LOOP if host_loop else 0, **kw)
        assert not host_loop or ("net_detect" in names and "net_lists" not in names)


def test_any_call_takes_the_lists_memory_when_out_of_its_own(pgc):
    """The lists that a D2 call left are freed for a D1, batched or D2 call that
    meets an out-of-memory, which then succeeds; without them it reports it."""
    g, wide = gen.rmat(10, 8, seed=5), gen.stencil3d(30, 30, 30, points=7)
    d1 = oracle.color_d1(g.row_ptr, g.col_idx, seed=1)
    batch = gen.make_batch([g, g])
    calls = {
        "d1": lambda: pgc.pgc_color_d1(dev(g.row_ptr), dev(g.col_idx)).colors.cpu().numpy(),
        "batch": lambda: pgc.pgc_color_d1_batch(
            batch.vtx_off, batch.nnz_off, batch.row_ptr, batch.col_idx).colors[:g.n],
        "d2": lambda: pgc.pgc_color_d2(dev(wide.row_ptr), dev(wide.col_idx), seed=2
                                       ).colors.cpu().numpy(),
    }
    expect = {"d1": d1.colors, "batch": d1.colors, "d2": wanted(wide).colors}
    for name, call in calls.items():
        for held in (True, False):
            pgc.pgc_release()
            if held:
                assert "net_lists" in color(pgc, PATTERN)
            pgc.pgc_test_fail_alloc(0)
            try:
                if held:
                    assert np.array_equal(call(), expect[name]), name
                else:
                    with pytest.raises(pgc.PgcError) as e:
                        call()
                    assert e.value.status == 3, name
            finally:
                pgc.pgc_test_fail_alloc(-1)
            assert np.array_equal(call(), expect[name]), name


def _chords(n, shifts):
    """Column i in a row with column i + s for each shift s: two nets of two per
    shift and vertex."""
    a = np.arange(n)
    return _equal_rows(np.concatenate([np.stack([a, (a + s) % n], 1) for s in shifts]), n)


def _equal_rows(rows, n):
    count, length = rows.shape
    row_ptr = np.arange(0, length * count + 1, length, dtype=np.int32)
    col_idx = rows.reshape(-1).astype(np.int32)
    order = np.argsort(col_idx, kind="stable")
    col_ptr = np.zeros(n + 1, np.int32)
    col_ptr[1:] = np.cumsum(np.bincount(col_idx, minlength=n))
    return gen.Bipartite(count, n, row_ptr, col_idx, col_ptr, (order // length).astype(np.int32))


def _plus_row(b, members):
    """b and one more row of the first columns."""
    extra = np.arange(members, dtype=np.int32)
    row_ptr = np.append(b.row_ptr, b.row_ptr[-1] + members).astype(np.int32)
    col_idx = np.append(b.col_idx, extra)
    at = np.repeat(np.arange(b.n_rows + 1), np.diff(row_ptr))
    order = np.argsort(col_idx, kind="stable")
    col_ptr = np.zeros(b.n_cols + 1, np.int32)
    col_ptr[1:] = np.cumsum(np.bincount(col_idx, minlength=b.n_cols))
    return gen.Bipartite(b.n_rows + 1, b.n_cols, row_ptr, col_idx, col_ptr,
                         at[order].astype(np.int32))


# Which way colors: the number of vertices (700,000 or more), the nets per vertex
# (here fewer than 3.5 + about 0.6 for the one other member of each, for the mesh
# fewer than 3.5 + 0.63 * 6) and the largest net (32 at most) decide.
@pytest.mark.parametrize("make,lists", [
    (lambda: _chords(699_999, [1]), True),
    (lambda: _chords(700_000, [1]), False),
    (lambda: _chords(1_200_001, [1, 7]), False),
    (lambda: _chords(1_200_001, [1, 7, 100]), True),
    (lambda: _plus_row(_chords(700_000, [1]), 32), False),
    (lambda: _plus_row(_chords(700_000, [1]), 33), True),
    (lambda: gen.stencil3d(110, 110, 110, points=7), False),
], ids=["699999", "700000", "4 nets", "6 nets", "net of 32", "net of 33", "mesh"])
def test_large_problems_with_few_nets_per_vertex_take_net_rounds(pgc, make, lists):
    x = make()
    names = color(pgc, x)
    assert ("net_lists" in names, "net_detect" in names) == (lists, not lists)
    color(pgc, x, flags=0)
    pgc.pgc_test_list_room(1 << 30 if not lists else 1, 0)   # the other way, same colors
    try:
        names = color(pgc, x)
        assert ("net_lists" in names, "net_detect" in names) == (not lists, lists)
    finally:
        pgc.pgc_test_list_room(0, 0)
