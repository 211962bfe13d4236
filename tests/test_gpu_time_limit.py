"""timeout_ms: the device loop looks at the clock once a round wherever its rounds
run, and a coloring over conflict lists is charged for their build."""
import numpy as np
import pytest

import oracle
from paper_2107_00075_gb300 import inputs as gen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pgc():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2107_00075_gb300 as p
    yield p
    p.pgc_test_core_barrier(0, -1, 0)
    p.pgc_test_mid_barrier(0, -1, 0, 1)


def timed_out(pgc, call):
    with pytest.raises(pgc.PgcError) as e:
        call()
    assert e.value.status == 5 and "timeout_ms" in str(e.value)


def test_list_build_counts(pgc):
    """Groups of eight columns in 200 equal rows each: a set of 1600 members per
    column and lists of seven, so the build takes several milliseconds and the
    eight rounds far less than one."""
    import torch
    cols, per = 1 << 19, 200
    rows = cols // 8 * per
    row = torch.arange(rows, device="cuda", dtype=torch.int32)
    eight = torch.arange(8, device="cuda", dtype=torch.int32)
    row_ptr = torch.arange(rows + 1, device="cuda", dtype=torch.int32) * 8
    col_idx = ((row // per * 8)[:, None] + eight).reshape(-1)
    col_ptr = torch.arange(cols + 1, device="cuda", dtype=torch.int32) * per
    col = torch.arange(cols, device="cuda", dtype=torch.int32)
    row_idx = ((col // 8 * per)[:, None] +
               torch.arange(per, device="cuda", dtype=torch.int32)).reshape(-1)
    args = (rows, cols, row_ptr, col_idx, col_ptr, row_idx)
    prof = pgc.Profile(trace_cap=16)
    r = pgc.pgc_color_pd2(*args, profile=prof, flags=pgc.PGC_HOST_LOOP)
    assert r.num_colors == 8 and prof.kernel_ms["net_lists"] > 2.0
    timed_out(pgc, lambda: pgc.pgc_color_pd2(*args, timeout_ms=1))
    assert torch.equal(pgc.pgc_color_pd2(*args).colors, r.colors)


def color(pgc, g, **kw):
    import torch
    return pgc.pgc_color_d1(torch.from_numpy(g.row_ptr).cuda(), torch.from_numpy(g.col_idx).cuda(),
                            seed=3, **kw)


# Few rounds each, one of them 20 ms longer than the others: a block of the mid
# loop held back in its first round of a grid (5 rounds in all), one of the core
# phase before its first round of K_12 (rounds 3 to 12).
GRID = gen.grid2d(1000)
CASES = [("mid", GRID, 0), ("mid", GRID, 0x20), ("core", gen.complete(12), 0)]


@pytest.mark.parametrize("host_loop", [0, 0x4])
@pytest.mark.parametrize("where,g,flags", CASES, ids=["mid", "mid_dynamic", "core"])
def test_one_long_round(pgc, where, g, flags, host_loop):
    hook = pgc.pgc_test_mid_barrier if where == "mid" else pgc.pgc_test_core_barrier
    hook(0, 1, 20_000)
    try:
        timed_out(pgc, lambda: color(pgc, g, flags=flags | host_loop, timeout_ms=5))
        r = color(pgc, g, flags=flags | host_loop)   # within the default limit
    finally:
        hook(0, -1, 0)
    want = (oracle.color_d1_priority(g.row_ptr, g.col_idx, oracle.PRIO_DYNAMIC, seed=3) if flags
            else oracle.color_d1(g.row_ptr, g.col_idx, seed=3))
    assert r.rounds == want.rounds and np.array_equal(r.colors.cpu().numpy(), want.colors)
