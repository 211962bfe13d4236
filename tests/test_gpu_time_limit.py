"""timeout_ms: the device loop looks at the clock once a round wherever its rounds
run, and a coloring over conflict lists is charged for their build."""
import pytest

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
