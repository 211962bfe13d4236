"""A server's requests hold device memory inside its budget alone, the core phase's
adjacency bits included: nothing is allocated while it runs, and a request that
fits only without them is colored without the core phase."""
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
    return p


def core_bytes(n):
    """k x ceil(k / 32) words for the at most 4096 vertices of the core phase, in
    256-byte units."""
    k = min(n, 4096)
    return (k * ((k + 31) // 32) * 4 + 255) // 256 * 256


def run_all(srv, graphs, count):
    ids = [srv.submit_d1(graphs[i % len(graphs)].row_ptr, graphs[i % len(graphs)].col_idx)
           for i in range(count)]
    return [srv.wait(i) for i in ids]


def test_growing_requests_allocate_nothing(pgc):
    import torch
    long = [gen.complete(1500)]         # 1500 rounds, 0.3 MB of adjacency bits
    large = [gen.rmat(16, 8, seed=2)]   # 2 MB
    with pgc.PgcServer(hbm_budget_bytes=1 << 30, max_active=4) as srv:
        run_all(srv, long, 16)
        assert srv.stats()["max_active_seen"] == 4   # every slot's own buffers exist
        free = torch.cuda.mem_get_info()[0]
        out = run_all(srv, large, 40)
        assert free - torch.cuda.mem_get_info()[0] < 1 << 20
    want = oracle.color_d1(large[0].row_ptr, large[0].col_idx, seed=1)
    for colors, info in out:
        assert np.array_equal(colors, want.colors) and info.rounds == want.rounds


@pytest.mark.parametrize("g", [gen.complete(300), gen.rmat(12, 8, seed=4)], ids=["K_300", "rmat12"])
def test_budget_without_room_for_the_core_phase(pgc, g):
    want = oracle.color_d1(g.row_ptr, g.col_idx, seed=1)
    with pgc.PgcServer(hbm_budget_bytes=256 << 20, max_active=2) as srv:
        (colors, info), = run_all(srv, [g], 1)
    assert np.array_equal(colors, want.colors)
    whole, without = info.footprint_bytes, info.footprint_bytes - core_bytes(g.n)
    for budget, footprint in ((whole, whole), (whole - 1, without), (without, without)):
        with pgc.PgcServer(hbm_budget_bytes=budget, max_active=2) as srv:
            for colors, info in run_all(srv, [g], 3):
                assert np.array_equal(colors, want.colors) and info.rounds == want.rounds
                assert info.footprint_bytes == footprint
            assert srv.stats()["peak_bytes"] <= budget
    with pgc.PgcServer(hbm_budget_bytes=without - 1, max_active=2) as srv:
        with pytest.raises(pgc.PgcError) as e:
            srv.submit_d1(g.row_ptr, g.col_idx)
        assert e.value.status == 6
