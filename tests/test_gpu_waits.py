"""The engine's two bounded waits among blocks -- the mid loop's grid barriers and
the core phase's meeting -- each give up by themselves: one block is held back by
a bounded, host-set delay under a short poll limit, the call returns
PGC_ERR_TIMEOUT naming the wait, and the next call is the oracle's."""
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


def color(pgc, g, **kw):
    import torch
    return pgc.pgc_color_d1(torch.from_numpy(g.row_ptr).cuda(), torch.from_numpy(g.col_idx).cuda(),
                            seed=3, **kw)


def matches_oracle(pgc, g):
    r, want = color(pgc, g), oracle.color_d1(g.row_ptr, g.col_idx, seed=3)
    assert (r.rounds, r.num_colors) == (want.rounds, want.num_colors)
    assert np.array_equal(r.colors.cpu().numpy(), want.colors)


# K_64 commits one vertex a round: round 1 in the setup, round 2 in the mid loop
# (barrier 1 after its assign, barrier 2 after its detection), which then hands
# the 62 others to the core phase.  The block that is late, the barrier it is late
# at, and the worklists traced when the call gave up:
@pytest.mark.parametrize("host_loop", [False, True])
@pytest.mark.parametrize("wait,block,at,worklists", [
    ("core", 1, 1, [64, 63, 62]),   # the core phase had been reached
    ("core", 0, 1, [64, 63, 62]),
    ("mid", 1, 1, [64, 63]),
    ("mid", 0, 1, [64, 63]),        # the block that keeps the round's state
    ("mid", 0, 2, [64, 63, 62]),    # the others leave at the hand-over's barrier
])
def test_wait_gives_up(pgc, wait, block, at, worklists, host_loop):
    g = gen.complete(64)
    prof = pgc.Profile(trace_cap=8)
    if wait == "core":
        pgc.pgc_test_core_barrier(200, block, 50_000)
    else:
        pgc.pgc_test_mid_barrier(200, block, 50_000, at)
    try:
        with pytest.raises(pgc.PgcError) as e:
            color(pgc, g, profile=prof, flags=pgc.PGC_HOST_LOOP if host_loop else 0)
    finally:
        pgc.pgc_test_core_barrier(0, -1, 0)
        pgc.pgc_test_mid_barrier(0, -1, 0, 1)
    assert e.value.status == 5 and f"grid barrier of the {wait} loop" in str(e.value)
    assert [int(x) for x in prof.trace_w if x] == worklists
    matches_oracle(pgc, g)
    matches_oracle(pgc, gen.rmat(12, 16, seed=2))


@pytest.mark.parametrize("wait", ["core", "mid"])
def test_late_block_within_the_limit(pgc, wait):
    hook = pgc.pgc_test_core_barrier if wait == "core" else pgc.pgc_test_mid_barrier
    hook(0, 1, 2_000)
    try:
        matches_oracle(pgc, gen.complete(40))
    finally:
        hook(0, -1, 0)


def test_hook_arguments(pgc):
    for bad in (lambda: pgc.pgc_test_mid_barrier(0, 1, 2_000_001), lambda:
                pgc.pgc_test_mid_barrier(0, 1, 10, 0)):
        with pytest.raises(pgc.PgcError) as e:
            bad()
        assert e.value.status == 1
