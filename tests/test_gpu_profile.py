"""What pgc_profile's arrays hold after a call through the C ABI: every entry of
every array that is not NULL is written, whatever it held before."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2107_00075_gb300 import binding
from paper_2107_00075_gb300 import inputs as gen

pytestmark = pytest.mark.gpu

NAMES = ("trace_w", "trace_s", "trace_h", "trace_nets", "trace_members")


@pytest.mark.parametrize("skip", [None, "trace_nets", "trace_members"])
@pytest.mark.parametrize("loop", [0, binding.PGC_HOST_LOOP])
def test_distance2_over_lists_fills_reused_arrays(loop, skip):
    g = gen.stencil3d(9, 8, 7, points=27)
    want = oracle.color_d2(g.row_ptr, g.col_idx, seed=1)
    L, cap = binding.lib(), 512
    arrays = {k: np.full(cap, -7, np.int64) for k in NAMES if k != skip}
    prof = binding.PgcProfileC()
    for k, a in arrays.items():
        setattr(prof, k, a.ctypes.data)
    prof.trace_cap = cap
    o = binding.PgcOptsC()
    L.pgc_opts_init(ctypes.byref(o))
    o.flags, o.profile = loop, ctypes.pointer(prof)
    colors = np.zeros(g.n, np.int32)
    rounds, ncol = ctypes.c_int32(0), ctypes.c_int32(0)
    st = L.pgc_color_d2(g.n, g.row_ptr.ctypes.data, g.col_idx.ctypes.data, ctypes.c_uint64(1),
                        colors.ctypes.data, ctypes.byref(rounds), ctypes.byref(ncol),
                        ctypes.byref(o), None)
    assert st == 0 and np.array_equal(colors, want.colors)
    r = rounds.value
    assert np.array_equal(arrays["trace_w"][:r], want.trace_w)
    assert np.array_equal(arrays["trace_s"][:r], want.trace_s)
    for k, a in arrays.items():
        assert not a[r:].any(), k
        if k in ("trace_nets", "trace_members"):   # the rounds visit no net
            assert not a.any(), k
