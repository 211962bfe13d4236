"""CPU checks of the byte models that bench.py's roofline uses: the phases of a
profiled coloring (launched rounds, mid loop, core phase) and their bytes, by hand
on small traces, and the hand-over rules against the engine's constants."""
import os
import re
from types import SimpleNamespace

import numpy as np
import pytest

import bench

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2107_00075_gb300", "csrc", "d1_engine.cuh")


def profile(w, s=None, h=None, kernels=("d1_mid", "d1_core")):
    z = [0] * len(w)
    return SimpleNamespace(trace_w=np.array(w), trace_s=np.array(s or z), trace_h=np.array(h or z),
                           kernel_ms={k: 1.0 for k in kernels})


def test_constants_are_the_engine_s():
    src = open(CSRC).read()
    const = {k: int(v) for k, v in re.findall(r"constexpr int (k\w+) = (\d+);", src)}
    assert bench.MID_W == const["kMidMax"] and bench.CORE_W == const["kCoreMax"]
    assert bench.CORE_PACE == const["kCoreRounds"]
    # the rule that d1_phases applies
    assert "nxt <= P.tail_w && (long long)(cur - nxt) * kCoreRounds < nxt" in src
    assert "st->mid = (!done && nxt <= P.mid_w) ? 1 : 0;" in src


@pytest.mark.parametrize("w,mid,core", [
    ([100000, 65537, 65536, 100, 50], 2, 5),     # exactly the mid loop's size, one above it
    ([70000, 65537, 66000, 65537], 4, 4),        # never that small
    ([65536, 60000], 1, 2),                      # from round 2 on
    ([9000, 4609, 4097, 3641], 1, 4),            # 456 * 8 = 3648 >= 3641: too fast
    ([9000, 4609, 4097, 3642], 1, 3),            # 455 * 8 = 3640 < 3642
    ([9000, 8999, 4097, 4096, 4095], 1, 3),      # one above the core's size, then at it
    ([4000, 3999, 3998], 1, 2),                  # never in the mid loop's own first round
])
def test_phases(w, mid, core):
    assert bench.d1_phases(profile(w)) == (mid, core)
    assert bench.d1_phases(profile(w, kernels=("d1_mid",))) == (mid, len(w))
    assert bench.d1_phases(profile(w, kernels=())) == (len(w), len(w))


def test_list_entries_read_at_least():
    # H = 90, 60, 20, 3: rounds 2 to 4 end with 40, 17 and 3 entries of winners;
    # losers W_{r+1} = 6, 2, 0 read four entries each, or what there is of them
    w, s, h = [10, 8, 6, 2], [0, 0, 0, 0], [90, 60, 20, 3]
    _, least, _ = bench.d1_round_bytes(w, s, h, whole_lists=False)
    _, most, _ = bench.d1_round_bytes(w, s, h)
    entries = [0, 40 + 20, 17 + 3, 3]          # min(4 * 6, 20), min(4 * 2, 3), none
    fixed = most - 8.0 * np.array([0, 60, 20, 3])
    assert np.allclose(least - fixed, 8.0 * np.array(entries))
    assert np.all(least <= most)


def test_phase_bytes_on_a_hand_trace():
    # rounds: 1 in the setup, 2 launched, 3 and 4 in the mid loop, 5 in the core
    w = [200000, 100000, 60000, 4001, 4000]
    s, h = [900, 700, 500, 300, 200], [800, 600, 450, 200, 150]
    p = profile(w, s, h)
    assert bench.d1_phases(p) == (2, 4)
    asg, det, psh = bench.d1_round_bytes(w, s, h, whole_lists=False)
    nb = bench.d1_phase_bytes(p, {"a": 10.0, "b": 20.0}, "b")
    assert nb["a"] == 10.0 and nb["b"] == pytest.approx(20.0 + det[0] + psh[0])
    assert nb["d1_assign"] == pytest.approx(32 * 100000)
    assert nb["d1_detect"] == pytest.approx(det[1]) and nb["d1_push"] == pytest.approx(psh[1])
    assert nb["d1_mid"] == pytest.approx((asg + det + psh)[2:4].sum())
    assert nb["d1_core"] == 12 * 150 + 28 * 4000
    # conflict lists: the trace's degrees are not row lengths, so a mean row is
    # what a winner pushes to
    nb = bench.d1_phase_bytes(p, {"b": 0.0}, "b", row_mean=6.0)
    won = 100000 - 60000
    assert nb["d1_push"] == pytest.approx(16 * 6.0 * won)
    # no core phase
    nb = bench.d1_phase_bytes(profile(w, s, h, kernels=("d1_mid",)), {"b": 0.0}, "b")
    assert nb["d1_core"] == 0.0 and nb["d1_mid"] == pytest.approx((asg + det + psh)[2:].sum())


def test_list_setup_bytes():
    b = bench.list_setup_bytes(n=10, n_nets=4, memberships=30, members=200, h1=45)
    assert b["net_init"] == 20 * 10 + 12 * 30 + 4 * 4
    assert b["net_lists"] == 12 * 30 + 4 * 200 + 24 * 45 + 44 * 10
