"""The FP64 continuation with trials ahead in spare lanes: any number of lanes a star
gives the first accepted trial, and the statistics count the trials up to it.
Mixed and FP64 mode against the same models inside an ensemble, where the list is
long enough for other splits (16, 8, 4, 2, 1 lanes a star); FP64 mode also against
bisection, whose trials are one after the other.  Bit for bit."""
import numpy as np
import pytest

import initial_conditions as ic

pytestmark = pytest.mark.gpu
KEYS = ("r", "vr", "vt", "m", "id", "phi")


def _run(g, parts, seeds, **cfg):
    cat = {k: np.concatenate([p[k] for p in parts]) for k in ("r", "vr", "vt", "m", "id")}
    c = g.Cluster(cat, seeds, sizes=[len(p["r"]) for p in parts], **cfg)
    c.step(2)
    return c.get_state(), c.stats()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("beside", [3_000, 20_000, 60_000, 150_000, 600_000])
def test_first_accepted_trial(g_stage, precision, beside):
    n = 5_003
    a = ic.plummer(n, seed=3, masses="salpeter")
    b = ic.plummer(beside, seed=4)
    st, stats = _run(g_stage, [a], [11], precision=precision)
    both, both_stats = _run(g_stage, [a, b], [11, 12], precision=precision)
    for k in KEYS:
        np.testing.assert_array_equal(st[k], both[k][:n], err_msg=k)
    assert stats[0] == both_stats[0]
    assert stats[0]["fp64_trials"] > 0


@pytest.mark.parametrize("max_trials", [1, 2, 3, 7])
@pytest.mark.parametrize("n", [300, 40_000, 60_000])
def test_trial_cap(g_stage, n, max_trials):
    d = ic.plummer(n, seed=6)
    x, sx = _run(g_stage, [d], [5], precision=0, max_trials=max_trials)
    y, sy = _run(g_stage, [d], [5], precision=2, max_trials=max_trials)
    for k in KEYS:
        np.testing.assert_array_equal(x[k], y[k], err_msg=k)
    for k in ("trials", "cap_hits", "violations"):
        assert sx[0][k] == sy[0][k], k


@pytest.mark.parametrize("sizes", [[25] * 2400, [31, 33, 64, 1, 2, 40_000, 95, 20_000]])
def test_warps_of_several_segments(g_stage, sizes):
    """Enough stars for the trials by rounds, in warps that hold stars of one segment
    and of several."""
    parts = [ic.plummer(n, seed=i + 1, masses="salpeter") for i, n in enumerate(sizes)]
    seeds = list(range(len(sizes)))
    x, sx = _run(g_stage, parts, seeds, precision=0)
    y, sy = _run(g_stage, parts, seeds, precision=2)
    for k in KEYS:
        np.testing.assert_array_equal(x[k], y[k], err_msg=k)
    for a, b in zip(sx, sy):
        assert a["trials"] == b["trials"] and a["violations"] == b["violations"]
