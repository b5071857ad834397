"""The sort's bounded device waits run out, on purpose, without faulting or
hanging anything: with a look-back limit of one poll a timestep's sort, by
counting or by radix passes, gives up on earlier tiles, reports CMC_ETIMEOUT and
poisons its context (later calls return CMC_EPOISONED), while another context on
the device is unaffected; so does the merge of a long run on the pass before; with
a tie-fix limit of a few moves the stage sort of a run of equal radii falls back to
sorting by id, then by radius, and still returns the (r, id) order.  Every wait
bound is host-set (cmc_set_wait_limits) and restored to its default afterwards."""
import numpy as np
import pytest

import initial_conditions as ic
from gpu_util import dev, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import paper_1206_5878_gb300 as lib
    lib.load()
    return lib


def _cluster(g, n, seed):
    d = ic.plummer(n, seed=seed)
    return g.Cluster({k: d[k] for k in ("r", "vr", "vt", "m", "id")}, [seed], autotune=0)


@pytest.mark.parametrize("packed", [0, 1])
def test_lookback_limit_times_out_and_poisons(g, packed):
    """The counting sort's scan (550 tiles) and the radix passes (489)."""
    other = _cluster(g, 50_000, 2)  # built before the limit: unaffected later
    d = ic.plummer(2_000_000, seed=1)
    c = g.Cluster({k: d[k] for k in ("r", "vr", "vt", "m", "id")}, [1], autotune=0,
                  sort_packed=packed)
    try:
        g.set_wait_limits(lookback_polls=1)
        with pytest.raises(g.CMCError) as ei:
            c.step(1)
        assert ei.value.status == 5  # CMC_ETIMEOUT
        assert "look-back" in str(ei.value)
        with pytest.raises(g.CMCError) as ei:
            c.energy()
        assert ei.value.status == 6  # CMC_EPOISONED
    finally:
        g.set_wait_limits()
        c.close()
    other.step(2)  # defaults again: a full-size wait budget
    st = other.get_state()
    fin = np.isfinite(st["r"])
    assert np.all(np.diff(st["r"][fin]) >= 0)


def test_stage_sort_reports_the_timeout(g):
    d = ic.plummer(2_000_000, seed=4)
    try:
        g.set_wait_limits(lookback_polls=1)
        with pytest.raises(g.CMCError) as ei:
            g.stage_sort_radius(dev(d["r"]), dev(d["id"]))
        assert ei.value.status == 5
    finally:
        g.set_wait_limits()
    perm = host(g.stage_sort_radius(dev(d["r"]), dev(d["id"])))
    assert np.all(np.diff(d["r"][perm.astype(np.int64)]) >= 0)


def test_tie_move_limit_falls_back_and_keeps_the_order(g, orc):
    n = 20_000
    r = np.full(n, 0.7)
    r[::7] = 0.3  # two long runs of equal radii
    ids = np.random.default_rng(3).permutation(n).astype(np.uint32)
    try:
        g.set_wait_limits(tie_moves=8)
        perm = host(g.stage_sort_radius(dev(r), dev(ids)))
    finally:
        g.set_wait_limits()
    np.testing.assert_array_equal(perm.astype(np.int64), orc.sort_perm(r, ids))


def test_the_merge_of_a_long_run_gives_up(g):
    """A thin shell that falls in: all stars in the innermost bin, two tiles to merge, and
    few enough bins for one tile of the scan, which then has nothing to wait for.
    The stars stay where they are, and a state set afterwards goes on as in a new
    context."""
    n = 3600
    q = np.random.default_rng(1)
    c = 2.0 * q.random(n) - 1.0
    d = {"r": 1.0 + 1e-6 * q.random(n), "vr": 0.5 * c, "vt": 0.5 * np.sqrt(1.0 - c * c),
         "m": np.full(n, 1.0 / n), "id": q.permutation(n).astype(np.uint32)}
    a, b = (g.Cluster(d, [1], autotune=0, precision=1) for _ in range(2))
    st = a.get_state()
    try:
        g.set_wait_limits(lookback_polls=1)
        with pytest.raises(g.CMCError) as ei:
            a.step(1)
        assert ei.value.status == 5  # CMC_ETIMEOUT
    finally:
        g.set_wait_limits()
    a.set_state(st, 0)
    a.step(2)
    b.step(2)
    sa, sb = a.get_state(), b.get_state()
    for k in ("r", "vr", "vt", "m", "id", "phi"):
        np.testing.assert_array_equal(sa[k], sb[k], err_msg=k)


def test_wait_limit_arguments(g):
    g.set_wait_limits(0, 0)
    g.set_wait_limits(-5, -1)  # non-positive: the defaults
