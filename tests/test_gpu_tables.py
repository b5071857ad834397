"""The orbit step's tables where the potential kernel's blocks share a tile or fill
long ranges together: FP64 mode with the tables (precision 0) against bisection
on the FP64 table (precision 2), two timesteps, bit for bit; Phi against exact
sums.  No tolerance for the states: both modes compute the same FP64 operations.
M and
Phi: each term is rounded to a unit of at most 2^-49 of its tile's largest (half
of it off, 4096 terms at most), the sums over the tile are exact, and fewer than
32 roundings of 2^-53 follow (the trees over the tiles, the product, the sums),
for the outer sum one more per product."""
import math

import numpy as np
import pytest

import initial_conditions as ic
from gpu_util import dev, host

pytestmark = pytest.mark.gpu


def _model(n, seed, kind="plummer"):
    d = ic.plummer(n, seed=seed, masses="salpeter")
    if kind == "gap":  # two thin shells a factor 10^3 apart: a thousand cells in one range
        r = np.where(np.arange(n) < n // 2, 1e-2, 10.0) * (1.0 + 1e-7 * np.arange(n))
        d["vr"], d["vt"] = np.zeros(n), np.sqrt((np.arange(n) + 1.0) / n / r) * 0.9
        d["r"] = r
    elif kind == "halo":  # stars out to 10^6 radii: most cells belong to few stars
        k = max(n // 50, 1)
        d["r"][:k] = np.geomspace(50.0, 1e6, k)
        d["vr"][:k], d["vt"][:k] = 0.0, 0.5 / np.sqrt(d["r"][:k])
    return d


def _agree(g, d, sizes=None):
    S = []
    for p in (0, 2):
        seeds = [5] if sizes is None else list(range(5, 5 + len(sizes)))
        c = g.Cluster({k: d[k] for k in ("r", "vr", "vt", "m", "id")}, seeds, precision=p, sizes=sizes)
        c.step(2)
        S.append(c.get_state())
    for k in ("r", "vr", "vt", "m", "id", "phi"):
        np.testing.assert_array_equal(S[0][k], S[1][k], err_msg=k)


@pytest.mark.parametrize("n", [1, 2, 31, 255, 256, 257, 511, 513, 2047, 2049, 4095, 4096, 4097,
                               8193, 19 * 4096 + 257, 38 * 4096 - 1, 38 * 4096 + 1,
                               77 * 4096 + 4095, 153 * 4096 + 1])
def test_parts_of_tiles(g_stage, n):
    _agree(g_stage, _model(n, n))


@pytest.mark.parametrize("kind", ["gap", "halo"])
@pytest.mark.parametrize("n", [64, 5000, 200_000])
def test_long_ranges(g_stage, n, kind):
    _agree(g_stage, _model(n, 3, kind))


def test_ragged_ensemble(g_stage):
    sizes = [1, 300, 4096, 256, 9001, 33, 4097, 2]
    parts = [_model(n, 40 + i) for i, n in enumerate(sizes)]
    _agree(g_stage, {k: np.concatenate([q[k] for q in parts]) for k in parts[0]}, sizes)


@pytest.mark.parametrize("n", [1, 256, 257, 4097, 38 * 4096 + 1])
def test_phi_of_parts(g_stage, n):
    d = _model(n, 9)
    p = np.argsort(d["r"], kind="stable")
    r, m = d["r"][p], d["m"][p]
    phi, M = (host(v) for v in g_stage.stage_potential(dev(r), dev(m), want_M=True))
    x = 1.0 / r
    mx = m * x
    t, u = min(n, 4096) * 2.0 ** -50, 32 * 2.0 ** -53
    for k in np.unique(np.linspace(0, n - 1, 40).astype(int)):
        Mk, Sk = math.fsum(m[: k + 1]), math.fsum(mx[k + 1:])
        dM, dS = t * m.max() + u * Mk, t * mx.max() + u * Sk
        assert abs(M[k] - Mk) <= dM
        want = math.fsum([Mk * x[k], Sk])
        assert abs(phi[k] + want) <= dM * x[k] + dS + u * want


@pytest.mark.parametrize("n", [511, 512, 513, 543, 545, 4095, 4097, 9 * 512 + 31, 64 * 4096,
                               64 * 4096 + 1, 152 * 4096, 152 * 4096 + 513])
def test_gather_in_parts(g_stage, n):
    """Stars gathered by parts of a tile, the tiles' sums by their last block: the
    step's Phi is the potential entry point's, whose sums are a kernel's of their
    own, bit for bit, and nothing is lost."""
    d = _model(n, n % 89)
    d["vr"][:: 3] *= 1.6  # some escape
    c = g_stage.Cluster({k: d[k] for k in ("r", "vr", "vt", "m", "id")}, [3], precision=1)
    c.step(3)
    st = c.get_state()
    nb = int(np.isfinite(st["r"]).sum())
    assert nb < n and np.array_equal(np.sort(st["id"]), np.sort(d["id"]))
    phi = host(g_stage.stage_potential(dev(st["r"][:nb]), dev(st["m"][:nb]), want_M=True)[0])
    np.testing.assert_array_equal(st["phi"][:nb], phi)


@pytest.mark.parametrize("n", [300_000, 700_000])
@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("packed", [0, 1])
def test_steps_after_a_sort_that_timed_out(g_stage, n, precision, packed):
    """A look-back that gives up is reported after the call; the steps until then
    run on stars only (no order that was never written).  Another context is as
    before, and so is this one once its state is set again: nothing of the steps that
    went wrong is left in its counters."""
    d = _model(n, 5)
    st = {k: d[k] for k in ("r", "vr", "vt", "m", "id")}
    other = g_stage.Cluster(st, [5], autotune=0, precision=precision, sort_packed=packed)
    c = g_stage.Cluster(st, [5], autotune=0, precision=precision, sort_packed=packed)
    seen = False
    for _ in range(30):  # (whether a poll finds its word is a race)
        c.set_state(st, 0)
        g_stage.set_wait_limits(lookback_polls=1)
        try:
            c.step(3)
        except g_stage.CMCError as e:
            assert e.status == 5  # CMC_ETIMEOUT
            seen = True
            break
        finally:
            g_stage.set_wait_limits()
    assert seen
    c.set_state(st, 0)
    c.step(2)
    other.step(2)
    sa, sb = c.get_state(), other.get_state()
    for k in ("r", "vr", "vt", "m", "id", "phi"):
        np.testing.assert_array_equal(sa[k], sb[k], err_msg=k)
    np.testing.assert_array_equal(c.nbound(), other.nbound())
    np.testing.assert_array_equal(c.dt(), other.dt())


@pytest.mark.parametrize("n", [40, 5000, (1 << 20) - 3, (1 << 20) + 1])
def test_end_of_the_step_with_the_velocities(g_stage, n):
    """The escapers' budget and the counters, by the velocities' kernel or (more than
    2^20 stars) after it: mass and energy booked per step against the stars that
    left, whose energies are exact to the rounding of at most n additions."""
    d = _model(n, 8)
    d["vr"][::7] *= 3.0
    d["vt"][::7] *= 3.0
    c = g_stage.Cluster({k: d[k] for k in ("r", "vr", "vt", "m", "id")}, [2], precision=1)
    was = np.isfinite(c.get_state()["r"]).sum()
    c.step(2)
    st, stat = c.get_state(), c.stats()[0]
    gone = ~np.isfinite(st["r"])
    assert stat["escaped"] == gone.sum() > 0 and c.nbound()[0] == was - gone.sum()
    assert st["step"] == 2
    me = c.escaped()[0]
    mass = math.fsum(st["m"][gone])
    assert abs(me[0] - mass) <= n * 2.0 ** -53 * mass
    assert np.isfinite(me[1]) and me[1] > 0.0


def test_bound_stars_of_a_state_in_order(g_stage):
    """N_bound from the stars' places: no, one, all but one and all stars of a
    segment escaped; Phi as the potential entry point's."""
    sizes, gone = [300, 1, 4097, 64, 513, 2], [0, 1, 1, 63, 513, 0]
    parts = [_model(n, 60 + i) for i, n in enumerate(sizes)]
    cat = {k: np.concatenate([p[k] for p in parts]) for k in ("r", "vr", "vt", "m", "id")}
    c = g_stage.Cluster(cat, list(range(6)), sizes=sizes, precision=1)
    st, o = c.get_state(), np.concatenate([[0], np.cumsum(sizes)])
    for s in range(6):
        st["r"][o[s + 1] - gone[s]:o[s + 1]] = np.inf
        tail = slice(o[s + 1] - gone[s], o[s + 1])
        p = np.argsort(st["id"][tail])
        for k in ("vr", "vt", "m", "id"):
            st[k][tail] = st[k][tail][p]
    c.set_state(st, 0)
    np.testing.assert_array_equal(c.nbound(), np.array(sizes) - np.array(gone))
    now = c.get_state()
    for s in range(6):
        b = slice(o[s], o[s + 1] - gone[s])
        if b.stop > b.start:
            phi = g_stage.stage_potential(dev(st["r"][b]), dev(st["m"][b]), want_M=True)[0]
            np.testing.assert_array_equal(now["phi"][b], host(phi))
    st["id"][5] = st["id"][7]
    with pytest.raises(g_stage.CMCError):
        c.set_state(st, 0)
