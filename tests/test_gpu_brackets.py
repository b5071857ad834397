"""The turning points' node brackets (signs of Q found in floats near a node where
it is known in float pairs, the FP64 evaluation where they cannot tell) against
FP64 bisection on the same table (precision 2): the orbit stage's outputs bit for
bit (for orbits on the verge of escape, which leave the model a millionfold, the
turning points), at the inputs where the brackets' branches differ -- one to a few
stars, radial and circular orbits, orbits on the verge of escape, units in
which 1/r, Phi, E or J leave the float pairs' range, and repeated radii.  No
tolerance: both compute the same FP64 operations at the same nodes."""
import numpy as np
import pytest

import initial_conditions as ic
from gpu_util import dev, host

pytestmark = pytest.mark.gpu


def _table(n, seed, masses="equal", ties=0):
    d = ic.plummer(n, seed=seed, masses=masses)
    if ties:
        d["r"][: n // 2] = np.repeat(d["r"][: n // (2 * ties)], ties)[: n // 2]
    p = np.lexsort((d["id"], d["r"]))
    d = {k: v[p] for k, v in d.items()}
    x = 1.0 / d["r"]
    mx = d["m"] * x
    d["phi"] = -(np.cumsum(d["m"]) * x + (np.cumsum(mx[::-1])[::-1] - mx))
    return d


def _compare(g, d, seed=5, step=2, keys=("code", "rmin", "rmax", "F", "r_new", "vr", "vt",
                                          "phi_new")):
    a = {k: dev(np.ascontiguousarray(d[k])) for k in ("r", "phi", "vr", "vt", "id")}
    out = [g.stage_orbit(a["r"], a["phi"], a["vr"], a["vt"], a["id"], seed, step, precision=p)
           for p in (0, 2)]
    for k in keys:
        x, y = host(out[0][k]), host(out[1][k])
        np.testing.assert_array_equal(x, y, err_msg=k)
    return out[0]


@pytest.mark.parametrize("n", [1, 2, 3, 5, 33, 257, 4099, 30_011])
@pytest.mark.parametrize("masses", ["equal", "salpeter"])
def test_sizes(g_stage, n, masses):
    _compare(g_stage, _table(n, n + 1, masses))


@pytest.mark.parametrize("kind", ["radial", "circular", "almost_circular", "verge"])
@pytest.mark.parametrize("n", [500, 20_000])
def test_orbit_shapes(g_stage, n, kind):
    d = _table(n, 3)
    v2 = d["vr"] ** 2 + d["vt"] ** 2
    if kind == "radial":
        d["vr"], d["vt"] = np.sqrt(v2), np.where(np.arange(n) % 2, 0.0, 1e-9)
    elif kind in ("circular", "almost_circular"):
        M = np.cumsum(d["m"]) - 0.5 * d["m"]
        d["vt"] = np.sqrt(M / d["r"])
        d["vr"] = np.zeros(n) if kind == "circular" else 1e-7 * d["vt"]
    else:  # E between -1e-3 and -1e-16 of |Phi|
        f = np.sqrt(-2.0 * d["phi"] * (1.0 - 10.0 ** np.linspace(-16, -3, n)) / v2)
        d["vr"], d["vt"] = d["vr"] * f, d["vt"] * f
    if kind == "verge":
        _compare(g_stage, d, keys=("rmin", "rmax"))
    else:
        _compare(g_stage, d)


@pytest.mark.parametrize("e", [-100, -64, -30, 30, 64, 100])
def test_units(g_stage, e):
    """Lengths times 2^e (potentials 2^-e, speeds 2^(-e/2)): beyond 2^60 the
    walks are FP64 throughout."""
    d = _table(5000, 7)
    d["r"] = d["r"] * 2.0 ** e
    d["phi"] = d["phi"] * 2.0 ** -e
    for k in ("vr", "vt"):
        d[k] = d[k] * 2.0 ** (-e // 2)
    # (at 2^-100 the floats of the envelope's bounds leave their range)
    out = _compare(g_stage, d, **({"keys": ("rmin", "rmax")} if e < -64 else {}))
    assert np.sum(host(out["code"]) == 0) > 4000


def test_repeated_radii_and_gaps(g_stage):
    _compare(g_stage, _table(6000, 9, ties=30))
    # two shells far apart: the walks start far from their nodes
    d = _table(4000, 11)
    d["r"] = np.where(np.arange(4000) < 2000, 0.5, 3.0) * (1.0 + 1e-12 * np.arange(4000))
    x = 1.0 / d["r"]
    mx = d["m"] * x
    d["phi"] = -(np.cumsum(d["m"]) * x + (np.cumsum(mx[::-1])[::-1] - mx))
    _compare(g_stage, d)
