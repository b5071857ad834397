"""Relaxation with two lanes a pair and with one: sizes on both sides of the rule
that chooses (16,384 pairs), odd stars out, radial pairs (the frame's other branch)
and equal velocities (no deflection), against the FP64 oracle bit for bit."""
import numpy as np
import pytest

from gpu_util import dev, host, sorted_plummer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 3, 63, 64, 65, 129, 4099, 32_767, 32_768, 32_769, 32_770])
@pytest.mark.parametrize("kind", ["plummer", "radial", "equal"])
def test_relax(g_stage, orc, n, kind):
    s = sorted_plummer(n, seed=n % 31 + 2, masses="salpeter")
    if kind == "radial":
        s["vt"][::3] = 0.0
        s["vt"][1::3] = 0.0
    elif kind == "equal":
        s["vr"][:] = 0.25
        s["vt"][:] = 0.0
    lnL = orc.coulomb_log(max(n, 100))
    dt, nbin = orc.timestep(s["r"], s["vr"], s["vt"], s["m"], lnL)
    dt = min(dt, 1.0)
    vr, vt = g_stage.stage_relax(dev(s["vr"]), dev(s["vt"]), dev(s["m"]), dev(s["id"]),
                                 dev(nbin), dt, lnL, 9, 4)
    out = orc.relax(s["vr"], s["vt"], s["m"], s["id"], nbin, dt, lnL, 9, 4)
    np.testing.assert_array_equal(host(vr), out[0])
    np.testing.assert_array_equal(host(vt), out[1])
