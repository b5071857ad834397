"""Eq. 7's bins by pairs and by bins: bin sizes from one pair to more pairs than a
block's threads, ragged last bins, numbers of bins on both sides of the rule that
chooses, the central timesteps over fewer and more than 300 stars; densities and
timesteps against the FP64 oracle bit for bit (sums in star order)."""
import numpy as np
import pytest

from gpu_util import dev, host, sorted_plummer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,bs", [(1, 2), (2, 2), (3, 2), (513, 2), (65_535, 2), (65_537, 2),
                                  (1000, 4), (997, 6), (5003, 50), (4097, 510), (4099, 512),
                                  (4101, 514), (3001, 1026), (40_001, 3000), (100, 256),
                                  (655_361, 20), (655_399, 20)])
def test_bins(g_stage, orc, n, bs):
    s = sorted_plummer(n, seed=n % 97 + 1, masses="salpeter")
    lnL = 7.5
    dt, nbin = g_stage.stage_timestep(*(dev(s[k]) for k in ("r", "vr", "vt", "m")), lnL,
                                      bin_size=bs)
    dto, nbo = orc.timestep(s["r"], s["vr"], s["vt"], s["m"], lnL, bin_size=bs)
    np.testing.assert_array_equal(host(nbin), nbo)
    assert host(dt)[0] == dto


def _central(s, P, R=None, A=None, xbb=0.0, xbs=0.0):
    """Eqs. 8-10, in star order."""
    r, m = s["r"], s["m"]
    v2 = np.float64(0.0)
    for a, b in zip(s["vr"][:P], s["vt"][:P]):
        v2 = v2 + (a * a + b * b)
    order = lambda t: np.float64(sum(t, np.float64(0.0)))
    ns = (3.0 * (P - 1)) / ((4.0 * np.pi) * (r[P - 1] * r[P - 1] * r[P - 1] - r[0] * r[0] * r[0]))
    sig2 = (v2 / P) / 3.0
    sig, T = np.sqrt(sig2), np.inf
    if R is not None:
        R2, MR = order(R[:P] * R[:P]) / P, order(m[:P] * R[:P]) / P
        inv = (((16.0 * np.sqrt(np.pi)) * ns) * R2) * sig
        T = min(T, 1.0 / (inv * (1.0 + MR / ((2.0 * sig2) * R2))))
    if A is not None:
        b = A[:P] > 0.0
        k = int(b.sum())
        a2, ma, am = (order(t[b]) / k for t in (A[:P] * A[:P], m[:P] * A[:P], A[:P]))
        if k < P:
            inv = (((4.0 * np.sqrt(np.pi)) * (ns * (float(P - k) / P))) * ((xbs * xbs) * a2)) * sig
            T = min(T, 1.0 / (inv * (1.0 + ((order(m[:P]) / P) * am) / ((sig2 * xbs) * a2))))
        inv = (((16.0 * np.sqrt(np.pi)) * (ns * (float(k) / P))) * ((xbb * xbb) * a2)) * sig
        T = min(T, 1.0 / (inv * (1.0 + ma / (((2.0 * sig2) * xbb) * a2))))
    return T


@pytest.mark.parametrize("n", [2, 31, 255, 257, 299, 300, 301, 5000])
@pytest.mark.parametrize("which", ["radii", "binaries", "both"])
def test_central(g_stage, n, which):
    """The segment's timestep is the shorter of the central one and Eq. 7's (a run
    without radii and axes)."""
    s = sorted_plummer(n, seed=3, masses="salpeter")
    rng = np.random.default_rng(n)
    R = 5.0 * (1.0 + rng.random(n)) if which != "binaries" else None
    A = None
    if which != "radii":
        A = np.where(rng.random(n) < 0.3, 5.0 * (1.0 + rng.random(n)), 0.0)
        A[0] = 7.0
    c = g_stage.Cluster({k: s[k] for k in ("r", "vr", "vt", "m", "id")}, [1], precision=1,
                        collisions=int(R is not None), binaries=int(A is not None))
    if R is not None:
        c.set_radii(R)
    if A is not None:
        c.set_binaries(A)
    st = c.get_state()
    cfg = c.cfg
    c.step(1)
    plain = g_stage.Cluster({k: s[k] for k in ("r", "vr", "vt", "m", "id")}, [1], precision=1)
    plain.step(1)
    assert c.dt()[0] == min(plain.dt()[0], _central(st, min(n, 300), R, A, cfg.x_bb, cfg.x_bs))
