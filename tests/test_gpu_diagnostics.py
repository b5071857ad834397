"""Energy, Lagrange radii and core diagnostics by tiles: against the same sums in
numpy (runs of 16 stars, a doubling scan, trees over 256), bit for bit, at sizes
around the runs, the halves of a block and the tiles, with and without escaped
stars, and for an ensemble."""
import numpy as np
import pytest

import initial_conditions as ic

pytestmark = pytest.mark.gpu
T, P = 256, 16  # threads and stars per thread of the sums: tiles of 4096


def _tree(v):
    v = v.copy()
    w = T // 2
    while w:
        v[:w] = v[:w] + v[w:2 * w]
        w //= 2
    return v[0]


def _chain(a):  # sums along the last axis, one after the other
    s = np.zeros(a.shape[:-1])
    for i in range(a.shape[-1]):
        s = s + a[..., i]
    return s


def _strided(v):  # thread h: elements h, h + 256, ...
    n = (len(v) + T - 1) // T * T
    return _chain(np.pad(v, (0, n - len(v))).reshape(-1, T).T)


def _runs(v, tiles):
    return np.pad(v, (0, tiles * T * P - len(v))).reshape(tiles, T, P)


def _energy(r, vr, vt, m):
    n, tiles = len(r), -(-len(r) // (T * P))
    mt = _runs(m, tiles)
    tile_m = np.array([_tree(_chain(q.reshape(P, T).T)) for q in mt.reshape(tiles, -1)])
    M = np.zeros((tiles, T, P))
    before = np.zeros((tiles, T, P))
    for t in range(tiles):
        base = _tree(_strided(tile_m[:t])) if t else 0.0
        s = _chain(mt[t])
        o = 1
        while o < T:
            s = np.concatenate([s[:o], s[:-o] + s[o:]])
            o *= 2
        b = base + np.concatenate([[0.0], s[:-1]])
        run = np.zeros(T)
        for i in range(P):
            before[t, :, i] = b + run
            run = run + mt[t, :, i]
            M[t, :, i] = b + run
    k = _runs(m * (vr * vr + vt * vt), tiles)
    w = _runs((m * before.ravel()[:n]) / r, tiles)
    K = _tree(_strided(np.array([_tree(_chain(q)) for q in k])))
    W = _tree(_strided(np.array([_tree(_chain(q)) for q in w])))
    return (0.5 * K, -W, 0.5 * K - W), M.ravel()[:n]


def _core(r, m):
    n, tiles = len(r), -(-len(r) // (T * P))
    rho, c = np.zeros(n), (r * r) * r
    k = np.arange(3, n - 3)
    if len(k):
        vol = ((4.0 * np.pi) / 3.0) * (c[k + 3] - c[k - 3])
        mass = (((m[k - 2] + m[k - 1]) + m[k]) + m[k + 1]) + m[k + 2]
        rho[k] = np.where(vol > 0.0, mass / np.where(vol > 0.0, vol, 1.0), 0.0)
    S = [_tree(_strided(np.array([_tree(_chain(q)) for q in _runs(v, tiles)])))
         for v in (rho, rho * rho, rho * r)]
    if not S[0] > 0.0:
        return 0.0, 0.0, 0.0
    return S[1] / S[0], S[2] / S[0], float(np.sum(vol > 0.0))


FRACS = [0.0, 1e-9, 0.01, 0.1, 0.37, 0.5, 0.9, 0.999999, 1.0]


def _check(c, i, r, vr, vt, m):
    e, M = _energy(r, vr, vt, m)
    assert tuple(c.energy()[i]) == e
    lag = c.lagrange_radii(FRACS)[i]
    for f, got in zip(FRACS, lag):
        assert got == r[np.searchsorted(M, f * M[-1])], f
    assert tuple(c.core()[i]) == _core(r, m)


@pytest.mark.parametrize("n", [2, 6, 7, 15, 17, 255, 257, 511, 513, 4095, 4096, 4097, 4102, 8191,
                               12_289, 300_007])
@pytest.mark.parametrize("steps", [0, 2])
def test_sums_in_order(g_stage, n, steps):
    d = ic.plummer(n, seed=n, masses="salpeter")
    if steps:
        d["vr"][::5] *= 2.0
    c = g_stage.Cluster({k: d[k] for k in ("r", "vr", "vt", "m", "id")}, [4], precision=1)
    c.step(steps)
    st = c.get_state()
    b = np.isfinite(st["r"])
    _check(c, 0, *(st[k][b] for k in ("r", "vr", "vt", "m")))


@pytest.mark.parametrize("sizes", [[9, 4097, 300, 20_000],
                                   [1, 2, 6, 7, 8, 15, 16, 17, 31, 33, 300, 511, 512, 5],  # a warp each
                                   [1, 2, 6, 7, 8, 15, 16, 17, 31, 33, 300, 511, 513, 5]])
def test_ensemble(g_stage, sizes):
    parts = [ic.plummer(n, seed=n, masses="salpeter") for n in sizes]
    cat = {k: np.concatenate([p[k] for p in parts]) for k in ("r", "vr", "vt", "m", "id")}
    c = g_stage.Cluster(cat, list(range(len(sizes))), sizes=sizes, precision=1)
    st, o = c.get_state(), np.concatenate([[0], np.cumsum(sizes)])
    for i in range(len(sizes)):
        _check(c, i, *(st[k][o[i]:o[i + 1]] for k in ("r", "vr", "vt", "m")))


def test_lagrange_radii_of_very_many_searches(g_stage):
    """More than 2^27 pairs of a cluster and a fraction (a warp searches for each, so
    their threads do not fit 32 bits): clusters of one star, whose radii are
    all the star's."""
    n, nf = 32769, 4096
    d = ic.plummer(n, seed=5)
    c = g_stage.Cluster({k: d[k] for k in ("r", "vr", "vt", "m", "id")}, list(range(n)),
                        sizes=[1] * n, autotune=0)
    got = c.lagrange_radii(np.linspace(0.0, 1.0, nf))
    assert got.shape == (n, nf) and np.all(got == d["r"][:, None])
