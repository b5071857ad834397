"""The timestep's counting sort on the shells (sort_packed = 1) against its
radix sort of keys and values (sort_packed = 0): the same states, bit for bit,
where the sort's branches differ.  Sizes sit at the edges of the gather's tiles
(4096 stars) and of its wide and narrow blocks (152 tiles); inputs crowd the new
radii into few shells (runs longer than 32 stars, which a kernel of their own
orders), leave none to sort, repeat radii, or spread the ids over 32 bits.
No tolerance: both sorts give the (r, id) order of the same stars."""
import numpy as np
import pytest

import initial_conditions as ic

pytestmark = pytest.mark.gpu

KEYS = ("r", "vr", "vt", "m", "id", "phi")


def _same(g, d, seeds, sizes=None, steps=3, **cfg):
    st = {k: d[k] for k in ("r", "vr", "vt", "m", "id")}
    a = g.Cluster(st, seeds, sizes=sizes, sort_packed=1, autotune=0, **cfg)
    b = g.Cluster(st, seeds, sizes=sizes, sort_packed=0, autotune=0, **cfg)
    for n in (1, steps - 1):
        a.step(n)
        b.step(n)
        sa, sb = a.get_state(), b.get_state()
        for k in KEYS:
            np.testing.assert_array_equal(sa[k], sb[k], err_msg=k)
    np.testing.assert_array_equal(a.nbound(), b.nbound())
    np.testing.assert_array_equal(a.escaped(), b.escaped())
    assert a.stats() == b.stats()
    return sa


def _thin_shell(n, seed, speed):
    """n stars within 1e-6 of r = 1 at one speed: their new radii lie outside
    and inside the whole shell, in the first and the last bins."""
    g = np.random.default_rng(seed)
    c = 2.0 * g.random(n) - 1.0
    return {"r": 1.0 + 1e-6 * g.random(n), "vr": speed * c, "vt": speed * np.sqrt(1.0 - c * c),
            "m": np.full(n, 1.0 / n), "id": g.permutation(n).astype(np.uint32)}


@pytest.mark.parametrize("n", [1, 2, 33, 4095, 4096, 4097, 8192 + 31, 12289])
@pytest.mark.parametrize("precision", [0, 1, 2])
def test_sizes_at_the_tile_edges(g_stage, n, precision):
    _same(g_stage, ic.plummer(n, seed=n), [7], precision=precision)


@pytest.mark.parametrize("n", [65, 4097, 30_000])
@pytest.mark.parametrize("precision", [0, 1, 2])
def test_runs_in_one_shell(g_stage, n, precision):
    """Nearly every new radius in two bins: runs of thousands of stars."""
    sa = _same(g_stage, _thin_shell(n, n, 1.2), [3], precision=precision)
    fin = np.isfinite(sa["r"])
    assert np.all(np.diff(sa["r"][fin]) >= 0)


@pytest.mark.parametrize("n", [300_000, 1_000_003])
def test_runs_of_many_tiles(g_stage, n):
    """The new radii of a thin shell: two runs of hundreds of tiles, merged in many
    passes, the bins counted in the orbit step's kernels (300,000) or apart."""
    _same(g_stage, _thin_shell(n, n, 1.2), [3], precision=1, steps=2)


def test_very_many_runs_of_all_lengths(g_stage):
    """Shells of 40 to 10,000 stars far apart, whose new radii lie just inside and just
    outside of them: more listed runs than blocks, short ones and ones of several
    tiles."""
    g = np.random.default_rng(8)
    lengths = np.concatenate([g.integers(40, 140, 900), [4000, 4096, 4200, 8000, 8192, 10_000]])
    g.shuffle(lengths)
    at = np.repeat(np.geomspace(1e-3, 1e3, len(lengths)), lengths)
    n = len(at)
    d = {"r": at * (1.0 + 1e-9 * g.random(n)), "m": np.full(n, 1.0 / n),
         "id": g.permutation(n).astype(np.uint32)}
    order = np.argsort(d["r"])
    inside = np.empty(n)
    inside[order] = (np.arange(n) + 1.0) / n
    v = np.sqrt(inside / d["r"])
    d["vr"], d["vt"] = 1e-3 * v * g.standard_normal(n), v * (1.0 + 1e-3 * g.standard_normal(n))
    _same(g_stage, d, [3], precision=1)
    _same(g_stage, d, [3], precision=0, max_trials=1)


@pytest.mark.parametrize("length", [32, 33, 64, 65, 2047, 2048, 2049, 4096, 4097, 9000])
def test_run_of_exactly(g_stage, length):
    """One radius many times over, by id: escapers in one bin (one star's large id
    makes the bins of ids that wide), as many as fill a list's entry, a tile, two."""
    n = 20_000
    d = ic.plummer(n, seed=5)
    g = np.random.default_rng(length)
    d["id"] = g.permutation(n).astype(np.uint32)
    fast = g.choice(n, length + 1, replace=False)
    d["id"][fast[0]] = 2**32 - 1
    d["vr"][fast[1:]] *= 100.0
    d["vt"][fast[1:]] *= 100.0
    for precision in (0, 1):
        sa = _same(g_stage, d, [5], precision=precision, steps=1, gamma=1e-9)  # no relaxation
        out = ~np.isfinite(sa["r"])
        assert out.sum() == length and np.all(np.diff(sa["id"][out].astype(np.int64)) > 0)


def test_no_slow_case_where_radii_crowd(g_stage):
    """The sort of a million stars in two bins within a small multiple of the radix
    passes' time (twice measured; one block for each run took two hundred times)."""
    d, t = _thin_shell(1_000_000, 2, 1.2), {}
    for packed in (0, 1):
        c = g_stage.Cluster(d, [3], precision=1, autotune=0, sort_packed=packed)
        st, t[packed] = c.get_state(), np.inf
        for _ in range(4):
            c.set_state(st, 0)
            t[packed] = min(t[packed], c.step_profiled(1)["sort"])
    assert t[1] < 10.0 * t[0]


def test_runs_across_tile_edges(g_stage):
    """Two thin shells inside a Plummer sphere: long runs beside runs of one
    or two stars, starting and ending anywhere in the tiles."""
    n = 20_000
    d = ic.plummer(n, seed=4)
    g = np.random.default_rng(4)
    for lo, hi, r in ((3000, 7000, 0.5), (11_000, 11_100, 2.0)):
        d["r"][lo:hi] = r * (1.0 + 1e-9 * g.random(hi - lo))
    for precision in (0, 1):
        _same(g_stage, d, [5], precision=precision)


def test_equal_radii_and_stars_that_stay(g_stage):
    """Groups of equal radii, some on circular orbits (they keep their radius:
    bins found by bisection, ties by id)."""
    n = 5000
    d = ic.plummer(n, seed=9)
    d["r"][:600] = np.repeat(d["r"][:20], 30)
    d["vr"][:300] = 0.0
    d["vt"][:300] = 0.3
    d["id"] = np.random.default_rng(1).permutation(n).astype(np.uint32)
    for precision in (0, 1, 2):
        _same(g_stage, d, [5], precision=precision)


@pytest.mark.parametrize("spread", ["top", "wide", "one"])
def test_escapers_with_sparse_ids(g_stage, spread):
    """Thousands of escapers over several steps, their bins taken from ids near
    2^32, spread over all of it, or dense but for one large id."""
    n = 9000
    d = ic.plummer(n, seed=2)
    g = np.random.default_rng(2)
    fast = g.choice(n, 3000, replace=False)
    d["vr"][fast] *= 3.0
    d["vt"][fast] *= 3.0
    base = g.permutation(n).astype(np.uint64)
    if spread == "top":
        base = base + (2**32 - n)
    elif spread == "wide":
        base = base * (2**32 // n)
    else:
        base[17] = 2**32 - 1
    d["id"] = base.astype(np.uint32)
    sa = _same(g_stage, d, [8], precision=1, steps=5)
    out = ~np.isfinite(sa["r"])
    assert out.sum() > 1000 and np.all(np.diff(sa["id"][out].astype(np.int64)) > 0)


def test_wide_blocks_and_a_ragged_ensemble(g_stage):
    """153 tiles and more (the gather's narrower blocks; above 262144 stars the
    bins are counted in a kernel of their own)."""
    sizes = [200_000, 4096, 1, 300_001, 4095, 33, 129_000]
    seeds = [300 + i for i in range(len(sizes))]
    parts = [ic.plummer(n, s) for n, s in zip(sizes, seeds)]
    ens = {k: np.concatenate([p[k] for p in parts]) for k in ("r", "vr", "vt", "m", "id")}
    _same(g_stage, ens, seeds, sizes=sizes, precision=1, steps=2)


def test_new_state_with_other_ids_and_one_step_at_a_time(g_stage):
    """set_state with larger ids rebinds the escapers; single steps, several
    steps and profiled steps take turns on the two sides of the radii."""
    n = 6000
    d = ic.plummer(n, seed=3)
    d["vr"][::7] *= 4.0
    st = {k: d[k] for k in ("r", "vr", "vt", "m", "id")}
    big = dict(st, id=(d["id"].astype(np.uint64) * 700_000 + 5).astype(np.uint32))
    c = g_stage.Cluster(st, [6], precision=1, autotune=0)
    c.step(1)
    c.set_state(big, 0)
    c.step(1)
    c.step_profiled(1)
    c.step(2)
    o = g_stage.Cluster(big, [6], precision=1, autotune=0, sort_packed=0)
    o.step(4)
    sa, sb = c.get_state(), o.get_state()
    for k in KEYS:
        np.testing.assert_array_equal(sa[k], sb[k], err_msg=k)


@pytest.mark.parametrize("packed", [0, 1])
def test_groups_of_equal_radii_are_counted(g_stage, packed):
    """The tie counter: groups of equal radii, several of them within the low bits
    that the radix passes leave.  One trial a step, so that most stars stay
    where they are."""
    n = 4000
    d = ic.plummer(n, seed=11)
    d["r"][:600] = 0.7 + np.repeat(np.arange(120), 5) * 2.0 ** -53
    d["r"][600:640] = 0.9
    c = g_stage.Cluster({k: d[k] for k in ("r", "vr", "vt", "m", "id")}, [4], precision=1, autotune=0,
                        max_trials=1, sort_packed=packed)
    want = 0
    for _ in range(3):
        c.step(1)
        r = c.get_state()["r"]
        r, count = np.unique(r[np.isfinite(r)], return_counts=True)
        want += int((count > 1).sum())
        assert want > 50 and c.stats()[0]["ties"] == want
