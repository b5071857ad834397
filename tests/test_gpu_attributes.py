"""Stellar radii and semi-major axes are checked on the device before they replace the
context's: a call with one bad value anywhere fails and leaves radii, axes and the
next steps as they were."""
import numpy as np
import pytest

import initial_conditions as ic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 255, 257, 30_001])
@pytest.mark.parametrize("bad", [-1e-300, -1.0, np.inf, -np.inf, np.nan])
def test_bad_values_change_nothing(g_stage, n, bad):
    d = ic.plummer(n, seed=2, masses="salpeter")
    rng = np.random.default_rng(n)
    R, A = 1e-4 * rng.random(n), np.where(rng.random(n) < 0.2, 1e-3, 0.0)
    R[0] = -0.0  # not negative
    c, twin = (g_stage.Cluster({k: d[k] for k in ("r", "vr", "vt", "m", "id")}, [3], precision=1,
                               collisions=1, binaries=1, autotune=0) for _ in range(2))
    for x in (c, twin):
        x.set_radii(R)
        x.set_binaries(A)
    for k in (0, n // 2, n - 1):
        for call, good in ((c.set_radii, R), (c.set_binaries, A)):
            v = good.copy()
            v[k] = bad
            with pytest.raises(g_stage.CMCError) as e:
                call(v)
            assert e.value.status == 1
    np.testing.assert_array_equal(c.radii(), R)
    c.step(2)
    twin.step(2)
    a, b = c.get_state(), twin.get_state()
    for k in ("r", "vr", "vt", "m", "id", "phi"):
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)
    np.testing.assert_array_equal(c.radii(), twin.radii())
    assert c.stats() == twin.stats()


def test_a_failed_call_leaves_nothing_to_the_next(g_stage):
    """A context whose diagnostics ring does not fit (419 GB: one allocation that is
    refused at once) is CMC_ENOMEM; the calls after it are as if it had not been."""
    import torch
    n = 5000
    d = ic.plummer(n, seed=1)
    st = {k: d[k] for k in ("r", "vr", "vt", "m", "id")}
    r = torch.from_numpy(np.sort(d["r"])).cuda()
    m = torch.from_numpy(d["m"]).cuda()
    phi = g_stage.stage_potential(r, m)

    def refused():
        with pytest.raises(g_stage.CMCError) as ei:
            g_stage.Cluster(st, list(range(n)), sizes=[1] * n, diag_ring=1 << 20)
        assert ei.value.status == 2  # CMC_ENOMEM

    refused()
    assert torch.equal(g_stage.stage_potential(r, m), phi)
    refused()
    c = g_stage.Cluster(st, [1], collisions=1)
    refused()
    c.set_radii(np.full(n, 1e-9))
    refused()
    c.step(1)


@pytest.mark.parametrize("precision,most", [(0, 304), (1, 240), (2, 168)])
def test_memory_per_star(g_stage, precision, most):
    """A context's device memory, which bounds the largest cluster, of 2 x 10^7 stars:
    the state (12 B and 5 doubles), the step's records and tables (241, 177 and 109 B),
    a few per cent for the allocator's granularity."""
    import gc

    import torch
    n = 20_000_000
    q = np.random.default_rng(1)
    d = {"r": q.random(n) + 0.5, "vr": np.zeros(n), "vt": q.random(n) * 0.1,
         "m": np.full(n, 1.0 / n), "id": np.arange(n, dtype=np.uint32)}
    gc.collect()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    c = g_stage.Cluster(d, [1], precision=precision, autotune=0)
    torch.cuda.synchronize()
    used = free - torch.cuda.mem_get_info()[0]
    c.step(1)
    assert 0 < used <= most * n, used / n
