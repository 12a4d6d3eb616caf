"""GPU test of atoms on the wall.  A load tests r <= R0 in FP32, so an atom on
the rim may start some grid units outside the cylinder that the step tests in
the integers.  If it moves inward slowly, its first step still ends outside
and the wall takes it, although it would be inside some steps later: a window
of steps has to see that as single steps do."""
import numpy as np
import pytest

from paper_1507_03392_gb300 import inputs as I

KEYS = ("x", "y", "z", "vx", "vy", "vz", "meta")
STEPS = 32


def rim_case(coulomb, n=20_000, seed=1):
    """Atoms on the rim, moving inward at up to 2 m/s (and a few ions in the middle)."""
    rp = I.RunParams(species=I.ARGON, nx=16, ny=16, nz=32, ne_in_cm3=1e11, n0_cm3=1e10, dt=1e-9, seed=7,
                     flags=I.F_ALL if coulomb else I.F_ALL_NO_COULOMB)
    rng = np.random.default_rng(seed)
    th = rng.uniform(0.0, 2.0 * np.pi, 3 * n)
    x, y = (rp.R0 * np.cos(th)).astype(np.float32), (rp.R0 * np.sin(th)).astype(np.float32)
    ok = x * x + y * y <= np.float32(rp.R0 * rp.R0)   # the load's test
    x, y, th = x[ok][:n], y[ok][:n], th[ok][:n]
    assert len(x) == n
    v = rng.uniform(0.0, 2.0, n)
    st = {"x": x, "y": y, "z": rng.uniform(0.1, 0.2, n).astype(np.float32), "vx": (-v * np.cos(th)).astype(np.float32),
          "vy": (-v * np.sin(th)).astype(np.float32), "vz": np.zeros(n, np.float32), "q": np.zeros(n, np.uint8)}
    ion = np.arange(n) % 97 == 0
    st["x"][ion] *= np.float32(0.3)
    st["y"][ion] *= np.float32(0.3)
    st["q"][ion] = 2
    return rp, st


def test_some_start_outside_and_end_inside():
    rp, st = rim_case(False)
    s = 2147483648.0 / rp.R0
    X, Y = np.rint(st["x"] * s).astype(object), np.rint(st["y"] * s).astype(object)
    DX, DY = (np.rint(st[k].astype(np.float64) * rp.dt * s).astype(object) for k in ("vx", "vy"))
    r2 = lambda k: (X + k * DX) ** 2 + (Y + k * DY) ** 2
    assert np.sum((r2(1) > 1 << 62) & (r2(STEPS) <= 1 << 62)) > 100


@pytest.mark.gpu
@pytest.mark.parametrize("coulomb", [False, True])
def test_a_window_takes_them_as_single_steps_do(coulomb):
    from paper_1507_03392_gb300 import ecris as E
    rp, st = rim_case(coulomb)
    one, many, batch = E.Run(rp), E.Run(rp), E.Batch()
    h = batch.add(rp, st)
    one.load(st)
    many.load(st)
    for _ in range(STEPS):
        one.step(1)
    many.step(STEPS)
    batch.step(STEPS)
    a, d = one.state(), one.diag(grids=True)
    assert d["lost"][0] > 100
    for state, diag in ((many.state(), many.diag(grids=True)), (batch.state(h), batch.diag(h, grids=True))):
        for k in KEYS:
            assert np.array_equal(state[k], a[k]), k
        for k in ("lost", "extracted", "cell_count", "cell_charge", "alive_by_q", "coulomb_collisions"):
            assert np.array_equal(diag[k], d[k]), k
    one.close()
    many.close()
    batch.close()
