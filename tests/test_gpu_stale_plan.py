"""GPU test of collisions whose ions have no place in the planned buckets: runs
that start as atoms, ionise fast and are seldom sorted, so that most ions are
chained to their cells, few or hundreds a cell.  The state is that of a run
sorted (and planned) often, bit for bit, alone and in a batch, and a step takes
about as long."""
import time

import numpy as np
import pytest

from paper_1507_03392_gb300 import inputs as I

pytestmark = pytest.mark.gpu
KEYS = ("x", "y", "z", "vx", "vy", "vz", "meta")


@pytest.fixture(scope="module")
def E():
    from paper_1507_03392_gb300 import ecris
    return ecris


def case(n, mesh, ne=1e13, ions=0.0, dt=1e-7, seed=3):
    rp = I.RunParams(species=I.ARGON, nx=mesh[0], ny=mesh[1], nz=mesh[2], ne_in_cm3=ne, ne_out_cm3=0.1 * ne, n0_cm3=1e10,
                     dt=dt, flags=I.F_ALL, seed=seed)
    return rp, I.make_particles(I.Workload("", rp, n=n, steps=0, atom_fraction=1.0 - ions, ion_qmax_init=3, ion_T_eV=1.0))


@pytest.mark.parametrize("n,mesh,steps,kw", [
    (3001, (16, 16, 32), 40, {}),              # a few ions a cell
    (60_001, (16, 16, 32), 40, {}),            # tens a cell, several cells at once by a warp
    (1_000_001, (32, 32, 64), 12, {"ne": 1e14}),   # the same in tens of thousands of cells
    (200_003, (16, 16, 32), 20, {}),           # hundreds: one at a time by a warp
    (200_003, (8, 8, 16), 20, {"ne": 1e14}),   # above 512: by a block, many of them at once
    (100_003, (4, 4, 8), 12, {"ne": 1e14}),    # thousands
    (60_001, (16, 16, 32), 40, {"ions": 0.3, "dt": 1e-6}),   # buckets that ions leave and others enter
])
def test_a_stale_plan_changes_nothing(E, n, mesh, steps, kw):
    rp, st = case(n, mesh, **kw)
    often, seldom, b = E.Run(rp), E.Run(rp), E.Batch()
    often.set_tuning(sort_every=4)
    seldom.set_tuning(sort_every=100_000)
    b.set_tuning(sort_every=100_000)
    h = b.add(rp, st)
    for r in (often, seldom):
        r.load(st)
    for part in (steps // 2, 1, steps - steps // 2 - 1):
        often.step(part)
        seldom.step(part)
        b.step(part)
    want, d = often.state(), often.diag(grids=True)
    assert d["alive_by_q"][1:].sum() > 0.2 * n and d["coulomb_collisions"] > n // 20
    for got, e in ((seldom.state(), seldom.diag(grids=True)), (b.state(h), b.diag(h, grids=True))):
        for k in KEYS:
            assert np.array_equal(got[k], want[k]), k
        for k in ("coulomb_collisions", "cell_count", "cell_charge", "lost", "extracted"):
            assert np.array_equal(e[k], d[k]), k
    often.close()
    seldom.close()
    b.close()


def test_seldom_sorted_steps_take_no_longer(E):
    # (a factor of 3 for the cost of particles out of order)
    import torch
    rp, st = case(1_000_000, (32, 32, 64), ne=1e12)
    t = {}
    for every in (32, 512):
        run, t[every] = E.Run(rp), 1e9
        run.set_tuning(sort_every=every)
        for _ in range(3):
            run.load(st)
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            run.step(256)
            torch.cuda.synchronize()
            t[every] = min(t[every], time.perf_counter() - t0)
        run.close()
    assert t[512] < 3.0 * t[32], t
