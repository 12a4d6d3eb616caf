"""GPU test of the collision kernel's ways through a cell: packed with others
into a warp's 128 ions, ranked alone by a warp up to 512, by a block up to
1024, in global memory above, with the ions in the cell's planned bucket or
past it.  Cell sizes on both sides of each line go in lock-step with the FP64
oracle; runs whose plan is stale (no sort for long, ions that change cells at
every step) must equal, bit for bit, runs planned anew at every step."""
import numpy as np
import pytest

from paper_1507_03392_gb300 import inputs as I
from tests import parity as P
from tests.test_gpu_coulomb import cells_state

pytestmark = pytest.mark.gpu
KEYS = ("x", "y", "z", "vx", "vy", "vz", "meta")


@pytest.fixture(scope="module")
def E():
    from paper_1507_03392_gb300 import ecris
    return ecris


@pytest.mark.parametrize("sizes,seed", [([1, 2, 3, 4, 5] * 30, 1), ([63, 64, 65, 126, 127, 128, 129, 130], 2),
                                        ([31] * 9 + [2] * 40, 3), ([255, 257, 511, 512, 513, 514], 4),
                                        ([1022, 1023, 1024, 1025, 1026], 5), ([2047, 2049, 3], 6)])
def test_cell_sizes_lockstep(E, sizes, seed):
    rp = I.RunParams(nx=8, ny=8, nz=16, flags=I.F_COULOMB, weight=5e7, dt=1e-8, seed=40 + seed)
    st = cells_state(rp, [round(m / 0.9) if m > 60 else m for m in sizes] + sizes, 40 + seed)
    run = E.Run(rp)
    run.load(st)
    t, orc = P.lockstep(run, rp, st, 3, vel_rel=5e-5)
    assert t["q"] == 0 and t["events"] == 0 and t["pos"] == 0 and t["vel"] == 0, t
    assert run.diag()["coulomb_collisions"] == orc.tally.coulomb_pairs
    run.close()


@pytest.mark.parametrize("mesh,n,dt", [((16, 16, 32), 20_000, 2e-7), ((4, 4, 8), 9_001, 2e-7), ((2, 2, 3), 4_003, 1e-7),
                                       ((48, 48, 96), 30_000, 3e-7), ((16, 16, 32), 3, 1e-7)])
def test_stale_plan_equals_fresh_plan(E, mesh, n, dt):
    rp = I.RunParams(species=I.OXYGEN, nx=mesh[0], ny=mesh[1], nz=mesh[2], ne_in_cm3=1e12, ne_out_cm3=1e11,
                     n0_cm3=1e11, dt=dt, flags=I.F_ALL, weight=1e7, seed=5)
    st = I.make_particles(I.Workload("", rp, n=n, steps=0, atom_fraction=0.3, ion_qmax_init=5, ion_T_eV=10.0,
                                     atoms_fill_chamber=True))
    out = []
    for every in (1, 1000):
        run = E.Run(rp)
        run.set_tuning(sort_every=every)
        run.load(st)
        run.step(1)      # on the load order, its buckets planned from the load's counts
        run.step(39)     # sorted first; then planned at every step, or not again
        out.append((run.state(), run.diag(grids=True)))
        run.close()
    for k in KEYS:
        assert np.array_equal(out[0][0][k], out[1][0][k]), k
    for k in ("extracted", "lost", "alive_by_q", "coulomb_collisions", "ke_lost_eV", "cell_count", "cell_charge"):
        assert np.array_equal(out[0][1][k], out[1][1][k]), k
    if n > 100:
        assert out[0][1]["coulomb_collisions"] > n   # the cells did collide
