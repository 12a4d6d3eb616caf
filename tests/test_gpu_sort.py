"""GPU test of the regrouping sort and the buckets' plan at the sizes where the
scan of their block totals changes shape: one block of bins, and totals on both
sides of one round of the last block's threads (256 blocks of 2048 bins or
cells).  A run sorted at every step must equal, bit for bit, one sorted once."""
import numpy as np
import pytest

from paper_1507_03392_gb300 import inputs as I

pytestmark = pytest.mark.gpu
KEYS = ("x", "y", "z", "vx", "vy", "vz", "meta")


@pytest.fixture(scope="module")
def E():
    from paper_1507_03392_gb300 import ecris
    return ecris


@pytest.mark.parametrize("mesh", [(2, 2, 2), (8, 8, 16), (64, 64, 63), (64, 64, 64), (64, 64, 128), (65, 64, 130)])
@pytest.mark.parametrize("flags", [I.F_ALL, I.F_ALL_NO_COULOMB])
def test_sorted_at_every_step_equals_sorted_once(E, mesh, flags):
    rp = I.RunParams(species=I.OXYGEN, nx=mesh[0], ny=mesh[1], nz=mesh[2], ne_in_cm3=1e12, ne_out_cm3=1e11,
                     n0_cm3=1e11, dt=1e-7, flags=flags, weight=1e7, seed=9)
    st = I.make_particles(I.Workload("", rp, n=20_005, steps=0, atom_fraction=0.4, ion_qmax_init=5, ion_T_eV=10.0,
                                     atoms_fill_chamber=True))
    out = []
    for every in (1, 1000):
        run = E.Run(rp)
        run.set_tuning(sort_every=every)
        run.load(st)
        run.step(12)
        out.append((run.state(), run.diag(grids=True)))
        run.close()
    for k in KEYS:
        assert np.array_equal(out[0][0][k], out[1][0][k]), k
    for k in ("extracted", "lost", "alive_by_q", "coulomb_collisions", "cell_count", "cell_charge"):
        assert np.array_equal(out[0][1][k], out[1][1][k]), k
    assert out[0][1]["alive_by_q"].sum() > 19_000
