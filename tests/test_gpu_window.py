"""GPU test of the windows of steps that runs without collisions between ions
take: a call's steps taken together give the same state, tallies, deposits and
first-passage records bit for bit as the same steps taken one call at a time
(which the lock-step tests hold to the oracle).  Cases where a window can go
wrong: particles that cross cells, leave or ionise inside it, frozen ones, a
device update of n_e in between, windows cut by sorts, every opt-in process,
ragged sizes, and a batch whose runs differ."""
import numpy as np
import pytest

from paper_1507_03392_gb300 import inputs as I

pytestmark = pytest.mark.gpu
KEYS = ("x", "y", "z", "vx", "vy", "vz", "meta")


@pytest.fixture(scope="module")
def E():
    from paper_1507_03392_gb300 import ecris
    return ecris


def case(n, dt, flags=I.F_ALL_NO_COULOMB, seed=3, opt_in=False, ions=0.3, **more):
    if opt_in:
        flags |= I.F_DOUBLE | I.F_ELASTIC | I.F_RECOMB
        more = dict(more, k3_factor=0.05, T_refl_eV=0.15)
    rp = I.RunParams(species=I.OXYGEN, nx=17, ny=16, nz=33, ne_in_cm3=2e12, ne_out_cm3=2e11, n0_cm3=2e11, r_ap=0.02,
                     dt=dt, flags=flags, seed=seed, **more)
    if opt_in:
        rp.B_axial = I.flat_axial_profile(rp)
    st = I.make_particles(I.Workload("", rp, n=n, steps=0, atom_fraction=1.0 - ions, ion_qmax_init=5, ion_T_eV=5.0,
                                     atoms_fill_chamber=True))
    return rp, st


def results(run, h=()):
    return run.state(*h), run.diag(*h, grids=True), run.fptd(*h), run.extraction_radius(*h)


def same(a, b):
    for k in KEYS:
        assert np.array_equal(a[0][k], b[0][k]), k
    for k in ("steps", "extracted", "lost", "alive_by_q", "ke_lost_eV", "cell_count", "cell_charge"):
        assert np.array_equal(a[1][k], b[1][k]), k   # (time_s and what divides by it: the host's sum of dt, call by call)
    assert np.array_equal(a[2]["hist"], b[2]["hist"]) and np.array_equal(a[2]["age_sum"], b[2]["age_sum"])
    assert np.array_equal(a[3], b[3])


@pytest.mark.parametrize("n,dt,kw", [
    (5001, 1e-9, {}),
    (5001, 1e-7, {}),
    (70_003, 3e-7, {}),                                       # most particles cross cells or leave in a window
    (5001, 1e-7, {"flags": I.F_ALL_NO_COULOMB & ~I.F_RECYCLE}),
    (3000, 1e-7, {"flags": I.F_PUSH | I.F_RECYCLE}),          # atoms draw no words
    (3000, 1e-7, {"flags": I.F_IONIZE | I.F_EIKICK}),         # nothing moves
    (5001, 1e-7, {"opt_in": True}),
    (2000, 1e-8, {"ions": 0.0}),
    (1, 1e-7, {}),
])
def test_window_equals_single_steps(E, n, dt, kw):
    rp, st = case(n, dt, **kw)
    Ef = I.make_efield(rp, 2e3, -1e3)
    one, many = E.Run(rp, E=Ef), E.Run(rp, E=Ef)
    for r in (one, many):
        r.load(st)
    for part in (3, 40, 1, 64):
        many.step(part)
        for _ in range(part):
            one.step(1)
        same(results(many), results(one))
        if part == 40:
            one.update_ne()
            many.update_ne()
    if n > 4000 and dt == 1e-7 and "flags" not in kw:
        d = many.diag()
        assert d["lost"].sum() > 100 and d["extracted"].sum() > 0   # particles did leave inside the windows
    one.close()
    many.close()


@pytest.mark.parametrize("every", [5, 200])
def test_windows_are_cut_by_sorts(E, every):
    rp, st = case(4000, 1e-7)
    ref, run = E.Run(rp), E.Run(rp)
    run.set_tuning(sort_every=every)
    for r in (ref, run):
        r.load(st)
        r.step(100)
    same(results(run), results(ref))
    run.close()
    ref.close()


@pytest.mark.parametrize("threads,vec", [(0, 0), (128, 1), (512, 4)])
def test_batch_windows_equal_the_runs_alone(E, threads, vec):
    specs = [case(n, dt, seed=s, opt_in=o) for s, (n, dt, o) in
             enumerate([(1, 1e-7, False), (4001, 1e-7, False), (0, 1e-7, False), (30_002, 1e-8, True),
                        (129, 2e-7, False)])]
    b = E.Batch()
    b.set_tuning(threads=threads, particles_per_thread=vec)
    hs = [b.add(rp, st) for rp, st in specs]
    b.step(45)
    b.remove(hs[1])
    b.step(1)
    b.step(34)
    for k in (0, 2, 3, 4):
        rp, st = specs[k]
        r = E.Run(rp)
        r.load(st)
        r.step(80)
        same(results(b, (hs[k],)), results(r))
        r.close()
    b.close()
