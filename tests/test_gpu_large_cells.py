"""GPU test of the cells on either side of the most ions that a warp ranks alone
(512) and that a block ranks in one window (1792), without atoms among them, in
lock-step with the FP64 oracle, and of the export by records of positions over
the whole fixed-point range."""
import numpy as np
import pytest

from paper_1507_03392_gb300 import inputs as I
from tests import parity as P
from tests.test_gpu_coulomb import cells_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[511, 512, 513], [1791, 1792, 1793], [3599, 3600, 5377]])
def test_lockstep(sizes):
    from paper_1507_03392_gb300 import ecris as E
    rp = I.RunParams(nx=8, ny=8, nz=16, flags=I.F_COULOMB, weight=5e7, dt=1e-8, seed=60)
    for seed in range(60, 200):   # cells that lie wholly in the cylinder
        st = cells_state(rp, sizes, seed)
        if len(st["x"]) == sum(sizes):
            break
    assert len(st["x"]) == sum(sizes)
    st["q"] = np.maximum(st["q"], 1)
    run = E.Run(rp)
    run.load(st)
    t, orc = P.lockstep(run, rp, st, 2, vel_rel=5e-5)
    assert t["q"] == 0 and t["events"] == 0 and t["pos"] == 0 and t["vel"] == 0, t
    assert run.diag()["coulomb_collisions"] == orc.tally.coulomb_pairs
    run.close()


@pytest.mark.parametrize("R0,L", [(0.05, 0.4), (1.0 / 3.0, 1.1)])
def test_records_give_the_rounded_product(R0, L):
    import torch

    from paper_1507_03392_gb300 import ecris as E
    n = 600_001
    rp = I.RunParams(nx=8, ny=8, nz=8, R0=R0, L=L, r_ap=0.1 * R0, inlet=(0.0, 0.0, 0.5 * L), flags=I.F_PUSH, dt=1e-9,
                     seed=1)
    rng = np.random.default_rng(n)
    def spread(top):   # even over the range, and over the orders of magnitude below it
        u = np.where(rng.random(n) < 0.5, rng.random(n), 2.0 ** (-32.0 * rng.random(n)))
        return (u * top).astype(np.float32)
    zero = np.zeros(n, np.float32)
    st = {"x": spread(0.7 * R0), "y": -spread(0.7 * R0), "z": spread(0.999 * L), "vx": zero, "vy": zero, "vz": zero,
          "q": np.zeros(n, np.uint8)}
    run = E.Run(rp)
    run.load(st)
    run.step(16)   # sorted (nothing moves): the state goes back through records
    out = {k: torch.zeros(n, dtype=torch.float32, device="cuda") for k in ("x", "y", "z", "vx", "vy", "vz")}
    run.state_to_device(out)
    torch.cuda.synchronize()
    run.close()
    for key, step in (("x", R0 / 2147483648.0), ("y", R0 / 2147483648.0), ("z", L / 4294967296.0)):
        got = out[key].cpu().numpy()
        k0 = np.rint(st[key].astype(np.float64) / step)
        off = 2147483648.0 if key == "z" else 0.0
        ok = np.zeros(n, bool)
        for dk in (-2, -1, 0, 1, 2):
            k = np.clip(k0 + dk, -2147483648.0 + off, 2147483647.0 + off)
            ok |= got == (k * step).astype(np.float32)
        assert ok.all(), (key, st[key][~ok][:5], got[~ok][:5])
