"""GPU test of the export's conversion of fixed-point positions to metres: the
FP32-pair arithmetic must give exactly (float)((double)k * step) for a grid
point k next to the loaded position, from the smallest coordinates to the
chamber's faces, for chamber sizes whose grid steps differ in their last bits,
in the export by records and in the one without."""
import numpy as np
import pytest

from paper_1507_03392_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [50_001, 1_000_003])
@pytest.mark.parametrize("R0,L", [(0.05, 0.4), (0.0315, 0.28), (1.0 / 3.0, 1.1), (2.0 ** -5, 0.25)])
def test_metres_are_the_rounded_product(n, R0, L):
    from paper_1507_03392_gb300 import ecris as E
    rp = I.RunParams(nx=8, ny=8, nz=8, R0=R0, L=L, r_ap=0.1 * R0, inlet=(0.0, 0.0, 0.5 * L), flags=I.F_PUSH, dt=1e-9,
                     seed=1)
    rng = np.random.default_rng(n)
    def spread(m, top):   # even over the range, and over the orders of magnitude below it
        u = np.where(rng.random(m) < 0.5, rng.random(m), 2.0 ** (-32.0 * rng.random(m)))
        return (u * top).astype(np.float32)
    st = {"x": spread(n, 0.7 * R0) * rng.choice((-1, 1), n).astype(np.float32),
          "y": spread(n, 0.7 * R0) * rng.choice((-1, 1), n).astype(np.float32), "z": spread(n, 0.999 * L)}
    st["x"][:3] = 0.0
    for k in ("vx", "vy", "vz"):
        st[k] = np.zeros(n, np.float32)
    st["q"] = np.zeros(n, np.uint8)
    run = E.Run(rp)
    run.load(st)
    for steps in (0, 16):   # in load order; sorted (nothing moves)
        if steps:
            run.step(steps)
        out = run.state()
        for key, step in (("x", R0 / 2147483648.0), ("y", R0 / 2147483648.0), ("z", L / 4294967296.0)):
            k0 = np.rint(st[key].astype(np.float64) / step)
            off = 2147483648.0 if key == "z" else 0.0
            ok = np.zeros(n, bool)
            for dk in (-2, -1, 0, 1, 2):
                k = np.clip(k0 + dk, -2147483648.0 + off, 2147483647.0 + off)
                ok |= out[key] == (k * step).astype(np.float32)
            assert ok.all(), (key, steps, st[key][~ok][:5], out[key][~ok][:5])
    run.close()
