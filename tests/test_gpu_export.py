"""GPU test of the two ways a run's state goes back to load order: runs from
2^18 particles export through 32-byte records on the device, smaller ones and
host copies by direct scatters.  Sizes around that line and ragged ones; both
give the same state bit for bit, on the load order and after a sort."""
import numpy as np
import pytest

from paper_1507_03392_gb300 import inputs as I

pytestmark = pytest.mark.gpu
KEYS = ("x", "y", "z", "vx", "vy", "vz")


@pytest.mark.parametrize("n", [1, 31, (1 << 18) - 1, 1 << 18, (1 << 18) + 3])
@pytest.mark.parametrize("steps", [1, 9])
def test_device_export_equals_host_export(n, steps):
    import torch

    from paper_1507_03392_gb300 import ecris as E
    rp = I.RunParams(nx=16, ny=16, nz=32, n0_cm3=1e10, ne_in_cm3=1e12, dt=2e-8)
    st = I.make_particles(I.Workload("", rp, n=n, steps=0, atom_fraction=0.5, ion_qmax_init=6,
                                     atoms_fill_chamber=True))
    run = E.Run(rp)
    run.load(st)
    run.step(steps)
    host = run.state()
    dev = {k: torch.zeros(n, dtype=torch.float32, device="cuda") for k in KEYS}
    dev["meta"] = torch.zeros(n, dtype=torch.int32, device="cuda")
    run.state_to_device(dev)
    torch.cuda.synchronize()
    for k in KEYS:
        assert np.array_equal(dev[k].cpu().numpy(), host[k]), k
    assert np.array_equal(dev["meta"].cpu().numpy().view(np.uint32), host["meta"])
    # some of the arrays only
    some = {k: dev[k].fill_(-1.0) if k in ("y", "vz") else None for k in KEYS}
    run.state_to_device(some)
    torch.cuda.synchronize()
    assert np.array_equal(some["y"].cpu().numpy(), host["y"]) and np.array_equal(some["vz"].cpu().numpy(), host["vz"])
    run.close()
