"""GPU test of ecris_run_bytes: what a budget charges for a run against what the
run holds on the device, for runs of many particles and runs of many cells,
with and without collisions and an E grid."""
import ctypes

import numpy as np
import pytest

from paper_1507_03392_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def pool_used(E):
    """bytes in use of the device's default memory pool, from which the library allocates"""
    import torch
    torch.cuda.synchronize()
    pool, used = ctypes.c_void_p(), ctypes.c_uint64()
    assert E.LIB.cudaDeviceGetDefaultMemPool(ctypes.byref(pool), 0) == 0
    assert E.LIB.cudaMemPoolGetAttribute(pool, 7, ctypes.byref(used)) == 0   # cudaMemPoolAttrUsedMemCurrent
    return used.value


@pytest.mark.parametrize("n,mesh,coulomb,field", [
    (4_000_001, (64, 64, 128), False, False),
    (4_000_001, (64, 64, 128), True, False),
    (100_003, (96, 96, 192), True, True),
    (100_003, (96, 96, 192), False, True),
    (10_000, (32, 32, 64), False, False),
    (1, (8, 8, 8), True, True),
])
def test_a_run_holds_what_it_is_charged(n, mesh, coulomb, field):
    from paper_1507_03392_gb300 import ecris as E
    rp = I.RunParams(nx=mesh[0], ny=mesh[1], nz=mesh[2], flags=I.F_ALL if coulomb else I.F_ALL_NO_COULOMB, seed=1)
    z = np.zeros(n, np.float32)
    st = {k: z for k in ("x", "y", "vx", "vy", "vz")} | {"z": np.full(n, 0.1, np.float32), "q": np.zeros(n, np.uint8)}
    before = pool_used(E)
    run = E.Run(rp, E=I.make_efield(rp, 2e3, -1e3) if field else None)
    run.load(st)
    for _ in range(3):
        run.step(20)
    held = pool_used(E) - before
    run.close()
    nc = mesh[0] * mesh[1] * mesh[2]
    charged = E.ecris_run_bytes(n, *mesh, int(coulomb))
    # up to an E grid and the longest on-axis table above what is held, never below; arrays
    # are rounded up to the allocator's granularity
    assert held <= charged + 4096
    assert charged <= held + (0 if field else 16 * nc) + (1 << 20) + (1 << 16), (held, charged)
