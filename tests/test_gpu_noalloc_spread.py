"""GPU test of the allocation-free collision step on ions that are spread
unevenly: few crowded cells of a large mesh, cells on either side of the sizes
at which a cell takes a bucket (2), the bucket's room grows (4), a warp ranks a
cell alone (128, 512) and a block does, in one window (1792) or several.  The
result is that of ecris_step bit for bit, and the time that of an even spread
within a small factor."""
import numpy as np
import pytest

from tests.test_zz_no_alloc import grouped_ions, run_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mesh,sizes", [
    ((32, 32, 64), [130 + i % 31 for i in range(400)]),       # crowded cells, each far above an even share
    ((32, 32, 64), [i % 7 for i in range(8000)]),             # cells of 0 to 6
    ((16, 16, 32), [2] * 900 + [1] * 900 + [3, 4, 5, 126, 127, 128, 129, 130, 255, 257, 511, 512, 513, 514]),
    ((16, 16, 32), [1791, 1792, 1793, 1990, 1991, 1992, 3600, 9001]),   # (a tenth of them atoms)
    ((16, 16, 32), [65_536]),
    ((16, 16, 32), [64] * 64),                               # the most particles and cells that one block prepares
    ((16, 16, 32), [64] * 64 + [1]),
    ((16, 19, 27), [64] * 40 + [3] * 7),                     # more cells than that
    ((4, 4, 4), [5]),
])
def test_equal_to_ecris_step(mesh, sizes):
    from paper_1507_03392_gb300 import inputs as I
    rp = I.RunParams(nx=mesh[0], ny=mesh[1], nz=mesh[2], flags=I.F_COULOMB, weight=5e7, dt=1e-8, seed=31)
    st, cell = grouped_ions(rp, sizes, seed=31)
    run_both(rp, st, cell)


def call_us(cells, n=60_000, ncells=65_536):
    """median time of a call with the ions in the given cells"""
    import torch

    from paper_1507_03392_gb300 import ecris as E
    g = torch.Generator("cuda").manual_seed(4)
    cell = torch.as_tensor(cells, device="cuda")[torch.randint(0, len(cells), (n,), generator=g, device="cuda")]
    cell = cell.sort().values.to(torch.int32)
    q = torch.full((n,), 3, dtype=torch.uint8, device="cuda")
    v = [1e4 * torch.randn(n, generator=g, device="cuda") for _ in range(3)]
    ev = torch.zeros(n, dtype=torch.int32, device="cuda")
    s = torch.cuda.current_stream()
    t = []
    for step in range(25):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(s)
        E.check(None, E.ecris_coulomb_collide_noalloc(n, cell.data_ptr(), q.data_ptr(), *[x.data_ptr() for x in v],
                                                      ev.data_ptr(), ncells, 40.0, 1e8, 1e-9, 10.0, 1e-9, 1, step,
                                                      s.cuda_stream, None))
        b.record(s)
        b.synchronize()
        t.append(a.elapsed_time(b) * 1e3)
    return float(np.median(t[5:]))


def test_crowded_cells_take_no_longer():
    # 150 ions in each of 400 cells are as much work as one in each (a factor of 20
    # allows for fewer blocks at work)
    even, crowded = call_us(np.arange(65_536)), call_us(np.arange(400) + 1000)
    assert crowded < 20.0 * even, (even, crowded)
