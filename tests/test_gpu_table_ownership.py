"""Who owns a context's coordinate tables: setting van der Waals radii, which replaces a
buffer of its own, gives back none of the tables' memory, and destroying the context
gives back all of it. Read off the device's free memory; nothing here reads a table.
"""
import gc

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_radii_leave_the_coordinate_tables():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0904_4887_gb300 import GPSolver
    n, grid, cell = 4096, (32, 32, 64), (40.0, 40.0, 80.0)
    rng = np.random.default_rng(3)
    pos = torch.tensor(rng.uniform(0.0, 1.0, (n, 3)) * cell, dtype=torch.float64, device="cuda")
    radii = torch.full((n,), 1.7, dtype=torch.float64, device="cuda")
    s = GPSolver(grid, cell)
    s.set_atoms(pos[:1])
    small = _free()
    s.set_atoms(pos)
    held = _free()
    tables = small - held
    assert tables > 24 << 20                       # the tables of 4096 atoms, and their coordinates
    s.ctx.gp_set_vdw_radii(radii)
    assert _free() <= held
    s.ctx.close()
    del s
    gc.collect()
    assert _free() >= held + tables
