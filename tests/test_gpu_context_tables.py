"""Tables a context keeps from one dielectric to the next: van der Waals radii set in
between leave the coordinate tables of the tabulated dielectric usable, so the next
dielectric and force are those of a fresh context.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,cell", [((32, 32, 64), (10.0, 10.0, 20.0))])
def test_radii_between_two_dielectrics(grid, cell):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0904_4887_gb300 import GPSolver
    at = W.slab_atoms(cell, 2, 4, seed=9)
    pos = torch.tensor(np.ascontiguousarray(at.pos), dtype=torch.float64, device="cuda")
    radii = torch.full((pos.shape[0],), 1.7, dtype=torch.float64, device="cuda")
    s, fresh = GPSolver(grid, cell), GPSolver(grid, cell)
    s.set_atoms(pos)
    s.ctx.gp_set_vdw_radii(radii)
    hold = torch.full((1 << 20,), float("nan"), dtype=torch.float64, device="cuda")
    s.set_atoms(pos)
    fresh.set_atoms(pos)
    # a tile lists its atoms in no fixed order: the products of at most 31 double-float factors
    # (2^-48 each) differ by 31 * 2 * 3.6e-15 = 2.2e-13 at most
    assert (s.eps() - fresh.eps()).abs().max() <= 1e-12 * fresh.eps().max()
    phi = torch.randn(s.eps().shape, dtype=torch.float64, device="cuda")
    zero = torch.zeros_like(phi)
    F, G = s.energy_forces(phi, zero)[2], fresh.energy_forces(phi, zero)[2]
    # the force sums are added atomically: their order differs from run to run
    assert (F - G).abs().max() <= 1e-11 * G.abs().max()
    del hold
