"""The tabulated switching function over its parameters: the share of the table
that holds 1 - s (u >= 4), its first interval near d = 0, narrow and wide
switches, a cut-off at the table's end. eps within 1e-13 of its largest value
and the solvent force within 1e-10 of the largest component, the tolerances
tests/test_gpu_parity.py holds the default parameters to.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as W
from oracle import gp_oracle as O

pytestmark = pytest.mark.gpu


def _t(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("r0,w,rcut", [(2.5, 0.5, 6.0), (2.5, 0.5, 5.5), (1.5, 0.3, 6.0), (2.0, 0.4, 6.0),
                                       (0.9, 0.2, 2.1)])
def test_eps_and_force_over_parameters(r0, w, rcut):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0904_4887_gb300 import GPSolver
    grid, cell = (24, 32, 48), (9.0, 10.0, 18.0)
    at = W.slab_atoms(cell, 2, 3, seed=2)
    p = O.DielectricParams(r0=r0, w=w, rcut=rcut)
    s = GPSolver(grid, cell, precision=0, r0=r0, w=w, rcut=rcut)
    s.set_atoms(_t(at.pos))
    eps = O.dielectric(grid, cell, at.pos, p)
    assert np.max(np.abs(s.eps().cpu().numpy() - eps)) < 1e-13 * np.max(eps)
    phi = W.random_field((grid[2], grid[1], grid[0]), seed=3)
    zero = np.zeros(len(at.Z))
    _, _, F = s.energy_forces(_t(phi), torch.zeros(s.shape, dtype=torch.float64, device="cuda"))
    Ge, _ = O.energy_gradient(phi, grid, cell, at.pos, zero, at.sigma_core, at.sigma_cloud, p)
    assert np.max(np.abs(F.cpu().numpy() + Ge)) < 1e-10 * np.max(np.abs(Ge))
