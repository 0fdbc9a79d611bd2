"""Sixth-order solves that a V-cycle per Krylov vector does not finish within
max_outer and `inner` steps of multigrid-preconditioned CG do: unequal spacings
with one sweep and one kept vector, and a single correction allowed. The
residual is the library's own for the returned (phi, mu), which
tests/test_gpu_solve6.py checks against the oracle's; the adjoint's residual is
formed here from the oracle's operator.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as W
from oracle import gp_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("grid,cell,repeats,layers,params", [
    ((32, 32, 32), (24.0, 8.0, 14.0), 3, 3, dict(nu1=1, nu2=0, nu_coarse=0, restart=1)),
    ((64, 64, 64), (17.0, 17.0, 16.0), 2, 4, dict(max_outer=2)),
])
def test_slow_cycles_go_over_to_the_inner_iteration(grid, cell, repeats, layers, params, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0904_4887_gb300 import GPSolver
    at = W.slab_atoms(cell, repeats, layers, seed=9)
    pos = torch.tensor(np.ascontiguousarray(at.pos), dtype=torch.float64, device="cuda")
    gauss = torch.tensor(np.stack([at.Z, at.sigma_core, at.sigma_cloud], 1), dtype=torch.float64, device="cuda")
    s = GPSolver(grid, cell, precision=precision, **params)
    s.set_atoms(pos)
    rho = s.build_rho(pos, gauss)
    phi, mu = s.solve6(rho, tol=1e-10)              # raises where it does not converge
    _, rel = s.residual6(rho, phi, mu)
    assert rel < 1.01e-10
    lam, nu = s.adjoint6(rho, tol=1e-10)
    r, l = rho.cpu().numpy(), lam.cpu().numpy()
    res = (r - r.mean()) - O.apply_A6_transpose(l, s.eps().cpu().numpy(), O.spacing(grid, cell)) - nu
    assert np.linalg.norm(res) < 1.01e-10 * np.linalg.norm(r - r.mean())
