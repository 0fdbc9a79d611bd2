"""Kernel groups of gp_profile on grids whose finest FP32 level takes the fused
sweeps: those launches belong to the smoother's groups, two sweeps each, and one
residual-and-restriction launch per V-cycle to the finest level's.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nu1,nu2", [(2, 2), (1, 1), (3, 2)])
def test_fused_sweeps_are_booked_as_smoothing(nu1, nu2):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0904_4887_gb300 import GPSolver
    grid, cell = (24, 24, 48), (10.0, 10.0, 20.0)
    at = W.slab_atoms(cell, 2, 3, seed=9)
    pos = torch.tensor(np.ascontiguousarray(at.pos), dtype=torch.float64, device="cuda")
    gauss = torch.tensor(np.stack([at.Z, at.sigma_core, at.sigma_cloud], 1), dtype=torch.float64, device="cuda")
    s = GPSolver(grid, cell, nu1=nu1, nu2=nu2, inner=3, max_outer=2)
    s.set_atoms(pos)
    rho = s.build_rho(pos, gauss)
    s.ctx.gp_profile(True)
    s.solve(rho, tol=1e-12, check=False)
    p = s.ctx.gp_get_profile()
    s.ctx.gp_profile(False)
    st = s.stats()
    assert st.sweep_shape == -1 and st.vcycles == 3
    assert p["smooth0_zero"]["launches"] == 3
    assert p["smooth0"]["launches"] == 3 * ((nu1 + 1) // 2 - 1 + (nu2 + 1) // 2)
    assert p["mg_fine"]["launches"] == 3
