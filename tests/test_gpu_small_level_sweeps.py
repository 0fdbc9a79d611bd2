"""nu_coarse on a first coarse level of at most 4096 points. With three levels and the
coarsest solved directly, that level's sweeps are all nu_coarse can change: four of
them in place of two must leave less of the residual after the first correction
(measured: a third on 3456 points, half on 4096).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("grid,cell", [((24, 24, 48), (10.0, 10.0, 20.0)), ((16, 32, 64), (8.5, 10.0, 20.0))])
def test_nu_coarse_acts_on_a_small_first_coarse_level(grid, cell, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0904_4887_gb300 import GPSolver
    at = W.slab_atoms(cell, 2, 3, seed=9)
    pos = torch.tensor(np.ascontiguousarray(at.pos), dtype=torch.float64, device="cuda")
    gauss = torch.tensor(np.stack([at.Z, at.sigma_core, at.sigma_cloud], 1), dtype=torch.float64, device="cuda")
    first = []
    for nu_coarse in (2, 4):
        s = GPSolver(grid, cell, precision=precision, levels=3, nu1=2, nu2=2, nu_coarse=nu_coarse,
                     inner=3, max_outer=2)
        s.set_atoms(pos)
        s.solve(s.build_rho(pos, gauss), tol=1e-12, check=False)
        assert s.stats().levels == 3
        first.append(s.stats().history[1])
    assert first[1] < 0.9 * first[0]
