"""How far below its tolerance an accelerated FP64 split solve ends. The inner GMRES of
the last correction stops at a thousandth of tol (its recursive residual; the true one
differs by rounding), and a solve at 1e-10 leaves at most twice 1e-13 of the right
side, which is what the solution's other errors are small against.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,cell,layers", [((64, 48, 128), (10.0, 10.0, 24.0), 4),
                                              ((48, 48, 128), (9.1, 10.0, 23.3), 5)])
def test_fp64_split_ends_well_below_its_tolerance(grid, cell, layers):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0904_4887_gb300 import GPSolver
    for seed in (1, 2, 3):
        at = W.slab_atoms(cell, 2, layers, seed=seed)
        pos = torch.tensor(np.ascontiguousarray(at.pos), dtype=torch.float64, device="cuda")
        gauss = torch.tensor(np.stack([at.Z, at.sigma_core, at.sigma_cloud], 1), dtype=torch.float64, device="cuda")
        s = GPSolver(grid, cell, precision=0, split=1)
        s.set_atoms(pos)
        s.solve(s.build_rho(pos, gauss), tol=1e-10)
        st = s.stats()
        assert st.split_active == 1
        assert st.residual < 2e-13, (seed, st.residual)
