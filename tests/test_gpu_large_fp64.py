"""An FP64 hierarchy above 2^29 points, where the finest level's face coefficients
are not stored: the context's memory per point stays that of the cell form (eps
and its derivative 20 bytes, seven finest-level arrays 56, the coarse levels 8,
tables and padding below 2; the faces would add 32), and its V-cycles, which form
the coefficients from eps, reduce the residual, which the library's FP64 residual
kernel measures, as they do on small grids (below 0.1 after three; 3.3e-3 on
24 x 24 x 48).
"""
import pytest

torch = pytest.importorskip("torch")

import workloads as W

pytestmark = pytest.mark.gpu


def test_cell_form_above_the_line():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.empty_cache()
    grid, cell = (1024, 1024, 768), (104.0, 104.0, 78.0)
    n = grid[0] * grid[1] * grid[2]
    if torch.cuda.mem_get_info()[0] < 130 * n:
        pytest.skip("needs 105 GB of device memory")
    from paper_0904_4887_gb300 import GPSolver
    at = W.slab_atoms((10.0, 10.0, 20.0), 2, 3, seed=9)
    pos = torch.tensor(at.pos + 30.0, dtype=torch.float64, device="cuda")
    gauss = torch.tensor([[z, a, b] for z, a, b in zip(at.Z, at.sigma_core, at.sigma_cloud)], dtype=torch.float64,
                         device="cuda")
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    s = GPSolver(grid, cell, precision=0, inner=3, max_outer=2)
    s.set_atoms(pos)
    torch.cuda.synchronize()
    assert (free - torch.cuda.mem_get_info()[0]) / n < 90.0
    rho = s.build_rho(pos, gauss)
    s.solve(rho, tol=1e-12, check=False)
    st = s.stats()
    assert st.vcycles == 3 and 0.0 < st.residual < 0.1
    del s, rho
    torch.cuda.empty_cache()
