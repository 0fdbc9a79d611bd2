"""The coarsest inverse beyond one CTA's shared memory (111 to 512 points), block
Gauss-Jordan over sixteen pivots at a time: whole and partial last blocks, the
periodic operator (shifted along the constant) and the band's Dirichlet one.
A wrong inverse leaves the lowest modes to the conjugate gradients, so the
V-cycles a solve takes show it: with the exact inverse they stay within two of
those of the deepest hierarchy, whose coarsest grid has at most 64 points.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as W

pytestmark = pytest.mark.gpu

# grid, cell, levels, split; coarsest points 216 (13.5 blocks), 288, 432, 512, and 5 x 5 planes short of them in the band
CASES = [
    ((24, 24, 24), (9.0, 9.0, 10.0), 3, 0),
    ((24, 24, 32), (9.0, 9.0, 14.0), 3, 0),
    ((24, 24, 48), (10.0, 10.0, 20.0), 3, 0),
    ((32, 32, 32), (10.0, 10.0, 14.0), 3, 0),
    ((24, 24, 48), (10.0, 10.0, 20.0), 3, 1),
    ((16, 16, 64), (8.5, 8.5, 20.0), 3, 1),
]


def _t(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("grid,cell,levels,split", CASES)
def test_large_coarsest_grid(grid, cell, levels, split, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0904_4887_gb300 import GPSolver
    at = W.slab_atoms(cell, 2, 4, seed=8)
    pos = _t(at.pos)
    gauss = _t(np.stack([at.Z, at.sigma_core, at.sigma_cloud], 1))
    phis, cycles = [], []
    for lv in (0, levels):
        s = GPSolver(grid, cell, precision=precision, split=split, levels=lv)
        s.set_atoms(pos)
        rho = s.build_rho(pos, gauss)
        phis.append(s.solve(rho, tol=1e-12))
        cycles.append(s.stats().vcycles)
        assert s.stats().split_active == split
    assert cycles[1] <= cycles[0] + 2
    # both residuals are below 1e-12; phi moves by at most that times the operator's condition
    assert float((phis[0] - phis[1]).abs().max()) < 1e-8 * float(phis[0].abs().max())
