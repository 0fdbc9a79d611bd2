"""The accelerated dry/wet split, whose FFT solve runs between factors eps^-1/2,
against the full-box solve on the same inputs. Both stop at a relative residual
of 1e-12; phi differs by at most the residual times the condition of the
operator, far below the 1e-8 asked here (tests/test_gpu_parity.py holds each
to the oracle).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as W

pytestmark = pytest.mark.gpu

CASES = [
    # grid, cell, lattice repeats, layers, copies of the cell along x, kind, precision
    ((16, 24, 64), (8.5, 9.0, 24.0), 2, 4, 1, 0, 0),
    ((16, 24, 64), (8.5, 9.0, 24.0), 2, 4, 1, 0, 1),
    ((24, 16, 96), (9.0, 8.5, 30.0), 2, 4, 1, 2, 1),        # Eq. 19: a thick dry region
    ((768, 64, 64), (12.0, 12.0, 18.0), 3, 4, 8, 0, 0),     # rows beyond the compile-time transforms
    ((768, 64, 64), (12.0, 12.0, 18.0), 3, 4, 8, 0, 1),
]


def _t(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("grid,cell,n,layers,copies,kind,precision", CASES)
def test_split_matches_full_box(grid, cell, n, layers, copies, kind, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0904_4887_gb300 import GPSolver
    at = W.slab_atoms(cell, n, layers, seed=6)
    pos = _t(np.concatenate([at.pos + [c * cell[0], 0.0, 0.0] for c in range(copies)]))
    rv = _t(np.tile(W.vdw_radii(at.Z), copies))
    gauss = _t(np.tile(np.stack([at.Z, at.sigma_core, at.sigma_cloud], 1), (copies, 1)))
    cell = (copies * cell[0], cell[1], cell[2])
    zs = np.sort(at.pos[:, 2])
    per = len(zs) // layers
    phis = []
    for split in (0, 1):
        s = GPSolver(grid, cell, precision=precision, split=split, kind=kind, zlim=0.5 * (zs[per - 1] + zs[per]))
        s.set_atoms(pos, radii=rv)
        rho = s.build_rho(pos, gauss)
        phis.append(s.solve(rho, tol=1e-12))
        if split:
            assert s.stats().split_active == 1
    assert float((phis[0] - phis[1]).abs().max()) < 1e-8 * float(phis[0].abs().max())
