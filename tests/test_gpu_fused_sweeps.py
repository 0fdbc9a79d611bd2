"""The fused sweeps of the FP32 middle levels and small finest levels (one or two sweeps a launch on tiles
with a halo, the interpolation in the first launch after the coarse correction,
residual and restriction in one) against the FP64 hierarchy, which runs every
half sweep as a launch of its own. The residual after the first outer
correction is that of the same iteration in both (with the split, its plain
coupling: GMRES would stop at a step of its own in each precision): it stays near 1e-4 of the
right side here, so FP32's own rounding (1e-7 of it per operator) is below 1e-2
of that residual, and a wrong point, colour or halo moves it by more.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as W

pytestmark = pytest.mark.gpu

# grid, cell, split: level 1 ragged on the 8-point tiles, at the line to the one-CTA bottom, above one wave of tiles
CASES = [
    ((24, 24, 48), (10.0, 10.0, 20.0), 0),
    ((16, 16, 32), (8.5, 8.5, 16.0), 0),        # 1024 points: the bottom takes level 1
    ((48, 32, 96), (10.0, 8.5, 24.0), 0),
    ((96, 64, 96), (12.0, 9.0, 18.0), 0),       # level 1 of 73,728 points
    ((24, 32, 64), (9.0, 10.0, 22.0), 1),       # Dirichlet walls in z
    ((32, 24, 96), (10.0, 9.0, 28.0), 1),
    ((32, 32, 32), (10.0, 10.0, 12.0), 0),      # one-CTA bottom: its largest level, 4096 points
    ((32, 32, 96), (10.0, 10.0, 28.0), 0),      # two pairs a thread (1536 points), periodic and between walls
    ((32, 32, 96), (10.0, 10.0, 28.0), 1),
]


def _t(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("nu1,nu2,nu_coarse", [(2, 2, 4), (1, 1, 1), (2, 1, 3), (1, 2, 2), (3, 2, 5), (2, 2, 0)])
@pytest.mark.parametrize("grid,cell,split", CASES)
def test_first_correction_matches_fp64(grid, cell, split, nu1, nu2, nu_coarse):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0904_4887_gb300 import GPSolver
    at = W.slab_atoms(cell, 2, 4, seed=9)
    pos = _t(at.pos)
    gauss = _t(np.stack([at.Z, at.sigma_core, at.sigma_cloud], 1))
    got = []
    for precision in (0, 1):
        s = GPSolver(grid, cell, precision=precision, split=split, nu1=nu1, nu2=nu2, nu_coarse=nu_coarse, inner=3,
                     accel=0, max_outer=2)
        s.set_atoms(pos)
        rho = s.build_rho(pos, gauss)
        s.solve(rho, tol=1e-12, check=False)
        assert s.stats().history_len == 2
        assert s.stats().split_active == split
        got.append(s.stats().history[1])
    assert got[0] > 1e-6
    assert abs(got[1] - got[0]) < 1e-2 * got[0]
