"""Captured work follows what it depends on. A context whose smoother tile changes
between two dielectrics launches as many kernels per solve as a fresh context
with that tile: max_outer and restart bound every loop here, so the counts do not
hang on rounding. A context whose dry band has moved by whole planes takes the
GMRES steps of a fresh one (the same problem, translated).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as W

pytestmark = pytest.mark.gpu

GRID, CELL = (24, 24, 48), (10.0, 10.0, 20.0)


def _inputs(dz=0.0):
    at = W.slab_atoms(CELL, 2, 3, seed=9)
    at_pos = np.ascontiguousarray(at.pos) + np.array([0.0, 0.0, dz])
    pos = torch.tensor(at_pos, dtype=torch.float64, device="cuda")
    gauss = torch.tensor(np.stack([at.Z, at.sigma_core, at.sigma_cloud], 1), dtype=torch.float64, device="cuda")
    return pos, gauss


def _launches(gp, s, path, pos, rho):
    phi = s.zeros()
    n = gp.gp_launch_count()
    if path == "sixth":
        s.ctx.gp_solve6(rho, phi, 1e-14, check=False)
    else:
        s.solve(rho, phi, tol=1e-14, check=False)
    return gp.gp_launch_count() - n


@pytest.mark.parametrize("path,params", [("full", {}), ("graph", {"graph_outer": 1}), ("split", {"split": 1, "restart": 2}),
                                         ("sixth", {"restart": 3})])
def test_a_new_smoother_tile_is_the_one_that_runs(path, params):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0904_4887_gb300 import GPSolver, gp
    pos, gauss = _inputs()
    s = GPSolver(GRID, CELL, max_outer=2, **params)
    rho = s.build_rho(pos, gauss)
    got, want = [], []
    for shape in (-1, 0, -1):
        s.set_atoms(pos, sweep_shape=shape)
        assert s.stats().sweep_shape == shape
        got.append(_launches(gp, s, path, pos, rho))
        f = GPSolver(GRID, CELL, max_outer=2, sweep_shape=shape, **params)
        f.set_atoms(pos)
        want.append(_launches(gp, f, path, pos, rho))
    assert want[0] != want[1]
    assert got == want


def test_a_moved_dry_band():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0904_4887_gb300 import GPSolver
    s = GPSolver(GRID, CELL, split=1)
    steps, first = [], []
    for k in (0, 9):
        pos, gauss = _inputs(k * CELL[2] / GRID[2])
        f = GPSolver(GRID, CELL, split=1)
        for g in (s, f):
            g.set_atoms(pos)
            g.solve(g.build_rho(pos, gauss), tol=1e-10)
            assert g.stats().split_active
            steps.append(g.stats().vcycles)
        first.append(s.stats().band_first)
    assert first[1] == (first[0] + 9) % GRID[2]
    assert max(steps) - min(steps) <= 2               # one GMRES step of two V-cycles, for rounding
