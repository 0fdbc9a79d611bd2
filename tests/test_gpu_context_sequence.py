"""One context through dielectrics of different kinds, atom counts, tails and radii,
against a fresh context at each step: tables, modes and work arrays kept from one call
to the next serve the next one. eps within 2e-13 of its largest value and the force
within 1e-11 of its largest component, what tests/test_gpu_gamma_split.py allows
between two routes of the same sum (the order of the sums differs from run to run).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as W

pytestmark = pytest.mark.gpu

GRID, CELL = (24, 24, 48), (10.0, 10.0, 20.0)
STEPS = [dict(kind=1, n=24), dict(kind=2, n=32, zlim=9.0), dict(kind=1, n=16), dict(kind=0, n=32),
         dict(kind=1, n=32, gamma_tail=1e-12), dict(kind=2, n=8, zlim=-1.0), dict(kind=2, n=32, zlim=12.0),
         dict(kind=1, n=32, gamma_tail=1e-6), dict(kind=0, n=8, r0=2.0, w=0.4), dict(kind=1, n=24)]


def test_one_context_for_all():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0904_4887_gb300 import GPSolver
    at = W.slab_atoms(CELL, 2, 4, seed=4)
    pos = torch.tensor(np.ascontiguousarray(at.pos), dtype=torch.float64, device="cuda")
    rv = torch.tensor(W.vdw_radii(at.Z), dtype=torch.float64, device="cuda")
    gen = torch.Generator(device="cuda").manual_seed(5)
    phi = torch.randn((GRID[2], GRID[1], GRID[0]), dtype=torch.float64, device="cuda", generator=gen)
    s = GPSolver(GRID, CELL)
    for step in STEPS:
        p = dict(dict(zlim=0.0, gamma_tail=1e-13, r0=2.5, w=0.5), **{k: v for k, v in step.items() if k != "n"})
        n = step["n"]
        got = []
        for c in (s, GPSolver(GRID, CELL)):
            c.set_atoms(pos[:n].contiguous(), radii=rv[:n] if p["kind"] else None, **p)
            _, _, F = c.energy_forces(phi, torch.zeros_like(phi))
            got.append((c.eps(), F))
        (e1, F1), (e2, F2) = got
        assert float((e1 - e2).abs().max()) < 2e-13 * 78.36, step
        assert float((F1 - F2).abs().max()) < 1e-11 * float(F2.abs().max()), step
