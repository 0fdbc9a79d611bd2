"""The two routes of the Eq. 9 sum against each other, through the C ABI: near
images plus a Fourier series (tails up to 1e-12) and the direct image sum
(looser tails). Tails of 1e-12 and 1.001e-12 put the cut-off radii within 1e-3 A
of each other, so the two answers differ by their own errors alone: each is
documented within 1e-13 of the largest eps, and within 1e-11 of the largest
force (the direct sum's far pairs are FP32 there).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as W

pytestmark = pytest.mark.gpu

# grid, cell, lattice repeats, layers, atoms kept, kind, share of the layers below z_lim (kind 2)
CASES = [
    ((16, 16, 32), (7.0, 7.0, 14.0), 1, 2, 1, 1, 0.0),        # one atom, images in every direction
    ((24, 24, 48), (10.0, 10.0, 20.0), 2, 3, 23, 1, 0.0),
    ((32, 64, 16), (12.0, 9.0, 13.0), 2, 4, 32, 1, 0.0),      # unequal extents and spacings
    ((64, 32, 48), (26.0, 13.0, 16.0), 4, 4, 128, 1, 0.0),    # 128 atoms: one staged chunk exactly
    ((64, 32, 48), (26.0, 13.0, 16.0), 5, 3, 129, 1, 0.0),    # and one more than that
    ((32, 32, 48), (14.4, 14.4, 21.6), 3, 4, 71, 1, 0.0),     # a coarse grid: a small K, a large near radius
    ((32, 32, 48), (20.0, 20.0, 30.0), 3, 4, 72, 1, 0.0),     # too coarse for the split
    ((24, 24, 48), (10.0, 10.0, 20.0), 2, 4, 32, 2, 0.0),     # Eq. 19 with no lower atom
    ((24, 24, 48), (10.0, 10.0, 20.0), 2, 4, 32, 2, 0.25),    # the lowest layer
    ((24, 24, 48), (10.0, 10.0, 20.0), 2, 4, 31, 2, 0.6),     # several layers: many planes between them
    ((24, 24, 48), (10.0, 10.0, 20.0), 2, 4, 32, 2, 1.0),     # every atom
    ((512, 16, 32), (60.0, 7.0, 14.0), 2, 2, 16, 2, 0.5),     # the longest transform, a thin cell
]


def _t(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("grid,cell,n,layers,keep,kind,low", CASES)
def test_split_and_direct_sums_agree(grid, cell, n, layers, keep, kind, low):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0904_4887_gb300 import GPSolver
    at = W.slab_atoms(cell, n, layers, seed=4)
    pos, rv = _t(at.pos[:keep]), _t(W.vdw_radii(at.Z)[:keep])
    zs = np.sort(at.pos[:keep, 2])
    m = int(round(low * keep))
    zlim = -1.0 if m == 0 else (zs[-1] + 0.1 if m >= keep else 0.5 * (zs[m - 1] + zs[m]))
    gen = torch.Generator(device="cuda").manual_seed(5)
    phi = torch.randn((grid[2], grid[1], grid[0]), dtype=torch.float64, device="cuda", generator=gen)
    got = []
    for tail in (1e-12, 1.001e-12):
        s = GPSolver(grid, cell, kind=kind, zlim=zlim, gamma_tail=tail)
        s.set_atoms(pos, radii=rv)
        _, _, F = s.energy_forces(phi, torch.zeros_like(phi))
        got.append((s.eps(), F))
    (e1, F1), (e2, F2) = got
    assert float((e1 - e2).abs().max()) < 2e-13 * 78.36
    assert float((F1 - F2).abs().max()) < 1e-11 * float(F2.abs().max())
