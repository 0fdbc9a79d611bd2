"""Eq. 9-10 with beta below 1/2 and a tight tail: eps follows gamma^(2 beta), whose slope
is unbounded where gamma vanishes, here in 100 A of solvent between a slab's images.
The sum's terms are positive and each is right to a few units of FP32 where gamma is
below 1e-7 (4 * 2^-24 of it), better elsewhere: eps within beta * sqrt(1e-7) * 2.4e-7 =
1.9e-11 of its largest value for beta = 1/4. Points with gamma below 1e-18 are left out:
there one image at the radius, which one side may take and the other not, counts.
Elsewhere such an image (7.4 exp(-46) = 8e-20) moves eps by beta * 8e-20 / sqrt(1e-18) * 2
= 4e-11: held to 1e-10.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads as W
from oracle import gp_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("beta,tail", [(0.25, 1e-16), (0.25, 1e-15)])
def test_eps_of_a_vanishing_gamma(beta, tail):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0904_4887_gb300 import GPSolver
    grid, cell = (16, 16, 192), (8.0, 8.0, 110.0)
    at = W.slab_atoms(cell, 1, 2, seed=4)
    rv = W.vdw_radii(at.Z)
    s = GPSolver(grid, cell, kind=1, beta=beta, gamma_tail=tail)
    s.set_atoms(torch.tensor(np.ascontiguousarray(at.pos), dtype=torch.float64, device="cuda"),
                radii=torch.tensor(rv, dtype=torch.float64, device="cuda"))
    p = O.GammaParams(beta=beta, tail=tail)
    gamma = O.dummy_density(grid, cell, at.pos, rv, p)
    eps = O.eps_of_gamma(gamma, p)
    assert gamma.min() < 1e-18
    assert np.max(np.abs(s.eps().cpu().numpy() - eps)[gamma > 1e-18]) < 1e-10 * np.max(eps)
