"""The work that users of the solver have it do, as measurable cases.

Every case is a periodic slab of atoms in solvent: atoms and Gaussian charges
are on the device, the solver object is kept between calls, and one pass is
what a program runs per configuration of the atoms. Sizes are those of the
repository's workloads, tests and benchmark, with small, anisotropic and
defective slabs beside them. Paths:

  step     set_atoms + build_rho + solve from zero + energy_forces (kind 0, 1 or 2 dielectric)
  frame    the same for the next frame of a trajectory, warm-started from the last frame's phi
  adjoint  poisson_energy through torch.autograd, with dE/drho and dE/dR
  sixth    the sixth-order solve, its adjoint, energy and forces
  vacuum   the FFT vacuum solve (FP64 or FP32)
"""
import math

import numpy as np
import torch

import paper_0904_4887_gb300 as gp

DEV = "cuda"
EXTENTS = (16, 24, 32, 48, 64, 96, 128, 192, 256, 384)
EPS0, R0, W, RCUT, BETA = 78.36, 2.5, 0.5, 6.0, 2.4     # the library's defaults
TOL = 1e-10                                             # GPSolver.solve's default


def _case(path, grid, cell, layers, **more):
    c = {"path": path, "nx": grid[0], "ny": grid[1], "nz": grid[2], "lx": cell[0], "ly": cell[1], "lz": cell[2],
         "layers": layers, "vacancies": 0, "widths": "fixed", "precision": 1, "kind": 0, "split": 0, "levels": 0}
    c.update(more)
    return c


def listed():
    full = dict(grid=(192, 192, 384), cell=(26.0, 26.0, 52.0), layers=4, widths="drawn")
    got = [
        # the smallest grid a first look uses: launches and host round trips are all of it
        _case("step", (24, 24, 48), (10.0, 10.0, 20.0), 3, name="step_mixed_24x24x48"),
        # the small validation slab, FP64 throughout
        _case("step", (32, 32, 64), (10.0, 10.0, 20.0), 3, precision=0, name="step_fp64_32x32x64"),
        # the paper's slab cell on the nearest grid, unequal extents and spacings, a defect
        _case("step", (96, 64, 192), (10.24, 7.56, 17.82), 4, vacancies=1, name="step_mixed_96x64x192"),
        # a production configuration: the benchmark's slab, from zero
        _case("step", name="step_mixed_192x192x384", **full),
        # one frame of molecular dynamics
        _case("frame", (128, 128, 256), (13.0, 13.0, 26.0), 8, name="frame_mixed_128x128x256"),
        # a differentiable energy in a larger torch program
        _case("adjoint", (64, 64, 128), (10.0, 10.0, 20.0), 6, precision=0, name="adjoint_fp64_64x64x128"),
        # the dry/wet split (Scheme 1) in FP64, five levels
        _case("step", (96, 96, 192), (13.0, 13.0, 40.0), 4, precision=0, split=1, levels=5,
              name="split_fp64_96x96x192"),
        # the paper's dielectric (Eq. 9-10) on the production configuration
        _case("step", kind=1, name="eq9_mixed_192x192x384", **full),
        # the paper's slab run: one face kept dry (Eq. 19), the split on the rest
        _case("step", (96, 96, 192), (13.0, 13.0, 40.0), 4, kind=2, split=1, name="eq19_split_96x96x192"),
        # the sixth-order stencil (Eq. 16-18) with its forces
        _case("sixth", (64, 64, 128), (10.0, 10.0, 20.0), 6, name="sixth_mixed_64x64x128"),
        # vacuum reference energies (Eq. 15), production grid in FP64 and an FP32 one
        _case("vacuum", precision=0, name="vacuum_fp64_192x192x384", **full),
        _case("vacuum", (128, 128, 256), (13.0, 13.0, 26.0), 8, name="vacuum_fp32_128x128x256"),
    ]
    return got


def _coarsens(n):
    """Whether a multigrid hierarchy exists: halving while every extent is even ends at <= 512 points."""
    n = list(n)
    while all(v % 2 == 0 and v >= 4 for v in n) and n[0] * n[1] * n[2] > 64:
        n = [v // 2 for v in n]
    return n[0] * n[1] * n[2] <= 512


def _image_pairs(c):
    """(grid point, atom image) pairs within 41 A, the reach of the Eq. 9 sum at its default tail."""
    return c["nx"] * c["ny"] * c["nz"] * _atom_count(c) * (4 * math.pi / 3 * 41.0 ** 3) / (c["lx"] * c["ly"] * c["lz"])


def draw(rng):
    path, kind, split, precision, most, least = rng.choice([
        ("step", 0, 0, 1, 14.2e6, 2e4), ("step", 0, 0, 1, 14.2e6, 2e4), ("step", 0, 0, 0, 2e6, 2e4),
        ("frame", 0, 0, 1, 4.2e6, 1e5), ("adjoint", 0, 0, 0, 1.2e6, 3e4), ("step", 0, 1, 0, 2e6, 1e5),
        ("step", 0, 1, 1, 4.2e6, 1e5), ("step", 1, 0, 1, 2e6, 2e4), ("step", 2, 0, 1, 2e6, 2e4),
        ("step", 2, 1, 1, 2e6, 1e5), ("sixth", 0, 0, 1, 1.2e6, 2e4), ("vacuum", 0, 0, 0, 14.2e6, 2e4),
        ("vacuum", 0, 0, 1, 14.2e6, 2e4)])
    while True:
        want = math.exp(rng.uniform(math.log(least), math.log(most)))
        grid = tuple(rng.choice(EXTENTS) for _ in range(3))
        pts = grid[0] * grid[1] * grid[2]
        if not (0.5 * want <= pts <= 2.0 * want and least <= pts <= most and _coarsens(grid)):
            continue
        h = math.exp(rng.uniform(math.log(0.1), math.log(0.4)))
        cell = tuple(round(n * h * rng.uniform(0.9, 1.15), 2) for n in grid)
        layers = rng.randint(3, 8)
        if not (7.5 <= min(cell[:2]) and max(cell) <= 56.0 and cell[2] >= layers + 9.0):
            continue
        c = _case(path, grid, cell, layers, kind=kind, split=split, precision=precision,
                  vacancies=rng.randint(0, 3), widths="drawn" if min(cell) >= 8.1 and rng.random() < 0.5 else "fixed")
        if kind and _image_pairs(c) > 1.6e10:
            continue
        return c


# ---------------------------------------------------------------- inputs
def _repeats(c):
    return max(1, round(c["lx"] / 4.6)), max(1, round(c["ly"] / 4.6))


def _atom_count(c):
    n1, n2 = _repeats(c)
    return 2 * n1 * n2 * c["layers"] - c["vacancies"]


def _atoms(c, seed):
    """A compact staggered two-species slab centred in the cell, jittered, with some atoms missing:
    numpy arrays pos (n, 3), gauss (n, 3) = (Z, sigma_core, sigma_cloud), rvdw (n,), zlim, velocities (n, 3) in A/fs."""
    rng = np.random.default_rng(seed)
    cell = np.array([c["lx"], c["ly"], c["lz"]])
    n1, n2 = _repeats(c)
    a, b = cell[0] / n1, cell[1] / n2
    pos, Z = [], []
    for l in range(c["layers"]):
        z = cell[2] / 2 + (l - (c["layers"] - 1) / 2)
        for i in range(n1):
            for j in range(n2):
                for q, s in ((4.0, 0.0), (6.0, 0.5)):
                    pos.append(((i + s + 0.5 * (l % 2)) * a, (j + s) * b, z))
                    Z.append(q)
    pos, Z = np.array(pos), np.array(Z)
    pos = np.mod(pos + rng.uniform(-0.05, 0.05, pos.shape), cell)
    n = len(Z)
    if c["widths"] == "drawn":
        core, cloud = rng.uniform(0.3, 1.0, n), rng.uniform(0.3, 1.0, n)
    else:
        core, cloud = np.full(n, 0.3), np.full(n, 0.8)
    keep = np.sort(rng.permutation(n)[: n - c["vacancies"]])
    gauss = np.stack([Z, core, cloud], 1)
    rvdw = np.where(Z == 6.0, 1.52, 2.0)
    zs = np.sort(pos[:, 2])
    per = n // c["layers"]
    zlim = float(0.5 * (zs[per - 1] + zs[per]))          # the lowest layer excludes the solvent below it
    mass = np.where(Z == 6.0, 15.999, 47.867)
    vel = rng.standard_normal((n, 3)) * np.sqrt(8.617333262e-5 * 300.0 / mass * 9.648533212e-3)[:, None]
    return pos[keep], gauss[keep], rvdw[keep], zlim, vel[keep]


def _moved(c, pos, vel):
    return np.mod(pos + 0.5 * vel, np.array([c["lx"], c["ly"], c["lz"]]))     # half a femtosecond on


def _t(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device=DEV)


def _density(c, seed):
    """A charge density of the slab's kind for the vacuum solve: smoothed noise of zero mean."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    f = torch.randn((c["nz"], c["ny"], c["nx"]), dtype=torch.float64, device=DEV, generator=g)
    for ax in range(3):
        f = f + torch.roll(f, 1, ax)
    return f - f.mean()


def prepare(case, seed):
    c = case
    grid, cell = (c["nx"], c["ny"], c["nz"]), (c["lx"], c["ly"], c["lz"])
    if c["path"] == "vacuum":
        f = _density(c, seed)
        return {"case": c, "solver": gp.GPSolver(grid, cell, precision=c["precision"]),
                "src": f if c["precision"] == 0 else f.float()}
    pos, gauss, rvdw, zlim, vel = _atoms(c, seed)
    more = {"graph_outer": 2, "inner": 4} if c["path"] == "frame" else {}
    s = gp.GPSolver(grid, cell, precision=c["precision"], kind=c["kind"], split=c["split"], levels=c["levels"],
                    zlim=zlim, **more)
    st = {"case": c, "solver": s, "pos": _t(pos), "gauss": _t(gauss), "rho": s.zeros()}
    if c["kind"]:
        s.ctx.gp_set_vdw_radii(_t(rvdw))
    if c["path"] == "frame":
        # the frame before, as the program has it: its phi starts this frame's solve
        s.set_atoms(st["pos"])
        s.build_rho(st["pos"], st["gauss"], out=st["rho"])
        st["last"] = s.solve(st["rho"], tol=TOL)
        st["phi"] = s.zeros()
        st["pos"] = _t(_moved(c, pos, vel))
    elif c["path"] == "adjoint":
        s.build_rho(st["pos"], st["gauss"], out=st["rho"])
        st["pos"].requires_grad_(True)
        st["rho"].requires_grad_(True)
    return st


# ---------------------------------------------------------------- one pass
def run(state):
    s, c = state["solver"], state["case"]
    if c["path"] == "vacuum":
        return s.fft_poisson(state["src"]) if c["precision"] == 0 else s.fft_poisson_f32(state["src"])
    pos, gauss, rho = state["pos"], state["gauss"], state["rho"]
    if c["path"] == "adjoint":
        E, phi = gp.poisson_energy(pos, rho, s, tol=TOL)
        gpos, grho = torch.autograd.grad(E, (pos, rho))
        return {"energy": E.detach(), "phi": phi, "grad_pos": gpos, "grad_rho": grho}
    s.set_atoms(pos)
    s.build_rho(pos, gauss, out=rho)
    if c["path"] == "sixth":
        phi, mu = s.solve6(rho, tol=TOL)
        lam, _ = s.adjoint6(rho, tol=TOL)          # its multiplier is zero for a neutral rho
        E, F = s.energy_forces6(phi, mu, lam, rho, gauss)
        return {"rho": rho, "phi": phi, "mu": mu, "lam": lam, "energy": E, "forces": F}
    if c["path"] == "frame":
        phi = state["phi"]
        phi.copy_(state["last"])
        s.solve(rho, phi, tol=TOL)
    else:
        phi = s.solve(rho, tol=TOL)
    E, E2, F = s.energy_forces(phi, rho, gauss)
    return {"rho": rho, "phi": phi, "energy": E, "field_energy": E2, "forces": F}


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    """Bytes: the grid-sized inputs and outputs, and per solve one reading of eps, rho and phi for the residual that
    accepts it. Flops: the 7-point (19-point) residual, the FFT's butterflies, and one short evaluation per (point,
    atom) pair of the dielectric, the charge and the two force terms where they are not negligible."""
    c = case
    n = c["nx"] * c["ny"] * c["nz"]
    if c["path"] == "vacuum":
        return {"bytes": 2.0 * n * (8 if c["precision"] == 0 else 4), "flops": 5.0 * n * math.log2(n)}
    dv = c["lx"] * c["ly"] * c["lz"] / n
    at = _atom_count(c)
    diel = at * 4 * math.pi / 3 * RCUT ** 3 / dv if c["kind"] == 0 else at * 4 * math.pi / 3 * 10.0 ** 3 / dv
    fields = 8.0 * n * (8 if c["path"] == "sixth" else 5)
    flops = 10.0 * diel * 2 + n * (200.0 if c["path"] == "sixth" else 25.0)
    return {"bytes": fields, "flops": flops}


# ---------------------------------------------------------------- the same in 64 bits, plainly
def _windows(center, reach, n, h, L):
    """Slices of one axis within `reach` of `center`'s images, as (first, last+1, displacement tensor)."""
    got = []
    for m in range(-int(math.ceil(reach / L)) - 1, int(math.ceil(reach / L)) + 2):
        x = center + m * L
        lo, hi = max(0, math.ceil((x - reach) / h)), min(n - 1, math.floor((x + reach) / h))
        if lo <= hi:
            got.append((lo, hi + 1, torch.arange(lo, hi + 1, dtype=torch.float64, device=DEV) * h - x))
    return got


def _boxes(c, p, reach):
    """The grid boxes within `reach` of one atom's images: ((z, y, x) slices, displacements)."""
    ax = [_windows(p[k], reach, c["n" + "xyz"[k]], c["l" + "xyz"[k]] / c["n" + "xyz"[k]], c["l" + "xyz"[k]]) for k in range(3)]
    for z0, z1, dz in ax[2]:
        for y0, y1, dy in ax[1]:
            for x0, x1, dx in ax[0]:
                near = sum(min(abs(float(d[0])), abs(float(d[-1]))) ** 2 if float(d[0]) * float(d[-1]) > 0 else 0.0 for d in (dx, dy, dz))
                if near < reach * reach:
                    yield (slice(z0, z1), slice(y0, y1), slice(x0, x1)), (dx[None, None, :], dy[None, :, None], dz[:, None, None])


def _switch(d):
    return 0.5 * torch.special.erfc(-(d - R0) / W)


def _erf_product(c, pos):
    P = torch.ones((c["nz"], c["ny"], c["nx"]), dtype=torch.float64, device=DEV)
    for p in pos:
        for box, (dx, dy, dz) in _boxes(c, p, RCUT):
            d = torch.sqrt(dx * dx + dy * dy + dz * dz)
            P[box] *= torch.where(d < RCUT, _switch(d), torch.ones_like(d))
    return P


def _decay(d, rv):
    return torch.exp(rv - d)


def _below(c, p, zlim):
    """How many planes lie below an atom that excludes the solvent under it (0: it does not)."""
    if c["kind"] != 2 or p[2] > zlim:
        return 0
    return int(math.ceil(p[2] / (c["lz"] / c["nz"])))


def _nearest(c, p):
    out = []
    for k in range(3):
        n, L = c["n" + "xyz"[k]], c["l" + "xyz"[k]]
        d = torch.arange(n, dtype=torch.float64, device=DEV) * (L / n) - p[k]
        out.append(d - L * torch.round(d / L))
    return out[0][None, None, :], out[1][None, :, None], out[2][:, None, None]


REACH9 = 40.0


def _gamma(c, pos, rvdw, zlim):
    g = torch.zeros((c["nz"], c["ny"], c["nx"]), dtype=torch.float64, device=DEV)
    for p, rv in zip(pos, rvdw):
        k0 = _below(c, p, zlim)
        for box, (dx, dy, dz) in _boxes(c, p, REACH9):
            d = torch.sqrt(dx * dx + dy * dy + dz * dz)
            t = _decay(d, rv)
            t[d > REACH9] = 0
            skip = max(0, min(k0, box[0].stop) - box[0].start)
            if skip < t.shape[0]:
                g[box][skip:] += t[skip:]
        if k0:
            dx, dy, dz = _nearest(c, p)
            g[:k0] += torch.exp(torch.sqrt(dx * dx + dy * dy + dz[:k0] ** 2) - rv)
    return g


def _eps(c, pos, rvdw, zlim):
    """eps and what each atom's motion changes of it: the product of switches, or d eps / d gamma."""
    if c["kind"] == 0:
        P = _erf_product(c, pos)
        return 1.0 + (EPS0 - 1.0) * P, P
    g = _gamma(c, pos, rvdw, zlim)
    g2 = g ** (2 * BETA)
    sat = g2 > 1e17 if c["kind"] == 2 else g2 > 1e300
    eps = torch.where(sat, torch.ones_like(g), 1.0 + (EPS0 - 1.0) / (1.0 + g2))
    de = -(EPS0 - 1.0) * 2 * BETA * (g2 / g) / (1.0 + g2) ** 2
    return eps, torch.where(sat, torch.zeros_like(de), de)


def _eps_pull(c, pos, rvdw, zlim, fac, weight):
    """sum_i weight_i d eps_i / d R_a for every atom."""
    out = torch.zeros((len(pos), 3), dtype=torch.float64, device=DEV)
    wf = weight * fac * ((EPS0 - 1.0) if c["kind"] == 0 else 1.0)
    for a, p in enumerate(pos):
        reach = RCUT if c["kind"] == 0 else REACH9
        k0 = _below(c, p, zlim)
        for box, (dx, dy, dz) in _boxes(c, p, reach):
            d = torch.sqrt(dx * dx + dy * dy + dz * dz).clamp_min(1e-12)
            if c["kind"] == 0:
                t = -torch.exp(-((d - R0) / W) ** 2) / (W * math.sqrt(math.pi)) / _switch(d) / d
            else:
                t = _decay(d, rvdw[a]) / d
                t[: max(0, min(k0, box[0].stop) - box[0].start)] = 0
            t = torch.where(d < reach, t * wf[box], torch.zeros_like(d))
            for k, dd in enumerate((dx, dy, dz)):
                out[a, k] += (t * dd).sum()
        if k0:
            dx, dy, dz = _nearest(c, p)
            dz = dz[:k0]
            d = torch.sqrt(dx * dx + dy * dy + dz * dz).clamp_min(1e-12)
            t = torch.where(wf[:k0] != 0, -torch.exp((d - rvdw[a]).clamp_max(300.0)) / d * wf[:k0], torch.zeros_like(d))
            for k, dd in enumerate((dx, dy, dz)):
                out[a, k] += (t * dd).sum()
    return out


def _axis_gaussian(n, L, x, sigma, slope):
    """One axis of a Gaussian cut at 8 sigma, summed over images; with `slope` its derivative by the centre."""
    g = torch.arange(n, dtype=torch.float64, device=DEV) * (L / n)
    out = torch.zeros(n, dtype=torch.float64, device=DEV)
    for m in range(-1, 2):
        d = g - (x + m * L)
        e = torch.where(d.abs() < 8 * sigma, torch.exp(-0.5 * (d / sigma) ** 2), torch.zeros_like(d))
        out += e * d / sigma ** 2 if slope else e
    return out


def _factors(c, p, sigma):
    val = [_axis_gaussian(c["n" + "xyz"[k]], c["l" + "xyz"[k]], p[k], sigma, False) for k in range(3)]
    der = [_axis_gaussian(c["n" + "xyz"[k]], c["l" + "xyz"[k]], p[k], sigma, True) for k in range(3)]
    return val, der, (2 * math.pi * sigma ** 2) ** -1.5


def _rho(c, pos, gauss):
    rho = torch.zeros((c["nz"], c["ny"], c["nx"]), dtype=torch.float64, device=DEV)
    for p, (Z, s1, s2) in zip(pos, gauss):
        for q, sg in ((Z, s1), (-Z, s2)):
            (X, Y, V), _, nrm = _factors(c, p, sg)
            rho.addcmul_((q * nrm * V)[:, None, None], Y[:, None] * X[None, :])
    return rho - rho.mean()


def _rho_pull(c, pos, gauss, weight):
    """sum_i weight_i d rho_i / d R_a for a weight of zero mean."""
    out = torch.zeros((len(pos), 3), dtype=torch.float64, device=DEV)
    for a, (p, (Z, s1, s2)) in enumerate(zip(pos, gauss)):
        for q, sg in ((Z, s1), (-Z, s2)):
            (X, Y, V), (dX, dY, dV), nrm = _factors(c, p, sg)
            wz, wdz = torch.tensordot(V, weight, 1), torch.tensordot(dV, weight, 1)
            out[a] += q * nrm * torch.stack([(Y @ (wz @ dX)), (dY @ (wz @ X)), (Y @ (wdz @ X))])
    return out


def _spacing(c):
    return c["lx"] / c["nx"], c["ly"] / c["ny"], c["lz"] / c["nz"]


def _A(c, eps, u):
    out = torch.zeros_like(u)
    for ax, h in zip((2, 1, 0), _spacing(c)):
        flux = (eps + torch.roll(eps, -1, ax)) * (torch.roll(u, -1, ax) - u) * (0.5 / (h * h))
        out += flux - torch.roll(flux, 1, ax)
    return out


def _symbol(c, of):
    s = [of(2 * math.pi * torch.arange(n, dtype=torch.float64, device=DEV) / n) / h ** 2
         for n, h in zip((c["nx"], c["ny"], c["nz"]), _spacing(c))]
    s = s[2][:, None, None] + s[1][None, :, None] + s[0][None, None, : c["nx"] // 2 + 1]
    s[0, 0, 0] = 1.0
    return s


def _inverse(c, sym, src):
    f = torch.fft.rfftn(src) / sym
    f[0, 0, 0] = 0
    return torch.fft.irfftn(f, s=src.shape)


def _second(t):
    return -4 * torch.sin(0.5 * t) ** 2


def _solve(c, eps, rho):
    """Conjugate gradients, preconditioned by the vacuum solve scaled by eps^-1/2 on either side."""
    sym, w = _symbol(c, _second), eps.rsqrt()
    b = 4 * math.pi * rho
    x, r, p, rz = torch.zeros_like(b), b.clone(), None, None
    stop = 1e-14 * float(b.norm())
    for it in range(400):
        z = -w * _inverse(c, sym, w * r)
        new = torch.dot(r.flatten(), z.flatten())
        p = z if p is None else z + (new / rz) * p
        rz = new
        q = -_A(c, eps, p)
        al = rz / torch.dot(p.flatten(), q.flatten())
        x += al * p
        r -= al * q
        if it % 8 == 7:
            r = b + _A(c, eps, x) if it % 64 == 63 else r
            if float(r.norm()) < max(stop, 3e-14 * float(b.norm())):
                break
    return x - x.mean()


FD1 = (0.0, 3 / 4, -3 / 20, 1 / 60)
FD2 = (-49 / 18, 3 / 2, -3 / 20, 1 / 90)


def _d1(c, u, ax):
    h = _spacing(c)[2 - ax]
    return sum(FD1[m] * (torch.roll(u, -m, ax) - torch.roll(u, m, ax)) for m in (1, 2, 3)) / h


def _d2(c, u, ax):
    h = _spacing(c)[2 - ax]
    return (FD2[0] * u + sum(FD2[m] * (torch.roll(u, -m, ax) + torch.roll(u, m, ax)) for m in (1, 2, 3))) / h ** 2


def _A6(c, eps, u, adj):
    if adj:
        return sum(_d2(c, eps * u, ax) - _d1(c, _d1(c, eps, ax) * u, ax) for ax in range(3))
    return sum(_d1(c, eps, ax) * _d1(c, u, ax) + eps * _d2(c, u, ax) for ax in range(3))


def _solve6(c, eps, b, adj):
    """Restarted GMRES on A6 x + m eps = b, sum x = 0 (adj: A6' x + m = b, sum eps x = 0), on unknowns (x, m),
    preconditioned by the FFT inverse of D2 between factors eps^-1/2."""
    sym = _symbol(c, lambda t: FD2[0] + 2 * sum(FD2[m] * torch.cos(m * t) for m in (1, 2, 3)))
    n, shape = b.numel(), b.shape

    def K(v):
        x, m = v[:n].view(shape), v[n]
        if adj:
            return torch.cat([(_A6(c, eps, x, True) + m).flatten(), (eps * x).sum().view(1)])
        return torch.cat([(_A6(c, eps, x, False) + m * eps).flatten(), x.sum().view(1)])

    w, weps = eps.rsqrt(), eps.sum()

    def M(v):
        r, s = v[:n].view(shape), v[n]
        m = r.mean() if adj else (r.sum() / weps)
        r = r - m if adj else r - m * eps
        x = w * _inverse(c, sym, w * r)
        x = x + (s - (eps * x).sum()) / weps if adj else x + (s - x.sum()) / n
        return torch.cat([x.flatten(), m.view(1)])

    rhs = torch.cat([b.flatten(), torch.zeros(1, dtype=torch.float64, device=DEV)])
    v, nb = torch.zeros_like(rhs), float(rhs.norm())
    for _ in range(12):
        r = rhs - K(v)
        beta = float(r.norm())
        if beta < 2e-14 * nb:
            break
        V, Z, H = [r / beta], [], np.zeros((81, 80))
        for j in range(80):
            Z.append(M(V[j]))
            w_ = K(Z[j])
            for _twice in range(2):
                h = torch.stack(V) @ w_
                w_ = w_ - h @ torch.stack(V)
                H[: j + 1, j] += h.cpu().numpy()
            H[j + 1, j] = float(w_.norm())
            V.append(w_ / H[j + 1, j])
            if j % 8 == 7 or j == 79:
                e = np.zeros(j + 2)
                e[0] = beta
                y, *_r = np.linalg.lstsq(H[: j + 2, : j + 1], e, rcond=None)
                if np.linalg.norm(e - H[: j + 2, : j + 1] @ y) < 1e-14 * nb:
                    break
        v = v + _t(y) @ torch.stack(Z[: len(y)])
    return v[:n].view(shape), v[n]


def _field_weight(c, phi):
    """Half the squared face gradients around each point."""
    out = torch.zeros_like(phi)
    for ax, h in zip((2, 1, 0), _spacing(c)):
        g = ((torch.roll(phi, -1, ax) - phi) / h) ** 2
        out += 0.5 * (g + torch.roll(g, 1, ax))
    return out


def exact(case, seed):
    c = case
    n = c["nx"] * c["ny"] * c["nz"]
    if c["path"] == "vacuum":
        f = _density(c, seed)
        return _inverse(c, _symbol(c, _second), f if c["precision"] == 0 else f.float().double())
    if c["kind"] and _image_pairs(c) > 1.2e10:
        return None                      # the plain image sum would take too long
    pos, gauss, rvdw, zlim, vel = _atoms(c, seed)
    if c["path"] == "frame":
        pos = _moved(c, pos, vel)
    hx, hy, hz = _spacing(c)
    dv = hx * hy * hz
    eps, fac = _eps(c, pos, rvdw, zlim)
    rho = _rho(c, pos, gauss)
    if c["path"] == "sixth":
        phi, mu = _solve6(c, eps, -4 * math.pi * rho, False)
        lam, _ = _solve6(c, eps, rho, True)
        g = sum(lam * _d2(c, phi, ax) - _d1(c, lam * _d1(c, phi, ax), ax) for ax in range(3))
        wr = 0.5 * (phi - 4 * math.pi * lam)
        F = 0.5 * dv * _eps_pull(c, pos, rvdw, zlim, fac, g + mu * lam) - dv * _rho_pull(c, pos, gauss, wr - wr.mean())
        return {"rho": rho, "phi": phi, "mu": mu, "lam": lam, "energy": float(0.5 * dv * (rho * phi).sum()),
                "forces": F}
    phi = _solve(c, eps, rho)
    E = float(0.5 * dv * (rho * phi).sum())
    wf = _field_weight(c, phi)
    Ge = -dv / (8 * math.pi) * _eps_pull(c, pos, rvdw, zlim, fac, wf)
    if c["path"] == "adjoint":
        return {"energy": torch.tensor(E, dtype=torch.float64), "phi": phi, "grad_pos": Ge, "grad_rho": dv * phi}
    E2 = float(dv / (8 * math.pi) * (eps * wf).sum())
    F = -(Ge + dv * _rho_pull(c, pos, gauss, phi))
    return {"rho": rho, "phi": phi, "energy": E, "field_energy": E2, "forces": F}
