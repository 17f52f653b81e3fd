"""The calls of this framework whose speed counts, with inputs, work and FP64 results.

Every case is one call sequence that a user's program makes, at the sizes of the repository's own
workloads (workloads.py, bench.py, the tests) and at odd sizes in between:

  particle  pic_step of one relativistic macro-electron in 2D vacuum (the self-field study)
  scan      pic_batch_step of many independent single-particle runs of uneven size
  phases    pic_gather_push, pic_deposit, pic_field_advance called one by one on a cold plasma
  beam      pic_step of a relativistic beam in plasma, moving window, wake behind the beam
  fields    pic_step of fields alone (vacuum propagation on a large grid)
  grad      StencilLoss.loss_and_grad: forward steps, checkpoints, replay and adjoint steps
  kspace    pic_step of a charged line with the spectral, [k1]_t or PSATD solver
  diag      pic_gauss and pic_diag on a beam-in-plasma state

prepare() draws everything on the GPU from the seed; exact() restates the step in FP64 torch.
"""
import ctypes
import math

import numpy as np
import torch

import paper_1910_13529_gb300 as pic
from paper_1910_13529_gb300.runtime import Simulation, StencilLoss, make_config

HLEN = 24          # taps of the current correction kept on each side
WAKE_CORE = 1.0    # radius of the wake, c/omega_p


def _beam(name, ndim, nz, nx, ny, solver, shape, n_beam, steps, **kw):
    c = dict(kind="beam", ndim=ndim, nz=nz, nx=nx, ny=ny, solver=solver, M=16, shape=shape, n_beam=n_beam,
             steps=steps, ppz=2, ppx=2 if ndim == 2 else 1, filter=False, autotune=True, positions=True)
    c.update(kw)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the paper's single-particle study: a step is a handful of small launches, and a program that
        # looks at the fields after every step makes one call per step
        dict(name="particle_2d", kind="particle", nz=256, nx=128, solver="yee", M=1, shape=1, filter=False, steps=1),
        # the batched scan over gamma, dt and stencil: 256 independent runs, 32 of their 400 steps
        dict(name="scan_2d", kind="scan", n=256, nz_min=128, nz_max=1024, nx_min=64, nx_max=256, shape=1, steps=32),
        # a program with its own loop over the phases of the step (1e6 particles, Yee, linear shapes)
        dict(name="phases_2d", kind="phases", ndim=2, nz=1024, nx=256, ny=1, solver="yee", M=1, shape=1, ppc=4),
        # a beam in plasma at odd sizes (rows not 16-byte aligned), with the current filter, in which
        # most of the other options differ too: Yee, linear shapes, default tile
        _beam("beam_2d_odd", 2, 1001, 237, 1, "yee", 1, 200_000, 2, filter=True, autotune=False),
        # the 2D beam in plasma: 2048 x 512, 4 per cell, 1e6 beam particles, customised stencil
        _beam("beam_2d", 2, 2048, 512, 1, "custom", 2, 1_000_000, 8),
        # a small 3D run with linear shapes and Yee at odd sizes
        _beam("beam_3d_odd", 3, 251, 120, 117, "yee", 1, 300_000, 4, autotune=False),
        # the 3D beam in plasma: 512 x 256 x 256, 2 per cell and 4e6 beam particles, customised stencil
        # (the fields, the current and all momenta come back; cell indices of 71e6 particles are left
        # out, as the rounding of a field decides for a few of them on which side of a cell edge they are)
        _beam("beam_3d", 3, 512, 256, 256, "custom", 2, 4_000_000, 2, positions=False),
        # vacuum propagation on a grid far above L2 with the 32-point axial stencil
        dict(name="fields_2d", kind="fields", ndim=2, nz=8192, nx=2048, ny=1, solver="custom", M=16, autotune=True,
             steps=4),
        # one evaluation of the stencil-tuning loss and its gradient: 500 steps, checkpoints every 50
        dict(name="grad_2d", kind="grad", nz=1024, nx=256, M=4, nline=64, nsteps=500, every=50, filter=False),
        # the solvers that the paper compares with: spectral on the 2D grid, PSATD on a 3D one
        dict(name="spectral_2d", kind="kspace", ndim=2, nz=2048, nx=512, ny=1, solver="spectral", nline=64, steps=4),
        dict(name="psatd_3d", kind="kspace", ndim=3, nz=256, nx=128, ny=128, solver="psatd", nline=64, steps=2),
        # the diagnostics of a running 2D simulation: Gauss residual at every node, energies, counts
        dict(name="diag_2d", kind="diag", ndim=2, nz=2048, nx=512, ny=1, solver="custom", M=16, shape=2, ppz=2, ppx=2,
             n_beam=1_000_000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _solver(rng):
    s = rng.choice(["yee", "custom", "custom"])
    return dict(solver=s, M=1 if s == "yee" else rng.choice([4, 8, 16, 16]))


def draw(rng):
    kind = rng.choice(["particle", "scan", "phases", "beam", "beam", "beam", "beam", "fields", "grad", "kspace", "diag"])
    if kind == "particle":
        return dict(kind=kind, nz=_log(rng, 96, 1024), nx=_log(rng, 24, 256), shape=rng.choice([1, 2]),
                    filter=rng.random() < 0.3, steps=rng.choice([1, 2, 5, 10]), **_solver(rng))
    if kind == "scan":
        return dict(kind=kind, n=_log(rng, 16, 256), nz_min=128, nz_max=_log(rng, 256, 1024), nx_min=64,
                    nx_max=_log(rng, 96, 256), shape=rng.choice([1, 2]), steps=rng.choice([8, 17, 32, 50]))
    if kind == "phases":
        nd = rng.choice([2, 3])
        size = (_log(rng, 256, 2048), _log(rng, 64, 512), 1) if nd == 2 else (_log(rng, 64, 256), _log(rng, 32, 96),
                                                                             _log(rng, 32, 96))
        return dict(kind=kind, ndim=nd, nz=size[0], nx=size[1], ny=size[2], shape=rng.choice([1, 2]),
                    ppc=4 if nd == 2 else 2, **_solver(rng))
    if kind in ("beam", "diag"):
        nd = rng.choice([2, 3])
        size = (_log(rng, 256, 2048), _log(rng, 64, 512), 1) if nd == 2 else (_log(rng, 128, 384), _log(rng, 48, 160),
                                                                             _log(rng, 48, 160))
        if rng.random() < 0.5:
            size = (4 * max(size[0] // 4, 16), size[1], size[2])      # whole 16-byte groups along z
        c = _beam(None, nd, size[0], size[1], size[2], "custom", rng.choice([1, 2, 2]), _log(rng, 20_000, 500_000),
                  rng.choice([1, 2, 4, 8]), filter=rng.random() < 0.25, autotune=rng.random() < 0.7)
        c.update(_solver(rng))
        if kind == "diag":
            return dict(kind=kind, **{k: c[k] for k in ("ndim", "nz", "nx", "ny", "solver", "M", "shape", "ppz", "ppx",
                                                        "n_beam")})
        return c
    if kind == "fields":
        nd = rng.choice([2, 3])
        size = (_log(rng, 512, 8192), _log(rng, 128, 2048), 1) if nd == 2 else (_log(rng, 128, 512), _log(rng, 64, 256),
                                                                               _log(rng, 64, 256))
        if rng.random() < 0.5:
            size = (4 * (size[0] // 4), size[1], size[2])
        return dict(kind=kind, ndim=nd, nz=size[0], nx=size[1], ny=size[2], autotune=rng.random() < 0.7,
                    steps=rng.choice([1, 2, 4]), **_solver(rng))
    if kind == "grad":
        return dict(kind=kind, nz=_log(rng, 256, 1024), nx=_log(rng, 64, 256), M=rng.choice([2, 4, 8]),
                    nline=rng.choice([1, 16, 48]), nsteps=_log(rng, 40, 400), every=rng.choice([10, 25, 50]),
                    filter=rng.random() < 0.3)
    nd = rng.choice([2, 3])
    size = (_log(rng, 128, 2048), _log(rng, 64, 1024), 1) if nd == 2 else (_log(rng, 64, 256), _log(rng, 48, 160),
                                                                          _log(rng, 48, 160))
    if rng.random() < 0.6:
        size = tuple(2 ** round(math.log2(v)) for v in size)
    return dict(kind=kind, ndim=nd, nz=size[0], nx=size[1], ny=size[2], solver=rng.choice(["spectral", "kt", "psatd"]),
                nline=rng.choice([1, 32]), steps=rng.choice([1, 2, 4]))


# ------------------------------------------------------------------------------ parameters ----

def _fit(kappa, M):
    """Appendix C fit of C_1..C_M to (kappa / pi) sin(pi k / kappa), constraint sum (2l-1) C_l = 1."""
    x, wq = np.polynomial.legendre.leggauss(1000)
    k, l = 0.25 * (x + 1.0), 2 * np.arange(1, M + 1) - 1
    w = 0.25 * wq * np.exp(-math.log(2.0) * (2.0 * k / 0.6) ** 10)
    s = np.sin(np.outer(l, math.pi * k))
    K = np.zeros((M + 1, M + 1))
    K[:M, :M] = 2.0 / math.pi ** 2 * (s * w) @ s.T
    K[:M, M] = K[M, :M] = l
    rhs = np.append(2.0 / math.pi * (s * w) @ (kappa / math.pi * np.sin(math.pi * k / kappa)), 1.0)
    return np.linalg.solve(K, rhs)[:M]


def _grid(case):
    """Cell sizes, dt and axial coefficients of a case."""
    kind = case["kind"]
    nd = case.get("ndim", 2)
    if kind in ("particle", "scan", "grad"):
        d, r = (0.05, 0.05, 0.05), 0.45 if kind == "particle" else 0.25
    elif nd == 2:
        d, r = (0.02, 0.02, 0.02), 0.5513
    else:
        d, r = (0.02, 0.05, 0.05), 0.68115
    if kind == "kspace":          # 0.9 of the spectral leapfrog's limit; PSATD at 0.9 of a cell
        r = 0.9 * (1.0 if case["solver"] == "psatd" else
                   2.0 / math.pi / math.sqrt(sum((d[0] / h) ** 2 for h in d[:nd])))
    solver = "custom" if kind == "grad" else case["solver"]
    C = _fit(1.0 / r, case["M"]) if solver == "custom" else np.array([1.0])
    return dict(ndim=nd, nz=case["nz"], nx=case["nx"], ny=case.get("ny", 1), dz=d[0], dx=d[1], dy=d[2], dt=r * d[0],
                solver=solver, C=C, shape=case.get("shape", 1), filter=bool(case.get("filter", False)))


def _config(g, **kw):
    c = dict(ndim=g["ndim"], nz=g["nz"], nx=g["nx"], ny=g["ny"], dz=g["dz"], dx=g["dx"], dy=g["dy"], dt=g["dt"],
             solver=g["solver"], shape=g["shape"], current_filter=g["filter"])
    if g["solver"] == "custom":
        c["coef"] = g["C"]
    return dict(c, **kw)


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _normal(gen, *shape):
    return torch.randn(shape, device="cuda", generator=gen)


def _uniform(gen, *shape):
    return torch.rand(shape, device="cuda", generator=gen).clamp_(1e-6, 1.0 - 1e-6)


# ---------------------------------------------------------------------------------- states ----

def _smooth(gen, g, amp, noise):
    """Three field components: a few long waves and a little noise, [c][y][x][z]."""
    z = torch.arange(g["nz"], device="cuda") * g["dz"]
    x = (torch.arange(g["nx"], device="cuda") + 0.5) / g["nx"]
    y = (torch.arange(g["ny"], device="cuda") + 0.5) / g["ny"]
    ph = torch.rand((3, 3), device="cuda", generator=gen) * 2.0 * math.pi
    out = torch.empty((3, g["ny"], g["nx"], g["nz"]), device="cuda")
    for c in range(3):
        w = torch.cos(z + ph[c, 0]) + 0.5 * torch.cos(2.7 * z + ph[c, 1])
        a = 1.0 + 0.5 * torch.cos(2.0 * math.pi * x + ph[c, 2])
        b = 1.0 + 0.5 * torch.cos(2.0 * math.pi * y - ph[c, 0]) if g["ndim"] == 3 else torch.ones_like(y)
        out[c] = amp * b[:, None, None] * a[None, :, None] * w[None, None, :]
        out[c] += noise * _normal(gen, g["ny"], g["nx"], g["nz"])
    return out


def _tile_key(g, iz, ix, iy):
    """Place of a cell in the order in which pic_sort leaves particles (include/pic.h)."""
    izg, nzg = iz + 1, g["nz"] + 2
    b = 3 if g["ndim"] == 2 else 2
    m = (1 << b) - 1
    ntz, ntx = (nzg + m) >> b, (g["nx"] + m) >> b
    ty = iy >> b if g["ndim"] == 3 else iy
    tx = ix >> b
    if g["ndim"] == 3:
        tx = torch.where(ty % 2 == 1, ntx - 1 - tx, tx)
    col = ty * ntx + tx
    tz = torch.where(col % 2 == 1, ntz - 1 - (izg >> b), izg >> b)
    inner = ((iy & m) << b if g["ndim"] == 3 else 0) + (ix & m)
    return (col * ntz + tz) * 64 + (inner << b) + (izg & m)


def _cells(g, iz, ix, iy):
    return ((iz + 1) + (g["nz"] + 2) * (ix + g["nx"] * iy)).to(torch.int32)


def _sorted_cells(g):
    """All cells (iz, ix, iy) in sorted order."""
    n = g["nz"] * g["nx"] * g["ny"]
    lin = torch.arange(n, device="cuda")
    iz, r = lin % g["nz"], lin // g["nz"]
    order = torch.argsort(_tile_key(g, iz, r % g["nx"], r // g["nx"]))
    iz, r = order % g["nz"], order // g["nz"]
    return iz.to(torch.int32), (r % g["nx"]).to(torch.int32), (r // g["nx"]).to(torch.int32)


def _beam_geometry(case, g):
    L = g["nz"] * g["dz"]
    return L - min(3.0, 0.4 * L), min(0.5, L / 10.0), 0.2 if g["ndim"] == 2 else 0.1


def _plasma(case, g, gen):
    """Cold quiet plasma ahead of the beam; behind it the wake, in which neighbours move together: a
    plasma wave of momentum 0.02 to 0.5 with a spread of a twentieth, the lattice displaced by it."""
    nd, pz, px = g["ndim"], case["ppz"], case["ppx"]
    iz, ix, iy = (t.repeat_interleave(pz * px) for t in _sorted_cells(g))
    n = iz.numel()
    sub = torch.arange(pz * px, device="cuda").repeat(n // (pz * px))
    z = iz.float() * g["dz"]
    wake = z < _beam_geometry(case, g)[0]
    x = ((ix.float() + 0.5) / g["nx"] - 0.5) * g["nx"] * g["dx"]
    y = ((iy.float() + 0.5) / g["ny"] - 0.5) * g["ny"] * g["dy"] if nd == 3 else torch.zeros_like(x)
    amp = torch.where(wake, 0.02 + 0.5 * torch.exp(-(x * x + y * y) / (2.0 * WAKE_CORE ** 2)), torch.zeros_like(x))
    ph = 2.0 * math.pi * torch.rand(3, device="cuda", generator=gen)
    off, u = torch.full((nd, n), 0.5, device="cuda"), 0.05 * _normal(gen, 3, n)
    off[0], off[1] = (sub // px + 0.5) / pz, (sub % px + 0.5) / px
    for a, t in enumerate((z, z + x, z + y)):
        u[a] = amp * (u[a] + torch.cos(t + ph[a]))
        if a < nd:
            moved = off[a] + 2.0 * torch.sin(t + ph[a])
            off[a] = torch.where(wake, (moved - torch.floor(moved)).clamp_max(1.0 - 2.0 ** -24), off[a])
    V = g["dz"] * g["dx"] * (g["dy"] if nd == 3 else 1.0)
    return _cells(g, iz, ix, iy), off, u, V / (pz * px)


def _beam_particles(case, g, gen):
    """Gaussian beam, gamma = 2e4 with 2% spread, peak density 100, truncated at 4 sigma, sorted."""
    nd, n = g["ndim"], case["n_beam"]
    zb, sz, sr = _beam_geometry(case, g)
    sig = (sz, sr, sr)[:nd]
    cen = (zb, 0.5 * g["nx"] * g["dx"], 0.5 * g["ny"] * g["dy"])
    lim = math.erf(4.0 / math.sqrt(2.0))
    xi = [(cen[a] + sig[a] * math.sqrt(2.0) * torch.erfinv(lim * (2.0 * _uniform(gen, n).double() - 1.0)))
          / (g["dz"], g["dx"], g["dy"])[a] for a in range(nd)]
    xi[0] = xi[0].clamp(1.0, g["nz"] - 1.001)
    c = [torch.floor(v) for v in xi]
    off = torch.stack([(v - w).float().clamp(0.0, 1.0 - 2.0 ** -24) for v, w in zip(xi, c)])
    c = [v.long() for v in c] + [torch.zeros(n, dtype=torch.long, device="cuda")] * (3 - nd)
    c = [c[0], c[1] % g["nx"], c[2] % g["ny"]]
    order = torch.argsort(_tile_key(g, *c), stable=True)
    gamma = 2e4 * (1.0 + 0.02 * (_uniform(gen, n) - 0.5))
    u = torch.zeros((3, n), device="cuda")
    u[0] = torch.sqrt(gamma * gamma - 1.0)
    total = 100.0 * (2.0 * math.pi) ** (nd / 2.0) * sz * sr ** (nd - 1) * lim ** nd
    return _cells(g, *c)[order], off[:, order].contiguous(), u, total / n


def _wake_fields(case, g, gen):
    """Plasma wave behind the beam, nothing ahead of it."""
    zb = _beam_geometry(case, g)[0]
    z = torch.arange(g["nz"], device="cuda") * g["dz"]
    x = ((torch.arange(g["nx"], device="cuda") + 0.5) / g["nx"] - 0.5) * g["nx"] * g["dx"]
    r2 = x[None, :, None] ** 2
    if g["ndim"] == 3:
        y = ((torch.arange(g["ny"], device="cuda") + 0.5) / g["ny"] - 0.5) * g["ny"] * g["dy"]
        r2 = r2 + y[:, None, None] ** 2
    env = torch.clamp((zb - z) / 0.5, 0.0, 1.0)[None, None, :] * (0.02 + torch.exp(-r2 / (2.0 * WAKE_CORE ** 2)))
    E, B = _smooth(gen, g, 0.3, 1e-3), _smooth(gen, g, 0.1, 1e-3)
    return E.mul_(env), B.mul_(env)


def _window(g, step):
    return int(math.floor(step * g["dt"] / g["dz"] + 1e-9))


FIRST_STEP = 1001        # a run resumed at this step; pic_step sorts when the step is a multiple of 20


def _particle_inputs(case, seed):
    rng = np.random.default_rng(seed)
    g = _grid(case)
    zx = (g["nz"] / 2 + rng.uniform(0, 4), g["nx"] / 2 + rng.uniform(0, 4))
    gamma = 10.0 ** rng.uniform(2.5, 3.5)
    gen = _gen(seed)
    return g, zx, math.sqrt(gamma * gamma - 1.0), _smooth(gen, g, 1e-2, 1e-4), _smooth(gen, g, 1e-2, 1e-4)


def _scan_inputs(case, seed):
    sizes_rng, rng = np.random.default_rng(4000), np.random.default_rng(seed)     # the grids belong to the case
    gen = _gen(seed)
    out = []
    for k in range(case["n"]):
        solver = "custom" if sizes_rng.integers(0, 2) else "yee"
        g = _grid(dict(kind="scan", nz=int(sizes_rng.integers(case["nz_min"], case["nz_max"] + 1)),
                       nx=int(sizes_rng.integers(case["nx_min"], case["nx_max"] + 1)), solver="yee",
                       shape=case["shape"]))
        frac = rng.uniform(0.3, 0.99)
        g["dt"] = frac * g["dz"] / (1.632488686516034 if solver == "custom" else math.sqrt(2.0))
        g["solver"], g["C"] = solver, _fit(g["dz"] / g["dt"], 16) if solver == "custom" else np.array([1.0])
        gamma = 10.0 ** rng.uniform(1, 5)
        cell = (g["nz"] // 8 + 2, g["nx"] // 2)
        off = rng.uniform(0.05, 0.95, 2).astype(np.float32)
        out.append((g, cell, off, np.float32(math.sqrt(gamma * gamma - 1.0))))
    sizes = [-(-3 * g["nz"] * g["nx"] // 64) * 64 for g, *_ in out]
    E = 1e-3 * _normal(gen, sum(sizes))
    return out, np.concatenate([[0], np.cumsum(sizes)]), E


def _phases_inputs(case, seed):
    g, gen = _grid(case), _gen(seed)
    iz, ix, iy = (t.repeat_interleave(case["ppc"]) for t in _sorted_cells(g))
    off, u = _uniform(gen, g["ndim"], iz.numel()), 1e-3 * _normal(gen, 3, iz.numel())
    V = g["dz"] * g["dx"] * (g["dy"] if g["ndim"] == 3 else 1.0)
    return g, _cells(g, iz, ix, iy), off, u, V / case["ppc"], _smooth(gen, g, 1e-2, 1e-4), _smooth(gen, g, 1e-2, 1e-4)


def _grad_inputs(case, seed):
    rng = np.random.default_rng(seed)
    g, n = _grid(case), case["nline"]
    C = g["C"] * (1.0 + 1e-3 * rng.standard_normal(case["M"]))
    C[0] += 1.0 - float(np.sum((2 * np.arange(1, case["M"] + 1) - 1) * C))
    ix = np.arange(g["nx"] // 2 - n // 2, g["nx"] // 2 - n // 2 + n)
    off = rng.uniform(0.3, 0.7, (2, 1)).astype(np.float32).repeat(n, axis=1)
    u = np.zeros((3, n), np.float32)
    u[0] = math.sqrt(1e8 - 1.0)
    sp = dict(iz=np.full(n, g["nz"] // 4), ix=ix, iy=np.zeros(n, np.int64), off=off, u=u, q=-1.0, m=1.0, w=1.0 / n)
    return g, C, sp


def _kspace_inputs(case, seed):
    g, gen, n = _grid(case), _gen(seed), case["nline"]
    k = torch.arange(n, device="cuda")
    # the line stays in the middle of z for as long as the fields run past it (momentum across z)
    iz = torch.full((n,), g["nz"] // 2, device="cuda", dtype=torch.long)
    ix = (g["nx"] // 2 - n // 2 + k) % g["nx"]
    iy = torch.full((n,), g["ny"] // 2, device="cuda", dtype=torch.long)
    off, u = _uniform(gen, g["ndim"], n), torch.zeros((3, n), device="cuda")
    u[1] = 1.0 + _uniform(gen, n)
    return g, _cells(g, iz, ix, iy), off, u, 1.0 / n, _smooth(gen, g, 1e-2, 1e-4), _smooth(gen, g, 1e-2, 1e-4)


def _bind(sim, s, cell, off, u, n, q, w):
    """A species held in device tensors (capacity = their length)."""
    cap = cell.numel()
    pic.pic_bind_species(sim.h, s, cell.data_ptr(), off.data_ptr(), u.data_ptr(), None, n, cap, q, 1.0, w)
    sim.species[s] = dict(cell=cell, off=off, u=u, id=None, q=q, m=1.0, w=w, cap=cap)


def _padded(cell, off, u, extra):
    if not extra:
        return cell, off, u
    n = cell.numel()
    c = torch.full((n + extra,), -1, dtype=torch.int32, device="cuda")
    o = torch.zeros((off.shape[0], n + extra), device="cuda")
    v = torch.zeros((3, n + extra), device="cuda")
    c[:n], o[:, :n], v[:, :n] = cell, off, u
    return c, o, v


def _front(case, g):
    return g["nx"] * g["ny"] * case["ppz"] * case["ppx"]


class _Scan:
    """A batch whose instances' fields and particles are pieces of a few large tensors."""

    def __init__(self, case, seed):
        inst, at, E = _scan_inputs(case, seed)
        self.E, self.B, self.J = E, torch.zeros_like(E), torch.zeros_like(E)
        n = len(inst)
        made = [make_config(**_config(g)) for g, *_ in inst]
        self.keep = made
        self.cell = torch.tensor([(c[0] + 1) + (g["nz"] + 2) * c[1] for g, c, _, _ in inst], dtype=torch.int32,
                                 device="cuda")
        self.off = torch.from_numpy(np.stack([o for _, _, o, _ in inst])).cuda()
        self.u = torch.zeros((n, 3), device="cuda")
        self.u[:, 0] = torch.from_numpy(np.array([u for *_, u in inst])).cuda()
        torch.cuda.synchronize()
        self.b = pic.pic_batch_create([m[0] for m in made])
        for k in range(n):
            h = pic.pic_batch_instance(self.b, k)
            o = 4 * int(at[k])
            pic.pic_bind_fields(h, self.E.data_ptr() + o, self.B.data_ptr() + o, self.J.data_ptr() + o)
            pic.pic_bind_species(h, 0, self.cell.data_ptr() + 4 * k, self.off.data_ptr() + 8 * k,
                                 self.u.data_ptr() + 12 * k, None, 1, 1, -1.0, 1.0, 1.0)

    def step(self, n):
        pic.pic_batch_step(self.b, n, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))

    def __del__(self):
        try:
            torch.cuda.synchronize()
            pic.pic_batch_destroy(self.b)
        except Exception:
            pass


def prepare(case, seed):
    kind = case["kind"]
    if kind == "scan":
        return case, _Scan(case, seed)
    if kind == "grad":
        g, C, sp = _grad_inputs(case, seed)
        grid = {k: g[k] for k in ("ndim", "nz", "nx", "ny", "dz", "dx", "dy", "dt", "shape")}
        grid["current_filter"] = g["filter"]
        return case, (StencilLoss(grid, [sp], nsteps=case["nsteps"], every=case["every"]), C)
    if kind == "particle":
        g, zx, uz, E, B = _particle_inputs(case, seed)
        sim = Simulation(**_config(g, moving_window=True))
        u = np.zeros((3, 1), np.float32)
        u[0] = uz
        off = np.array([[zx[0] % 1.0], [zx[1] % 1.0]], np.float32)
        sim.add_species(0, np.array([int(zx[0])]), np.array([int(zx[1])]), np.array([0]), off, u, -1.0, 1.0, 1.0)
    elif kind == "phases":
        g, cell, off, u, w, E, B = _phases_inputs(case, seed)
        sim = Simulation(**_config(g))
        _bind(sim, 0, cell, off, u, cell.numel(), -1.0, w)
    elif kind == "fields":
        g, gen = _grid(case), _gen(seed)
        E, B = _smooth(gen, g, 0.3, 1e-2), _smooth(gen, g, 0.3, 1e-2)
        sim = Simulation(**_config(g))
    elif kind == "kspace":
        g, cell, off, u, w, E, B = _kspace_inputs(case, seed)
        sim = Simulation(**_config(g))
        _bind(sim, 0, cell, off, u, cell.numel(), -1.0, w)
    else:                                                    # beam, diag
        g, gen = _grid(case), _gen(seed)
        E, B = _wake_fields(case, g, gen)
        sim = Simulation(**_config(g, moving_window=True, inject_species=0, inject_ppc=(case["ppz"], case["ppx"], 1),
                                   rho_bg=1.0, sort_every=20))
        cell, off, u, w = _plasma(case, g, gen)
        # room for the columns injected between two sorts
        _bind(sim, 0, *_padded(cell, off, u, 64 * _front(case, g) + 8192), cell.numel(), -1.0, w)
        del cell, off, u
        cell, off, u, w = _beam_particles(case, g, gen)
        _bind(sim, 1, cell, off, u, cell.numel(), -1.0, w)
        pic.pic_set_state(sim.h, FIRST_STEP, _window(g, FIRST_STEP), 0, 0)
    sim.E.copy_(E)
    sim.B.copy_(B)
    del E, B
    if case.get("autotune"):
        sim.autotune()
    torch.cuda.synchronize()
    return case, sim


def run(state):
    case, sim = state
    kind = case["kind"]
    if kind == "scan":
        sim.step(case["steps"])
        return dict(E=sim.E, B=sim.B, J=sim.J, cell=sim.cell, off=sim.off, u=sim.u)
    if kind == "grad":
        problem, C = sim
        loss, grad = problem.loss_and_grad(C)
        # the fields behind both are FP32: so is what the descent step takes
        return dict(loss=loss, grad=grad.astype(np.float32))
    if kind == "diag":
        G = sim.gauss()
        return dict(G=G, diag=[float(v) for k, v in sim.diag().items() if k != "status"])
    if kind == "phases":
        sim.gather_push()
        sim.deposit()
        sim.field_advance()
    else:
        sim.step(case["steps"])
    out = dict(E=sim.E, B=sim.B)
    for s, sp in sim.species.items():
        out["u%d" % s] = sp["u"]
        if case.get("positions", True):
            out["cell%d" % s], out["off%d" % s] = sp["cell"], sp["off"]
    if sim.species:
        out["J"] = sim.J
    return out


# ------------------------------------------------------------------------------------ work ----

def work(case):
    """Per step every cell reads E, B, J and writes E, B, and every particle reads and writes its cell,
    offsets and momenta."""
    kind = case["kind"]
    nd, K = case.get("ndim", 2), case.get("shape", 1) + 1
    M = case.get("M", 1)
    push = 2.0 * 6 * K ** nd + 2.0 * 3 * K * (K + 1) ** (nd - 1) + 150.0
    part = 2.0 * 4 * (1 + nd + 3)
    cells = case.get("nz", 0) * case.get("nx", 0) * case.get("ny", 1)
    field = 6 * 3.0 * M + 42.0
    if kind == "scan":
        cells = case["n"] * 0.25 * (case["nz_min"] + case["nz_max"]) * (case["nx_min"] + case["nx_max"])
        return dict(bytes=case["steps"] * 60.0 * cells, flops=case["steps"] * (6 * 3.0 * 8.5 + 42.0) * cells)
    if kind == "grad":
        # forward, replay and one adjoint step per step; the adjoint reads E, B, J and updates both adjoints
        return dict(bytes=case["nsteps"] * (60.0 + 60.0 + 84.0) * cells, flops=case["nsteps"] * 4 * field * cells)
    if kind == "kspace":
        return dict(bytes=case["steps"] * 60.0 * cells,
                    flops=case["steps"] * cells * (15 * 2.5 * math.log2(cells) + 60.0))
    if kind in ("beam", "diag"):
        n = cells * case["ppz"] * case["ppx"] + case["n_beam"]
    else:
        n = cells * case["ppc"] if kind == "phases" else 0 if kind == "fields" else case.get("nline", 1)
    if kind == "diag":
        return dict(bytes=cells * (24.0 + 8.0) + part / 2 * n, flops=cells * (3.0 * M + 20) + n * (3.0 * K ** nd + 20))
    s = case.get("steps", 1)
    return dict(bytes=s * (60.0 * cells + part * n), flops=s * (field * cells + push * n))


# ----------------------------------------------------------------------------- FP64 results ----

def _taps(C):
    """Impulse response of 1/P, P(phi) = sum_l C_l sin((2l-1) phi/2) / sin(phi/2), |m| <= HLEN."""
    n = 4096
    phi = 2.0 * math.pi * torch.arange(n, device=C.device, dtype=torch.float64) / n
    M = C.numel()
    P = torch.flip(torch.cumsum(torch.flip(C, [0]), 0), [0])         # P_m = sum_{l > m} C_l
    sym = P[0] + 2.0 * sum(P[m] * torch.cos(m * phi) for m in range(1, M)) if M > 1 else P[0] + 0.0 * phi
    h = torch.fft.ifft(1.0 / sym).real
    return torch.cat([h[n - HLEN:], h[:HLEN + 1]])


def _conv(F, h):
    """sum_m h[m] F[.., z - m], F = 0 outside the grid."""
    half = h.numel() // 2
    n = F.shape[-1] + 2 * half
    out = torch.fft.irfft(torch.fft.rfft(F, n=n) * torch.fft.rfft(h, n=n), n=n)
    return out[..., half:half + F.shape[-1]]


def _five_pass(J):
    for a, c in [(0.25, 0.5)] * 4 + [(-1.25, 3.5)]:
        p = torch.nn.functional.pad(J, (1, 1))
        J = a * (p[..., :-2] + p[..., 2:]) + c * J
    return J


def _dz(F, C, plus):
    n, M = F.shape[-1], C.numel()
    p = torch.nn.functional.pad(F, (M, M))
    out = 0.0
    for l in range(1, M + 1):
        a, b = (M + l, M - l + 1) if plus else (M + l - 1, M - l)
        out = out + C[l - 1] * (p[..., a:a + n] - p[..., b:b + n])
    return out


def _curl(F, g, C, plus):
    s = -1 if plus else 1
    d = lambda f, ax, h: (torch.roll(f, s, ax) - f) * (-s / h)                       # noqa: E731
    dx = lambda f: d(f, 1, g["dx"])                                                  # noqa: E731
    dy = lambda f: d(f, 0, g["dy"]) if g["ndim"] == 3 else torch.zeros_like(f)       # noqa: E731
    dz = lambda f: _dz(f, C, plus) / g["dz"]                                         # noqa: E731
    return torch.stack([dx(F[2]) - dy(F[1]), dy(F[0]) - dz(F[2]), dz(F[1]) - dx(F[0])])


def _advance(g, C, E, B, J):
    h = 0.5 * g["dt"]
    B = B - h * _curl(E, g, C, True)
    E = E + g["dt"] * (_curl(B, g, C, False) - J)
    return E, B - h * _curl(E, g, C, True)


def _kspace_advance(g, solver, E, B, J):
    nd, dt = g["ndim"], g["dt"]
    n = (g["nz"], g["nx"], g["ny"])
    hh = (g["dz"], g["dx"], g["dy"])
    ks, shape = [], [(1, 1, -1), (1, -1, 1), (-1, 1, 1)]
    for a in range(3):
        f = torch.fft.rfftfreq(n[a]) if a == 0 else torch.fft.fftfreq(n[a])
        ks.append((2.0 * math.pi / hh[a] * f.double().cuda()) if a < nd else torch.zeros(1, dtype=torch.float64).cuda())
        if a == 0 and n[0] % 2 == 0:
            ks[0] = ks[0].abs()
    fw = lambda F: torch.fft.rfftn(F, dim=(1, 2, 3))                                 # noqa: E731
    Ek, Bk, Jk = fw(E), fw(B), fw(J)
    yee = [2.0 / hh[a] * torch.sin(0.5 * ks[a] * hh[a]) for a in range(3)]
    kap = [k.clone() for k in ks] if solver != "kt" else [2.0 / dt * torch.sin(0.5 * ks[0] * dt), yee[1], yee[2]]
    ratio = [torch.where(kap[a] == 0, torch.ones_like(kap[a]), yee[a] / torch.where(kap[a] == 0, 1.0, kap[a]))
             for a in range(3)]
    Jk = torch.stack([Jk[a] * ratio[a].reshape(shape[a]) for a in range(3)])
    ph = [torch.exp(0.5j * ks[a] * hh[a]).reshape(shape[a]) for a in range(3)]
    kap = [v.reshape(shape[a]) for a, v in enumerate(kap)]

    def curl(d, F):
        return torch.stack([d[1] * F[2] - d[2] * F[1], d[2] * F[0] - d[0] * F[2], d[0] * F[1] - d[1] * F[0]])
    if solver != "psatd":
        dp = [1j * kap[a] * ph[a] for a in range(3)]
        dm = [1j * kap[a] * ph[a].conj() for a in range(3)]
        Bk = Bk - 0.5 * dt * curl(dp, Ek)
        Ek = Ek + dt * (curl(dm, Bk) - Jk)
        Bk = Bk - 0.5 * dt * curl(dp, Ek)
    else:
        pE = torch.stack(torch.broadcast_tensors(*[p.conj() for p in ph]))
        pB = torch.stack(torch.broadcast_tensors(*[(ph[1] * ph[2]).conj(), (ph[0] * ph[2]).conj(),
                                                   (ph[0] * ph[1]).conj()]))
        Ek, Bk, Jk = Ek * pE, Bk * pB, Jk * pE
        kn = torch.sqrt(kap[0] ** 2 + kap[1] ** 2 + kap[2] ** 2)
        zero = kn == 0
        k1 = torch.where(zero, torch.ones_like(kn), kn)
        kh = [k / k1 for k in kap]
        c, s = torch.cos(kn * dt), torch.sin(kn * dt)
        sk, ck = torch.where(zero, torch.full_like(kn, dt), s / k1), (1.0 - c) / k1
        dot = lambda F: kh[0] * F[0] + kh[1] * F[1] + kh[2] * F[2]                    # noqa: E731
        kv = torch.stack(torch.broadcast_tensors(*kh))
        En = c * Ek + 1j * s * curl(kh, Bk) - sk * Jk + (1.0 - c) * kv * dot(Ek) + (sk - dt) * kv * dot(Jk)
        Bn = c * Bk - 1j * s * curl(kh, Ek) + 1j * ck * curl(kh, Jk)
        keep = torch.ones_like(kn)
        for a in range(nd):
            if n[a] % 2 == 0:
                keep = keep * (torch.arange(ks[a].numel(), device="cuda") != n[a] // 2).double().reshape(shape[a])
        Ek, Bk = En * pE.conj() * keep, Bn * pB.conj() * keep
    inv = lambda F: torch.fft.irfftn(F, s=(n[2], n[1], n[0]), dim=(1, 2, 3))         # noqa: E731
    return inv(Ek), inv(Bk)


def _spline(order, d):
    d = d.abs()
    if order == 1:
        return (1.0 - d).clamp_min(0.0)
    return torch.where(d <= 0.5, 0.75 - d * d, 0.5 * (1.5 - d).clamp_min(0.0) ** 2)


_STAG = ((0.5, 0, 0), (0, 0.5, 0), (0, 0, 0.5), (0, 0.5, 0.5), (0.5, 0, 0.5), (0.5, 0.5, 0))


class _Grid64:
    """Gather and deposit in FP64 on arrays padded by PAD zeros at both z ends."""
    PAD = 4

    def __init__(self, g):
        self.g, self.nd, self.K = g, g["ndim"], g["shape"] + 1
        self.nzp = g["nz"] + 2 * self.PAD
        self.h = (g["dz"], g["dx"], g["dy"])

    def nodes(self, first, count, axis):
        """Wrapped node indices first .. first + count - 1 times the axis' stride."""
        if axis == 0:
            return [(first + a + self.PAD).clamp(0, self.nzp - 1) for a in range(count)]
        n, st = (self.g["nx"], self.nzp) if axis == 1 else (self.g["ny"], self.nzp * self.g["nx"])
        return [((first + a) % n) * st for a in range(count)]

    def first(self, xi):
        return torch.floor(xi + (0.5 if self.K == 3 else 0.0)).long() - (1 if self.K == 3 else 0)

    def gather(self, F, xi):
        """F: six padded components, xi: list of positions in cells."""
        out, half, node = [], [], []
        for a in range(self.nd):
            for lst, s in ((node, 0.0), (half, 0.5)):
                x = xi[a] - s
                b = self.first(x)
                lst.append((self.nodes(b, self.K, a), [_spline(self.K - 1, b + k - x) for k in range(self.K)]))
        for c in range(6):
            # in 2D the y staggering drops out
            ax = [half[a] if _STAG[c][a] else node[a] for a in range(self.nd)]
            f, acc = F[c].reshape(-1), 0.0
            for ky in range(self.K if self.nd == 3 else 1):
                for kx in range(self.K):
                    row, w = ax[1][0][kx], ax[1][1][kx]
                    if self.nd == 3:
                        row, w = row + ax[2][0][ky], w * ax[2][1][ky]
                    t = 0.0
                    for kz in range(self.K):
                        t = t + ax[0][1][kz] * f[row + ax[0][0][kz]]
                    acc = acc + w * t
            out.append(acc)
        return out

    def deposit(self, J, x0, x1, v3, qv):
        """Esirkepov current of moves x0 -> x1 added to the padded J; qv = q w / V (0: no particle)."""
        g, W = self.g, self.K + 1
        ax = []
        for a in range(self.nd):
            b = torch.minimum(self.first(x0[a]), self.first(x1[a]))
            s0 = [_spline(self.K - 1, b + k - x0[a]) for k in range(W)]
            ds = [_spline(self.K - 1, b + k - x1[a]) - s0[k] for k in range(W)]
            cum, run = [], 0.0
            for k in range(W - 1):
                run = run + ds[k]
                cum.append(run)
            ax.append((self.nodes(b, W, a), s0, ds, cum))
        f = [-qv * self.h[a] / g["dt"] for a in range(3)]
        add = lambda c, i, v: J[c].reshape(-1).index_add_(0, i, v)                  # noqa: E731
        if self.nd == 2:
            (nz, z0, dz, cz), (nx, s0, dx, cx) = ax
            for b in range(W):
                for a in range(W):
                    i = nz[a] + nx[b]
                    if a < W - 1:
                        add(0, i, f[0] * cz[a] * (s0[b] + 0.5 * dx[b]))
                    if b < W - 1:
                        add(1, i, f[1] * cx[b] * (z0[a] + 0.5 * dz[a]))
                    add(2, i, qv * v3 * (z0[a] * (s0[b] + 0.5 * dx[b]) + dz[a] * (0.5 * s0[b] + dx[b] / 3.0)))
            return
        for c, (p, r, q) in enumerate(((0, 1, 2), (1, 0, 2), (2, 0, 1))):
            for b in range(W):
                for k in range(W):
                    t = f[c] * (ax[r][1][b] * (ax[q][1][k] + 0.5 * ax[q][2][k])
                                + ax[r][2][b] * (0.5 * ax[q][1][k] + ax[q][2][k] / 3.0))
                    i = ax[r][0][b] + ax[q][0][k]
                    for a in range(W - 1):
                        add(c, i + ax[p][0][a], t * ax[p][3][a])

    def rho(self, out, xi, qv):
        ax = []
        for a in range(self.nd):
            b = self.first(xi[a])
            ax.append((self.nodes(b, self.K, a), [_spline(self.K - 1, b + k - xi[a]) for k in range(self.K)]))
        for ky in range(self.K if self.nd == 3 else 1):
            for kx in range(self.K):
                row, w = ax[1][0][kx], qv * ax[1][1][kx]
                if self.nd == 3:
                    row, w = row + ax[2][0][ky], w * ax[2][1][ky]
                for kz in range(self.K):
                    out.reshape(-1).index_add_(0, row + ax[0][0][kz], w * ax[0][1][kz])


class _Species64:
    """Positions (cells) and momenta in FP64, alive flags, charge q w / V and q dt / (2 m)."""

    def __init__(self, g, cell, off, u, w, q=-1.0, m=1.0):
        nd = g["ndim"]
        c = cell.long()
        izg, r = c % (g["nz"] + 2), c // (g["nz"] + 2)
        i = [izg - 1, r % g["nx"], r // g["nx"]]
        self.x = [i[a].double() + off[a].double() for a in range(nd)]
        self.u = u.double()
        self.alive = cell >= 0
        V = g["dz"] * g["dx"] * (g["dy"] if nd == 3 else 1.0)
        self.qv, self.eps = q * w / V, q * g["dt"] / (2.0 * m)


def _boris(u, eb, eps):
    um = u + eps * torch.stack(eb[:3])
    t = eps * torch.stack(eb[3:]) / torch.sqrt(1.0 + (um * um).sum(0))
    up = um + torch.linalg.cross(um, t, dim=0)
    return um + torch.linalg.cross(up, 2.0 * t / (1.0 + (t * t).sum(0)), dim=0) + eps * torch.stack(eb[:3])


def _push_all(g, E, B, species, shift, chunk=1 << 22):
    """Gather, push, move, deposit of every species; returns J."""
    G = _Grid64(g)
    pad = lambda F: torch.nn.functional.pad(F, (G.PAD, G.PAD))                       # noqa: E731
    F = torch.cat([pad(E), pad(B)])
    J = torch.zeros((3, g["ny"], g["nx"], G.nzp), dtype=torch.float64, device="cuda")
    n = (g["nz"], g["nx"], g["ny"])
    for sp in species:
        for k in range(0, sp.u.shape[1], chunk):
            s = slice(k, min(k + chunk, sp.u.shape[1]))
            x0 = [v[s].clone() for v in sp.x]
            if shift:
                x0[0] -= 1.0
            live = sp.alive[s] & (x0[0] >= 0) & (x0[0] < n[0])
            eb = G.gather(F, x0)
            u = torch.where(live, _boris(sp.u[:, s], eb, sp.eps), sp.u[:, s])
            gam = torch.sqrt(1.0 + (u * u).sum(0))
            x1 = [x0[a] + torch.where(live, g["dt"] / G.h[a] * u[a] / gam, 0.0) for a in range(G.nd)]
            G.deposit(J, x0, x1, u[2] / gam, sp.qv * live.double())
            sp.u[:, s] = u
            for a in range(G.nd):
                sp.x[a][s] = x1[a] % n[a] if a else x1[a]
            sp.alive[s] = live & (x1[0] >= 0) & (x1[0] < n[0])
    return J[..., G.PAD:G.PAD + n[0]].contiguous()


def _smooth_current(g, C, J):
    if g["filter"]:
        J = _five_pass(J)
    if C.numel() > 1:
        J = torch.cat([_conv(J[:1], _taps(C)), J[1:]])
    return J


def _steps(g, E, B, species, steps, first=0, window=False):
    C = torch.from_numpy(g["C"]).cuda()
    shifts, pending, J = _window(g, first), False, None
    for n in range(first + 1, first + steps + 1):
        J = _push_all(g, E, B, species, pending) if species else torch.zeros_like(E)
        pending = False
        if g["solver"] in ("spectral", "kt", "psatd"):
            E, B = _kspace_advance(g, g["solver"], E, B, J)
            continue
        J = _smooth_current(g, C, J)
        E, B = _advance(g, C, E, B, J)
        if window and _window(g, n) > shifts:
            shifts, pending = shifts + 1, True
            E, B = (torch.nn.functional.pad(F[..., 1:], (0, 1)) for F in (E, B))
    return E, B, J


def _exact_scan(case, seed):
    inst, at, E0 = _scan_inputs(case, seed)
    n = len(inst)
    out = {k: torch.zeros(E0.numel(), dtype=torch.float64, device="cuda") for k in "EBJ"}
    out["E"][:] = E0.double()
    u = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
    for k, (g, cell, off, uz) in enumerate(inst):
        m = 3 * g["nz"] * g["nx"]
        s = slice(int(at[k]), int(at[k]) + m)
        shp = (3, 1, g["nx"], g["nz"])
        c = torch.tensor([cell[0] + 1 + (g["nz"] + 2) * cell[1]], device="cuda")
        sp = _Species64(g, c, torch.from_numpy(off[:, None]).cuda(), torch.tensor([[uz], [0], [0]], device="cuda"), 1.0)
        E, B, J = _steps(g, E0[s].reshape(shp).double(), torch.zeros(shp, dtype=torch.float64, device="cuda"), [sp],
                         case["steps"])
        for key, F in zip("EBJ", (E, B, J)):
            out[key][s] = F.reshape(-1)
        u[k] = sp.u[:, 0]
    return dict(out, cell=None, off=None, u=u)


def _exact_grad(case, seed):
    g, C0, sp = _grad_inputs(case, seed)
    nz, nx = g["nz"], g["nx"]
    cell = torch.from_numpy((sp["iz"] + 1) + (nz + 2) * sp["ix"]).cuda()
    p = _Species64(g, cell, torch.from_numpy(sp["off"]).cuda(), torch.from_numpy(sp["u"]).cuda(), sp["w"], m=1e30)
    C = torch.from_numpy(C0).cuda().requires_grad_(True)
    E = B = torch.zeros((3, 1, nx, nz), dtype=torch.float64, device="cuda")
    zero = torch.zeros_like(E)
    for _ in range(case["nsteps"]):
        with torch.no_grad():
            J = _push_all(g, zero, zero, [p], False)
        E, B = _advance(g, C, E, B, _smooth_current(g, C, J))
    zc = max(int(torch.floor(p.x[0][p.alive].min())) - 2, 0)
    L = 0.5 * ((E[..., :zc] ** 2).sum() + (B[..., :zc] ** 2).sum()) * g["dz"] * g["dx"]
    L.backward()
    return dict(loss=float(L), grad=C.grad.cpu().numpy())


def _exact_diag(case, seed):
    g, gen = _grid(case), _gen(seed)
    E, B = (F.double() for F in _wake_fields(case, g, gen))
    G, C = _Grid64(g), torch.from_numpy(g["C"]).cuda()
    rho = torch.zeros((g["ny"], g["nx"], G.nzp), dtype=torch.float64, device="cuda")
    kin, count = 0.0, 0
    V = g["dz"] * g["dx"] * (g["dy"] if g["ndim"] == 3 else 1.0)
    for make in (_plasma, _beam_particles):
        cell, off, u, w = make(case, g, gen)
        sp = _Species64(g, cell, off, u, w)
        for k in range(0, cell.numel(), 1 << 22):
            s = slice(k, k + (1 << 22))
            G.rho(rho, [v[s] for v in sp.x], sp.qv * torch.ones_like(sp.x[0][s]))
        u2 = (sp.u * sp.u).sum(0)
        kin += float((u2 / (1.0 + torch.sqrt(1.0 + u2))).sum()) * w
        count += cell.numel()
    rho = rho[..., G.PAD:G.PAD + g["nz"]]
    dx = (E[1] - torch.roll(E[1], 1, 1)) / g["dx"]
    dy = (E[2] - torch.roll(E[2], 1, 0)) / g["dy"] if g["ndim"] == 3 else 0.0
    res = _dz(E[0], C.float().double(), False) / g["dz"] + dx + dy - rho - 1.0
    margin = g["C"].size + HLEN + 2 if g["C"].size > 1 else 2
    inner = res[..., margin:g["nz"] - margin]
    return dict(G=res, diag=[float(inner.abs().max()), float(inner.square().mean().sqrt()), float(rho.abs().max()),
                             0.5 * V * float(E.square().sum() + B.square().sum()), kin, float(count),
                             float(FIRST_STEP), float(_window(g, FIRST_STEP)), float(inner.numel())])


def exact(case, seed):
    kind = case["kind"]
    if kind == "scan":
        return _exact_scan(case, seed)
    if kind == "grad":
        return _exact_grad(case, seed)
    if kind == "diag":
        return _exact_diag(case, seed)
    if kind == "particle":
        g, zx, uz, E, B = _particle_inputs(case, seed)
        cell = torch.tensor([int(zx[0]) + 1 + (g["nz"] + 2) * int(zx[1])], device="cuda")
        off = torch.tensor([[zx[0] % 1.0], [zx[1] % 1.0]], device="cuda", dtype=torch.float32)
        species = [_Species64(g, cell, off, torch.tensor([[uz], [0], [0]], device="cuda", dtype=torch.float32), 1.0)]
    elif kind == "phases":
        g, cell, off, u, w, E, B = _phases_inputs(case, seed)
        species = [_Species64(g, cell, off, u, w)]
    elif kind == "kspace":
        g, cell, off, u, w, E, B = _kspace_inputs(case, seed)
        species = [_Species64(g, cell, off, u, w)]
    elif kind == "fields":
        g, gen = _grid(case), _gen(seed)
        E, B, species = _smooth(gen, g, 0.3, 1e-2), _smooth(gen, g, 0.3, 1e-2), []
    else:
        g, gen = _grid(case), _gen(seed)
        E, B = _wake_fields(case, g, gen)
        species = [_Species64(g, *make(case, g, gen)) for make in (_plasma, _beam_particles)]
    E, B, J = _steps(g, E.double(), B.double(), species, case.get("steps", 1), first=FIRST_STEP if kind == "beam" else 0,
                     window=kind in ("beam", "particle"))
    out = dict(E=E, B=B)
    for s, sp in enumerate(species):
        u = sp.u
        if kind == "beam" and s == 0:          # the injected columns are at rest
            u = torch.nn.functional.pad(u, (0, 64 * _front(case, g) + 8192))
        out["u%d" % s] = u
        if case.get("positions", True):
            out["cell%d" % s] = out["off%d" % s] = None
    if species:
        out["J"] = J
    return out
