"""GPU parity of dispatch branches at the sizes where they can go wrong, against the FP64 oracle.

Tolerances as in test_gpu_parity.py: FP32 kernels, fields within 1e-5 of the largest |field|,
positions within 1e-5 cell, momenta within 1e-5 of the largest |u|."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from oracle import fit  # noqa: E402
from paper_1910_13529_gb300 import workloads as wl  # noqa: E402

from parity_util import field_error, gpu_sim, oracle_sim, particle_errors  # noqa: E402

TOL = 1e-5


def _grid3(nz, nx, ny, shape):
    d = (0.5, 0.4, 0.45)
    return dict(ndim=3, nz=nz, nx=nx, ny=ny, dz=d[0], dx=d[1], dy=d[2], dt=0.9 * fit.cfl_dt(d[0], d[1:], None),
                solver="yee", shape=shape)


def _patch(n, nz, nx, ny, ext, seed):
    """n particles scattered over a patch of ext cells around the grid's middle (unsorted)."""
    sp = wl.random_particles(3, nz, nx, ny, n, seed=seed, u_scale=0.6, u_drift=(1.0, 0.2, -0.1), margin=4)
    rng = np.random.default_rng(seed + 50)
    for key, size, e in zip(("iz", "ix", "iy"), (nz, nx, ny), ext):
        sp[key] = (size - e) // 2 + rng.integers(0, e, n)
    return sp


@pytest.mark.parametrize("shape", [1, 2])
@pytest.mark.parametrize("nz", [48, 51])
def test_3d_chunks_of_every_path(shape, nz):
    """Three species whose chunks take the three 3D paths: compact (shared boxes of the main kernel, at
    their exact size limits along x and y), wide (general path) and scattered over the whole grid
    (per particle); the lists of all species are finished by one launch."""
    nx, ny = 40, 36
    grid = _grid3(nz, nx, ny, shape)
    top = 8 - (shape + 1)                    # cells along x and y whose gather box is 8 nodes wide
    sps = [_patch(700, nz, nx, ny, (9, top, top), 1), _patch(900, nz, nx, ny, (12, 14, 9), 2),
           _patch(500, nz, nx, ny, (nz - 10, nx, ny), 3)]
    sim, osim = gpu_sim(grid, sps), oracle_sim(grid, sps)
    rng = np.random.default_rng(4)
    for a, oa in ((sim.E, osim.E), (sim.B, osim.B)):
        v = (0.3 * rng.normal(size=oa.shape)).astype(np.float32)
        a.copy_(torch.from_numpy(v))
        oa[:] = v
    for _ in range(2):
        sim.step(1)
        osim.step()
        assert np.abs(sim.J.double().cpu().numpy() - osim.J).max() < TOL * np.abs(osim.J).max()
    assert field_error(sim, osim) < TOL
    for s in range(3):
        dx, du = particle_errors(sim, osim, s, 3)
        assert dx < TOL and du < TOL
    sim.close()


@pytest.mark.parametrize("M", [1, 5, 16])
@pytest.mark.parametrize("nz,nx", [(1504, 12), (1503, 9), (420, 40)])
def test_2d_marching_rows(nz, nx, M):
    """x-marching field advance (variants 8..11) with the window shift: several z segments, whole and
    ragged last segments, rows with and without 16-byte alignment, several chunks along x."""
    from oracle import core as oc
    from paper_1910_13529_gb300 import pic_set_tuning
    C = fit.fit_coefficients(2.5, M=M) if M > 1 else np.array([1.0])
    d = (0.5, 0.45)
    grid = dict(ndim=2, nz=nz, nx=nx, ny=1, dz=d[0], dx=d[1], dy=1.0, dt=0.9 * fit.cfl_dt(d[0], d[1:], C),
                solver="custom" if M > 1 else "yee", shape=1, moving_window=True)
    rng = np.random.default_rng(nz + M)
    start = [rng.normal(size=(3, 1, nx, nz)).astype(np.float32) for _ in range(3)]
    osim = oracle_sim(grid, [], coef=C)
    for oa, v in zip((osim.E, osim.B, osim.J), start):
        oa[:] = v
    shifted = []
    for _ in range(3):
        oc.field_advance(osim.g, osim.E, osim.B, osim.J)
        osim.n += 1
        shifted.append(oc.window_due(osim.n, osim.g.dt, osim.g.dz, osim.shifts))
        if shifted[-1]:
            osim.shift()
    assert any(shifted) and not all(shifted)
    for variant in (8, 9, 10, 11):
        sim = gpu_sim(grid, [], coef=C)
        pic_set_tuning(sim.h, variant)
        for a, v in zip((sim.E, sim.B, sim.J), start):
            a.copy_(torch.from_numpy(v))
        for _ in range(3):
            sim.field_advance()
        assert field_error(sim, osim) < TOL, variant
        sim.close()


@pytest.mark.parametrize("ndim,nz,nx,ny,M", [(2, 37, 9, 1, 4), (2, 530, 5, 1, 16), (2, 512, 4, 1, 8), (3, 45, 6, 5, 3),
                                             (3, 64, 5, 4, 16), (2, 50, 6, 1, 2)])
def test_adjoint_run(ndim, nz, nx, ny, M):
    """pic_step_record and pic_adjoint_run over two steps without particles, against FP64 central
    differences of the oracle: gradient to 1e-4 of its largest entry (the framework's bound), and the
    same result from pic_adjoint_step called step by step."""
    import paper_1910_13529_gb300 as P
    from oracle import core as oc
    C = fit.fit_coefficients(2.5, M=M) if M > 1 else np.array([1.0])
    d = (0.5, 0.45, 0.4)[:ndim]
    grid = dict(ndim=ndim, nz=nz, nx=nx, ny=ny, dz=d[0], dx=d[1], dy=d[2] if ndim == 3 else 1.0,
                dt=0.8 * fit.cfl_dt(d[0], d[1:], C), solver="custom", shape=1)
    rng = np.random.default_rng(100 * M + nz)
    shp = (3, ny, nx, nz)
    E0, B0, lE, lB = (rng.normal(size=shp).astype(np.float32) for _ in range(4))

    def loss(Cx):
        osim = oracle_sim(grid, [], coef=Cx)
        osim.E[:], osim.B[:] = E0, B0
        for _ in range(2):
            oc.field_advance(osim.g, osim.E, osim.B, osim.J)
        return np.sum(lE * osim.E) + np.sum(lB * osim.B)

    ref = np.zeros(M)
    for l in range(M):
        h = np.zeros(M)
        h[l] = 1e-5
        ref[l] = (loss(C + h) - loss(C - h)) / 2e-5
    sim = gpu_sim(grid, [], coef=C)
    dev = lambda a: torch.from_numpy(a).cuda()                                       # noqa: E731
    E = torch.empty((3, *shp), device="cuda")
    B, J = torch.empty_like(E), torch.empty((2, *shp), device="cuda")
    E[0], B[0] = dev(E0), dev(B0)
    P.pic_step_record(sim.h, 2, E.data_ptr(), B.data_ptr(), J.data_ptr(), sim.stream)
    grads = []
    for one_by_one in (False, True):
        aE, aB = dev(lE), dev(lB)
        grad = torch.zeros(M, dtype=torch.float64, device="cuda")
        if one_by_one:
            for k in (1, 0):
                P.pic_adjoint_step(sim.h, E[k].data_ptr(), B[k].data_ptr(), J[k].data_ptr(), aE.data_ptr(), aB.data_ptr(),
                                   grad.data_ptr(), sim.stream)
        else:
            P.pic_adjoint_run(sim.h, 2, E.data_ptr(), B.data_ptr(), J.data_ptr(), aE.data_ptr(), aB.data_ptr(),
                              grad.data_ptr(), sim.stream)
        torch.cuda.synchronize()
        grads.append(grad.cpu().numpy())
    scale = np.abs(ref).max()
    for g in grads:
        assert np.abs(g - ref).max() < 1e-4 * scale
    # <l, A x> = <A^T l, x>
    rhs = float((aE.double() * E[0].double()).sum() + (aB.double() * B[0].double()).sum())
    lhs = float((dev(lE).double() * E[2].double()).sum() + (dev(lB).double() * B[2].double()).sum())
    assert abs(lhs - rhs) < 1e-5 * np.linalg.norm(lE) * np.linalg.norm(E0)
    sim.close()


@pytest.mark.parametrize("ndim,shape", [(2, 1), (2, 2), (3, 1), (3, 2)])
@pytest.mark.parametrize("spread", ["cells", "patch", "grid"])
def test_rho_and_diagnostics(ndim, shape, spread):
    """FP64 charge density, Gauss residual and energies against the oracle: particles of a chunk in a few
    cells (shared nodes), in a patch across the periodic seam, and all over the grid (per-particle path).
    A contribution is rounded to 2^-45 of a particle's charge density and a divergence to 2^-46 of the
    sum of its terms: 1e-12 of the largest value leaves a factor of ten over the sums of 256."""
    from oracle import core as oc
    nz, nx, ny = (517, 30, 1) if ndim == 2 else (70, 24, 20)
    d = (0.5, 0.4, 0.45)[:ndim]
    C = fit.fit_coefficients(2.5, M=8)
    grid = dict(ndim=ndim, nz=nz, nx=nx, ny=ny, dz=d[0], dx=d[1], dy=d[2] if ndim == 3 else 1.0,
                dt=0.8 * fit.cfl_dt(d[0], d[1:], C), solver="custom", shape=shape, rho_bg=0.5)
    sp = wl.random_particles(ndim, nz, nx, ny, 700, seed=9, u_scale=0.3, u_drift=(5.0, 0, 0), margin=0)
    if spread != "grid":
        ext = 2 if spread == "cells" else 9
        rng = np.random.default_rng(3)
        sp["iz"] = nz - ext + rng.integers(0, ext, 700)
        sp["ix"] = (nx - ext // 2 + rng.integers(0, ext, 700)) % nx
        if ndim == 3:
            sp["iy"] = (ny - ext // 2 + rng.integers(0, ext, 700)) % ny
    sim, osim = gpu_sim(grid, [sp], coef=C), oracle_sim(grid, [sp], coef=C)
    rng = np.random.default_rng(1)
    for a, oa in ((sim.E, osim.E), (sim.B, osim.B)):
        v = rng.normal(size=oa.shape).astype(np.float32)
        a.copy_(torch.from_numpy(v))
        oa[:] = v
    s = osim.species[0]
    ref = oc.rho(osim.g, s.xi, s.Q)
    got = sim.rho().cpu().numpy()
    assert np.abs(got - ref).max() < 1e-12 * np.abs(ref).max()
    G = sim.gauss().cpu().numpy()
    g32 = oc.Grid(ndim, nz, nx, ny, *(float(np.float32(grid[k])) for k in ("dz", "dx", "dy", "dt")),
                  C=C.astype(np.float32).astype(np.float64), shape=shape)     # the GPU's FP32 constants
    Gref = oc.gauss(g32, osim.E, ref) - 0.5
    assert np.abs(G - Gref).max() < 1e-12 * np.abs(Gref).max()
    m = 8 + 24 + 2
    D = sim.diag()
    assert D["gauss_max"] == pytest.approx(np.abs(Gref[..., m:nz - m]).max(), rel=1e-11)
    assert D["gauss_rms"] == pytest.approx(np.sqrt(np.mean(Gref[..., m:nz - m] ** 2)), rel=1e-11)
    V = np.prod(d)
    assert D["field_energy"] == pytest.approx(0.5 * V * (np.sum(osim.E ** 2) + np.sum(osim.B ** 2)), rel=1e-12)
    u2 = np.sum(s.u ** 2, axis=1)
    assert D["kinetic"] == pytest.approx(sp["w"] * np.sum(u2 / (1 + np.sqrt(1 + u2))), rel=1e-12)
    assert D["count"] == 700
    sim.close()


@pytest.mark.parametrize("nz", [1024, 1021, 512, 260, 43])
def test_correction_of_paired_rows(nz):
    """The Sec. 3 correction on many short rows (two at a time, an odd number of them) against the oracle
    (24 taps each side on the GPU, 40 in the oracle: the tail is below 1e-9)."""
    nx, ny = 63, 65
    C = fit.fit_coefficients(2.5, M=16)
    grid = dict(ndim=3, nz=nz, nx=nx, ny=ny, dz=0.5, dx=0.6, dy=0.7, dt=0.2, solver="custom", shape=1)
    sp = wl.random_particles(3, nz, nx, ny, 4000, seed=nz, u_scale=1.0, margin=4)
    sim, osim = gpu_sim(grid, [sp], coef=C), oracle_sim(grid, [sp], coef=C)
    sim.step(1)
    osim.step()
    J = sim.J.double().cpu().numpy()
    assert np.abs(J - osim.J).max() < TOL * np.abs(osim.J).max()
    assert field_error(sim, osim) < TOL
    sim.close()


@pytest.mark.parametrize("ndim,nz,nx,ny,filt", [(2, 130, 24, 1, False), (2, 131, 25, 1, True), (2, 4100, 260, 1, False),
                                                (3, 50, 20, 18, False), (3, 48, 20, 18, True)])
def test_captured_steps(ndim, nz, nx, ny, filt):
    """Three steps captured into a CUDA graph by the caller and replayed once (launches chained from
    kernel to kernel, from the memset of a large J, and into the copies back), against the oracle."""
    d = (0.5, 0.4, 0.45)[:ndim]
    C = fit.fit_coefficients(2.5, M=4)
    grid = dict(ndim=ndim, nz=nz, nx=nx, ny=ny, dz=d[0], dx=d[1], dy=d[2] if ndim == 3 else 1.0,
                dt=0.8 * fit.cfl_dt(d[0], d[1:], C), solver="custom", shape=2, current_filter=filt)
    sp = wl.random_particles(ndim, nz, nx, ny, 900, seed=nz, u_scale=0.5, u_drift=(2.0, 0, 0), margin=8)
    sim, osim = gpu_sim(grid, [sp], coef=C), oracle_sim(grid, [sp], coef=C)
    sim.step(1)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        sim.step(3)
    graph.replay()
    torch.cuda.synchronize()
    for _ in range(4):
        osim.step()
    assert field_error(sim, osim) < TOL
    dx, du = particle_errors(sim, osim, 0, ndim)
    assert dx < TOL and du < TOL
    sim.close()


@pytest.mark.parametrize("nz,nx,ny", [(512, 65, 65), (512, 64, 64), (516, 64, 65), (1020, 65, 65), (1024, 63, 67)])
def test_correction_in_pairs_of_rows(nz, nx, ny):
    """The Sec. 3 correction where it takes two rows at a time (at least 4096 aligned rows of 512 to 1024 cells): two pairs
    and one pair per CTA, an odd number of rows, a last CTA with an idle group, rows that end inside a lane's eight
    cells; against the oracle as above."""
    assert nz % 4 == 0 and nx * ny >= 4096
    C = fit.fit_coefficients(2.5, M=8)
    grid = dict(ndim=3, nz=nz, nx=nx, ny=ny, dz=0.5, dx=0.6, dy=0.7, dt=0.2, solver="custom", shape=1)
    sp = wl.random_particles(3, nz, nx, ny, 4000, seed=nz + nx, u_scale=1.0, margin=1)
    sim, osim = gpu_sim(grid, [sp], coef=C), oracle_sim(grid, [sp], coef=C)
    sim.step(1)
    osim.step()
    J = sim.J.double().cpu().numpy()
    assert np.abs(J - osim.J).max() < TOL * np.abs(osim.J).max()
    assert field_error(sim, osim) < TOL
    sim.close()


@pytest.mark.parametrize("nz,nx,copies", [(64, 32, 1), (1500, 800, 2)])
def test_counted_launches(nz, nx, copies):
    """pic_timing_read counts what is launched: a call that ends in the second field buffers copies E and B back by one
    kernel, on large grids by two copies."""
    import paper_1910_13529_gb300 as P
    grid = dict(ndim=2, nz=nz, nx=nx, ny=1, dz=0.5, dx=0.5, dy=1.0, dt=0.1, solver="yee", shape=1)
    sim = gpu_sim(grid, [wl.random_particles(2, nz, nx, 1, 50, seed=1)])
    for nsteps in (1, 2, 3):
        P.pic_timing(sim.h, 1)
        sim.step(nsteps)
        _, n = P.pic_timing_read(sim.h, sim.stream)
        P.pic_timing(sim.h, 0)
        assert n["fields"] == nsteps + (copies if nsteps % 2 else 0)
        assert n["deposit"] == n["particles"] == nsteps
    P.pic_timing(sim.h, 1)
    sim.gather_push()
    sim.deposit()
    sim.field_advance()
    assert P.pic_timing_read(sim.h, sim.stream)[1]["fields"] == 1 + copies
    sim.close()


def test_wait_for_field_copies_runs_out():
    """With no look at all the 3D kernel gives up its copies (which do arrive), reports it and returns; the context stays
    usable, and a handle that has not been limited steps as ever."""
    import paper_1910_13529_gb300 as P
    grid = _grid3(48, 16, 16, 2)
    sp = _patch(600, 48, 16, 16, (9, 5, 5), 1)
    sim = gpu_sim(grid, [sp])
    with pytest.raises(P.PicError):
        P.pic_set_wait_limit(sim.h, -1)
    P.pic_set_wait_limit(sim.h, 0)
    sim.step(1)
    with pytest.raises(P.PicError) as e:
        sim.sync()
    assert "did not arrive" in str(e.value)
    sim.close()
    other, osim = gpu_sim(grid, [sp]), oracle_sim(grid, [sp])
    other.step(2)
    other.sync()
    for _ in range(2):
        osim.step()
    assert field_error(other, osim) < TOL
    other.close()
