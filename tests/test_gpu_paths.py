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
