"""Cost of one input relative to another through the same call, where a route once cost several times what its work
does.  Ratios of medians on one device with wide margins: no absolute times."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1910_13529_gb300 as P  # noqa: E402
from oracle import fit  # noqa: E402
from paper_1910_13529_gb300 import workloads as wl  # noqa: E402
from paper_1910_13529_gb300.runtime import Batch, Simulation  # noqa: E402


def median_ms(f, reps=9):
    for _ in range(3):
        f()
    ts = []
    for _ in range(reps):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        f()
        b.record()
        torch.cuda.synchronize()
        ts.append(a.elapsed_time(b))
    return float(np.median(ts))


def slow_particles(ndim, nz, nx, ny, n, seed=1):
    """In no order, slow enough to keep the order that a sort gives them."""
    return wl.random_particles(ndim, nz, nx, ny, n, seed=seed, u_scale=1e-3, margin=4)


def add(sim, sp):
    sim.add_species(0, sp["iz"], sp["ix"], sp["iy"], sp["off"], sp["u"], sp["q"], sp["m"], sp["w"])


@pytest.mark.parametrize("shape", [1, 2])
def test_unsorted_particles_3d(shape):
    """A step that gathers and deposits per particle (nothing sorted) against one whose chunks fit their boxes: 2.2 to
    4.7 times as long, 5.9 to 11 when the per-particle path had hardly any L1."""
    sim = Simulation(ndim=3, nz=128, nx=64, ny=64, dz=0.05, dx=0.05, dy=0.05, dt=0.025, shape=shape)
    add(sim, slow_particles(3, 128, 64, 64, 1 << 20))
    unsorted = median_ms(lambda: sim.step(1))
    sim.sort()
    assert unsorted < (4.2 if shape == 1 else 7.5) * median_ms(lambda: sim.step(1))
    sim.close()


@pytest.mark.parametrize("shape", [1, 2])
def test_unsorted_particles_of_a_batch(shape):
    """A batch never sorts.  Instances whose particles stand in no order against ones that were bound in tile order: 2.5 and
    4.1 times as long, 6 and 8 when the global path had hardly any L1."""
    d = 0.05
    times = []
    for ordered in (False, True):
        batch = Batch([dict(ndim=2, nz=256, nx=128, dz=d, dx=d, dt=0.5 * d, shape=shape)] * 16)
        for i, sim in enumerate(batch.instances):
            sp = slow_particles(2, 256, 128, 1, 4 * 256 * 128, seed=i)
            if ordered:
                o = np.lexsort((sp["iz"] % 8, sp["ix"] % 8, sp["iz"] // 8, sp["ix"] // 8))
                sp.update({k: sp[k][..., o] for k in ("iz", "ix", "iy", "off", "u")})
            add(sim, sp)
        batch.step(34)
        times.append(median_ms(lambda: batch.step(8)))
        batch.close()
    assert times[0] < (4.0 if shape == 1 else 6.0) * times[1]


@pytest.mark.parametrize("M", [1, 4, 16])
def test_field_advance_of_short_rows(M):
    """128 x 16384 cells against 16384 x 128: 0.7 to 1.2 times as long, 6 to 8 when the short rows' one column of segments was
    cut into 64 chunks."""
    times = []
    for nz, nx in ((128, 16384), (16384, 128)):
        kw = dict(solver="custom", coef=fit.fit_coefficients(4.0, M=M)) if M > 1 else {}
        sim = Simulation(ndim=2, nz=nz, nx=nx, dz=0.05, dx=0.05, dt=0.0125, **kw)
        times.append(median_ms(lambda: [sim.field_advance() for _ in range(4)]))
        sim.close()
    assert times[0] < 2.5 * times[1]


@pytest.mark.parametrize("dims", [(64, 32, 32), (65, 33, 31)])
def test_default_field_variant_of_small_3d_grids(dims):
    """A handle's own choice against the plain tile of variant 0: 0.5 to 0.7 times as long, 1.3 to 1.6 with the y-march."""
    sim = Simulation(ndim=3, nz=dims[0], nx=dims[1], ny=dims[2], dz=0.05, dx=0.05, dy=0.05, dt=0.025)
    own = median_ms(lambda: [sim.field_advance() for _ in range(20)])
    P.pic_set_tuning(sim.h, 0)
    assert own < 1.1 * median_ms(lambda: [sim.field_advance() for _ in range(20)])
    sim.close()
