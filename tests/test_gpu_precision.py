"""What the library forms in FP64, or wider out of FP32 parts, against exact rational arithmetic.  Tolerances
count the FP64 roundings of the result (u = 2^-53 each); the parts before them lose less than 2^-60."""
from decimal import Decimal, getcontext
from fractions import Fraction as Fr

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1910_13529_gb300 as P  # noqa: E402
from oracle import fit  # noqa: E402
from paper_1910_13529_gb300.runtime import Simulation  # noqa: E402

U = 2.0 ** -53


def _sim(nz, M=1, nx=4, **kw):
    C = dict(solver="custom", coef=fit.fit_coefficients(4.0, M=M)) if M > 1 else dict(solver="yee")
    return Simulation(device="cuda:0", ndim=2, nz=nz, nx=nx, dz=0.5, dx=0.5, dt=0.125, **C, **kw)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def _gradient(sim, M, E1, aE, aB, J):
    """The gradient of one recorded step whose first fields are zero: only the third stage (E1, aB) and the
    correction (J, aE) contribute."""
    E = torch.stack([torch.zeros_like(_dev(E1)), _dev(E1)])
    B, Jd, aEd, aBd = torch.zeros_like(E), _dev(J), _dev(aE), _dev(aB)
    grad = torch.zeros(M, dtype=torch.float64, device="cuda")
    P.pic_adjoint_run(sim.h, 1, E.data_ptr(), B.data_ptr(), Jd.data_ptr(), aEd.data_ptr(), aBd.data_ptr(),
                      grad.data_ptr(), sim.stream)
    torch.cuda.synchronize()
    return grad.cpu().numpy()


def _at(row, z):
    return Fr(float(row[z])) if 0 <= z < len(row) else Fr(0)


def _third_stage(E1, aB, M, scale):
    """scale sum l3 D+_l F2 - l2 D+_l F3 over the cells with (l2, l3) != 0, and the sum of the terms' sizes."""
    out, size = [Fr(0)] * M, [Fr(0)] * M
    _, _, nx, nz = E1.shape
    for x in range(nx):
        for z in range(nz):
            l2, l3 = Fr(float(aB[1, 0, x, z])), Fr(float(aB[2, 0, x, z]))
            if not l2 and not l3:
                continue
            for l in range(1, M + 1):
                for v, f in ((l3, E1[1, 0, x]), (-l2, E1[2, 0, x])):
                    t = v * (_at(f, z + l) - _at(f, z - l + 1))
                    out[l - 1] += scale * t
                    size[l - 1] += abs(scale * t)
    return out, size


@pytest.mark.parametrize("M", [3, 8, 16])
@pytest.mark.parametrize("la,lf", [(0, 0), (-60, -60), (-120, 30), (60, 63), (-20, -128)])
def test_gradient_sums(M, la, lf):
    """The third stage's terms over the range of FP32 (aB times 2^la, E' times 2^lf).  Roundings: two where a
    warp's sum becomes FP64 and three of the four rows' additions; the factor -h/dz is a power of two."""
    nz = 4
    sim = _sim(nz, M)
    worst = 0.0
    for seed in range(12):
        rng = np.random.default_rng(1000 * M + seed)
        E1, aB = np.zeros((3, 1, 4, nz), np.float32), np.zeros((3, 1, 4, nz), np.float32)
        E1[1:] = np.ldexp(rng.normal(size=(2, 1, 4, nz)).astype(np.float32), lf)
        aB[1:] = np.ldexp(rng.normal(size=(2, 1, 4, nz)).astype(np.float32), la)
        got = _gradient(sim, M, E1, np.zeros_like(E1), aB, np.zeros_like(E1))
        ref, size = _third_stage(E1, aB, M, Fr(-1, 8))
        for l in range(M):
            if size[l]:
                worst = max(worst, float(abs(Fr(float(got[l])) - ref[l]) / size[l]))
            else:
                assert got[l] == 0.0
    assert worst <= 5 * U + 2.0 ** -60, worst
    sim.close()


@pytest.mark.parametrize("far", [1.0, np.inf])
def test_gradient_sums_where_large_cells_take_no_part(far):
    """Products 2^-100 of what the largest cells of the row could give: a warp that spans both, and one that
    spans an infinity that no term reads."""
    M, nz = 4, 120
    sim = _sim(nz, M)
    rng = np.random.default_rng(7)
    E1, aB = np.zeros((3, 1, 4, nz), np.float32), np.zeros((3, 1, 4, nz), np.float32)
    E1[1:, :, :, :12] = np.ldexp(rng.normal(size=(2, 1, 4, 12)).astype(np.float32), -100)
    aB[1:, :, :, :8] = rng.normal(size=(2, 1, 4, 8)).astype(np.float32)
    E1[1:, :, :, 100] = far
    got = _gradient(sim, M, E1, np.zeros_like(E1), aB, np.zeros_like(E1))
    E1[1:, :, :, 100] = 0.0                                  # (no cell with aB != 0 reaches it)
    ref, size = _third_stage(E1, aB, M, Fr(-1, 8))
    for l in range(M):
        # in FP64 from the first difference on: 16 terms, five shuffles, four warps, four rows
        assert abs(Fr(float(got[l])) - ref[l]) <= 32 * U * size[l]
    sim.close()


@pytest.mark.parametrize("M", [2, 5, 16])
@pytest.mark.parametrize("la,lj", [(0, 0), (-70, -60), (50, 70)])
def test_gradient_of_the_correction(M, la, lj):
    """dt <P^-1 aE1, P_l J1> for an aE1 of one cell per row, so that P^-1 aE1 is the taps themselves: 2 + 1 + 3
    FP64 roundings (rows of three warps; the factor dt is a power of two)."""
    nz = 96
    sim = _sim(nz, M)
    taps = sim.coefficients()[1].astype(np.float32)
    rng = np.random.default_rng(M)
    aE, J = np.zeros((3, 1, 4, nz), np.float32), np.zeros((3, 1, 4, nz), np.float32)
    aE[0, 0, :, 41] = np.ldexp(1.0, la)
    J[0] = np.ldexp(rng.normal(size=(1, 4, nz)).astype(np.float32), lj)
    got = _gradient(sim, M, np.zeros_like(aE), aE, np.zeros_like(aE), J)
    c = len(taps) // 2
    for l in range(1, M + 1):
        ref, size = Fr(0), Fr(0)
        for x in range(4):
            for m in range(-c, c + 1):
                v = Fr(float(np.ldexp(taps[c + m], la)))
                for k in range(-(l - 1), l):
                    t = Fr(1, 8) * v * _at(J[0, 0, x], 41 + m + k)
                    ref += t
                    size += abs(t)
        assert abs(Fr(float(got[l - 1])) - ref) <= 6 * U * size + size * Fr(1, 2 ** 60)
    sim.close()


def test_kinetic_energy():
    """gamma - 1 of one particle, from slow to fast and beyond the range of FP32 squares."""
    getcontext().prec = 60
    sim = _sim(16)
    rng = np.random.default_rng(2)
    for k in range(48):
        u = (rng.normal(size=3) * 2.0 ** rng.uniform(-14, 40 if k % 8 else 80)).astype(np.float32)
        if k % 5 == 0:
            u[1:] = 0.0
        one = np.ones(1, np.int64)
        sim.add_species(0, 8 * one, 2 * one, 0 * one, np.full((2, 1), 0.25, np.float32), u[:, None], -1.0, 1.0, 1.0)
        x = sum(Decimal(float(v)) ** 2 for v in u)
        ref = x / (1 + (1 + x).sqrt())
        got = Decimal(sim.diag()["kinetic"])
        assert abs(got - ref) <= 3 * Decimal(U) * ref, (u, got, ref)
    sim.close()


def _exact_gauss(E, C, h):
    _, _, nx, nz = E.shape
    G, size = np.empty((nx, nz), object), np.empty((nx, nz), object)
    for x in range(nx):
        for z in range(nz):
            a = [Fr(float(C[l])) * s * _at(E[0, 0, x], z + o) / h for l in range(len(C))
                 for s, o in ((1, l), (-1, -l - 1))]
            a += [_at(E[1, 0, x], z) / h, -_at(E[1, 0, (x - 1) % nx], z) / h]
            G[x, z], size[x, z] = sum(a), sum(abs(v) for v in a)
    return G, size


@pytest.mark.parametrize("M", [1, 3, 8, 16])
@pytest.mark.parametrize("lf", [0, -115, 100])
def test_gauss_residual(M, lf):
    """d-.E of random fields times 2^lf, without particles: two roundings where the axial sum becomes FP64, one of the
    x difference and three sums (the divisions by 1/2 are exact); out of the range of FP32 products FP64
    from the first difference on, M + 6."""
    nz = 21
    sim = _sim(nz, M)
    rng = np.random.default_rng(M)
    E = np.ldexp(rng.normal(size=(3, 1, 4, nz)).astype(np.float32), lf)
    sim.E.copy_(_dev(E))
    C = np.ones(1, np.float32) if M == 1 else sim.coefficients()[0].astype(np.float32)
    ref, size = _exact_gauss(E, C, Fr(1, 2))
    got = sim.gauss().cpu().numpy()[0]
    worst = max(float(abs(Fr(float(got[x, z])) - ref[x, z]) / size[x, z]) for x in range(4) for z in range(nz))
    assert worst <= (6 if lf == 0 else M + 6) * U, worst
    sim.close()


@pytest.mark.parametrize("M", [1, 3, 16])
def test_gauss_residual_of_infinite_fields(M):
    """A field that has overflowed shows: the nodes whose difference reads it are infinite or not a number as FP64
    has them, the others stay finite, and gauss_max is infinite."""
    nz, z0 = 160, 80
    sim = _sim(nz, M)
    E = np.ones((3, 1, 4, nz), np.float32)
    E[0, 0, 1, z0] = np.inf
    sim.E.copy_(_dev(E))
    got = sim.gauss().cpu().numpy()[0]
    hit = np.zeros((4, nz), bool)
    hit[1, z0 - M + 1:z0 + M + 1] = True
    assert np.array_equal(np.isinf(got), hit) and np.isfinite(got[~hit]).all()
    assert np.isinf(sim.diag()["gauss_max"])
    sim.close()


@pytest.mark.parametrize("ndim,shape", [(2, 1), (2, 2), (3, 1), (3, 2)])
def test_charge_density(ndim, shape):
    """rho of five particles in one cell.  Weights in units of 2^-63 and products in units of 2^-62 and 2^-61 put a
    contribution within 2^-59 of a particle's density; then three roundings of the node's sum."""
    nz, nx, ny = 12, 6, 6 if ndim == 3 else 1
    sim = Simulation(device="cuda:0", ndim=ndim, nz=nz, nx=nx, ny=ny, dz=0.5, dx=0.5, dy=0.5, dt=0.125, shape=shape)
    qv = Fr(-1) / Fr(1, 2) ** ndim
    rng = np.random.default_rng(10 * ndim + shape)
    for _ in range(6):
        off = rng.random((ndim, 5)).astype(np.float32)
        one = np.ones(5, np.int64)
        sim.add_species(0, 5 * one, 2 * one, 2 * one if ndim == 3 else 0 * one, off, np.zeros((3, 5), np.float32), -1.0, 1.0, 1.0)

        def weights(o):
            o = Fr(float(o))
            if shape == 1:
                return {0: 1 - o, 1: o}
            b = 1 if o >= Fr(1, 2) else 0
            d = o - b
            return {b - 1: (Fr(1, 2) - d) ** 2 / 2, b: Fr(3, 4) - d * d, b + 1: (Fr(1, 2) + d) ** 2 / 2}

        ref = {}
        for p in range(5):
            w = [weights(off[a, p]) for a in range(ndim)] + ([{0: Fr(1)}] if ndim == 2 else [])
            for a, wa in w[0].items():
                for b, wb in w[1].items():
                    for c, wc in w[2].items():
                        n = (c + 2 if ndim == 3 else 0, b + 2, a + 5)
                        ref[n] = ref.get(n, Fr(0)) + qv * wa * wb * wc
        got = sim.rho().cpu().numpy()
        for n, v in ref.items():
            assert abs(Fr(float(got[n])) - v) <= 3 * U * abs(v) + 5 * abs(qv) * Fr(1, 2 ** 59)
    sim.close()


def test_charge_density_of_an_offset_that_is_not_a_number():
    sim = _sim(16, nx=8, shape=2)
    one = np.ones(3, np.int64)
    off = np.full((2, 3), 0.25, np.float32)
    off[0, 1] = np.nan
    sim.add_species(0, 8 * one, 4 * one, 0 * one, off, np.zeros((3, 3), np.float32), -1.0, 1.0, 1.0)
    bad = np.isnan(sim.rho().cpu().numpy()[0])
    assert bad[3:6, 7:10].all() and bad.sum() == 9
    sim.close()
