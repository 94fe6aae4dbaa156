"""Fields of nodes far from rho = rho0 and of populations far from 1, against long double: densities
next to nothing, populations whose sums leave the FP32 range, and large reference densities."""

import pytest

torch = pytest.importorskip("torch")
np = pytest.importorskip("numpy")

pytestmark = pytest.mark.gpu

EX, EY = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)
W = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2002_05265_gb300 import lbm
    return lbm


def _fields_of(L, f, storage, rho0, shift=(0.0, 0.0)):
    """(populations as stored, the six moments) of a lattice set to f."""
    _, ny, nx = f.shape
    lat = L.Lattice(nx, ny, "chm", (1.5, 1.2, 1.0), storage=L.STORAGES[storage], rho0=rho0)
    if shift != (0.0, 0.0):
        lat.set_shift_velocity(*shift)
    lat.set_populations(torch.from_numpy(np.ascontiguousarray(f)).cuda())
    stored = torch.empty((9, ny, nx), dtype=torch.float64, device="cuda")
    lat.get_populations(stored)
    out = [torch.empty((ny, nx), dtype=torch.float64, device="cuda") for _ in range(6)]
    lat.moments(*out)
    lat.close()
    return stored.cpu().numpy(), [o.cpu().numpy() for o in out]


@pytest.mark.parametrize("shift", [(0.0, 0.0), (0.1, -0.04)])
@pytest.mark.parametrize("storage", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("nx", [33, 64])
def test_velocity_of_thin_nodes(L, storage, nx, shift):
    """Densities from 1 down to 1e-8 of rho0.  A population read back carries 2^-54 of rounding and
    the sum closes with 2^-53 of rho0 = 1, together below 1e-15 of density and momentum: a velocity
    is within 1e-15 (1 + |u|) / rho of the one summed here."""
    g = np.random.Generator(np.random.Philox(3))
    rho = 10.0 ** g.uniform(-8, 0, (24, nx))
    stored, (r, ux, uy, *_) = _fields_of(L, rho * W[:, None, None] * (1 + 0.3 * g.uniform(-1, 1, (9, 24, nx))), storage, 1.0, shift)
    f = stored.astype(np.longdouble)
    want = sum(f)
    ok = np.abs(want) > 1e-9
    assert np.all(np.abs(r - want) <= 1e-15)
    for got, e in ((ux, EX), (uy, EY)):
        u = sum(e[i] * f[i] for i in range(9))[ok] / want[ok]
        off = np.abs(got[ok] - u) * np.abs(want[ok]) / (1 + np.abs(u))
        assert float(np.max(off)) <= 1e-15, float(np.max(off))


@pytest.mark.parametrize("storage", ["f64", "f32", "bf16"])
def test_second_moments_beyond_the_fp32_range(L, storage):
    """Populations of 2^127 that cancel in rho and j but not in Pi (2^128 is no FP32 number): every
    sum is exact in FP64."""
    f = np.ones((9, 5, 33)) * W[:, None, None]
    big = np.zeros((5, 33), bool)
    big[2, 7] = big[4, 32] = True
    for i, v in ((0, 0.0), (1, 1.0), (2, -1.0), (3, 1.0), (4, -1.0), (5, 0.0), (6, 0.0), (7, 0.0), (8, 0.0)):
        f[i][big] = v * 2.0 ** 127
    _, (rho, ux, uy, pxx, pxy, pyy) = _fields_of(L, f, storage, 1.0)
    assert np.all(pxx[big] == 2.0 ** 128) and np.all(pyy[big] == -(2.0 ** 128))
    assert np.all(np.abs(pxy[big]) <= 1.0) and np.all(np.isfinite(rho)) and np.all(np.isfinite(ux)) and np.all(np.isfinite(uy))
    assert np.all(np.abs(pxx[~big] - 1 / 3) <= (2e-2 if storage == "bf16" else 1e-6))


@pytest.mark.parametrize("rho0", [1e-30, 1.1, 2.0 ** 60, 2.0 ** 120])
@pytest.mark.parametrize("storage", ["f64", "f32"])
def test_moments_at_any_reference_density(L, storage, rho0):
    """Velocities and stresses scale with nothing: those of populations c f about c rho0 are those of
    f.  Rounding: that of a population read back and of the sums, 1e-15 of rho0 as above."""
    g = np.random.Generator(np.random.Philox(4))
    f = rho0 * W[:, None, None] * (1 + 0.3 * g.uniform(-1, 1, (9, 6, 35)))
    stored, out = _fields_of(L, f, storage, rho0)
    s = stored.astype(np.longdouble) / rho0
    m = lambda p, q: sum(EX[i] ** p * EY[i] ** q * s[i] for i in range(9))
    rho = m(0, 0)
    for got, want, scale in zip(out, (rho, m(1, 0) / rho, m(0, 1) / rho, m(2, 0), m(1, 1), m(0, 2)),
                                (rho0, 1.0, 1.0, rho0, rho0, rho0)):
        off = np.abs(got / scale - want)
        assert float(np.max(off)) <= 2e-15, float(np.max(off))


def _phi(s, u):
    return np.longdouble(2) / 3 - u * u if s == 0 else (u * u + s * u + np.longdouble(1) / 3) / 2


@pytest.mark.parametrize("storage,precision", [("f32", 24), ("f16", 11), ("bf16", 8)])
@pytest.mark.parametrize("uref", [(0.0, 0.0), (0.9, 0.9), (-0.99, 0.3), (0.8164965, -0.8164966)])
def test_equilibrium_far_from_the_reference_velocity(L, storage, precision, uref):
    """2^20 nodes with |u| up to 1.9 about reference velocities up to 0.99: every stored g = f^eq - s
    lies within half a unit in the last place of its exact value; 2^-49 allowed for its FP64
    evaluation, terms of size up to 8 in FP64 (2^-52 of them), and for reading f = g + s back."""
    n = 1024
    g = np.random.Generator(np.random.Philox(8))
    rho = 1.0 + 0.2 * g.uniform(-1, 1, (n, n))
    ux, uy = (-r + g.uniform(-1, 1, (n, n)) if r else g.uniform(-1, 1, (n, n)) for r in uref)
    lat = L.Lattice(n, n, "chm", (1.9, 1.2, 0.9), storage=L.STORAGES[storage])
    if uref != (0.0, 0.0):
        lat.set_shift_velocity(*uref)
    lat.init_equilibrium(*[torch.from_numpy(v).cuda() for v in (rho, ux, uy)])
    f = torch.empty((9, n, n), dtype=torch.float64, device="cuda")
    lat.get_populations(f)
    lat.close()
    f = f.cpu().numpy()
    R, X, Y = (v.astype(np.longdouble) for v in (rho, ux, uy))
    ur = [np.longdouble(v) for v in uref]
    for i in range(9):
        s = _phi(EX[i], ur[0]) * _phi(EY[i], ur[1])
        want = R * _phi(EX[i], X) * _phi(EY[i], Y) - s
        off = np.abs(f[i] - s - want).astype(np.float64)
        half = 2.0 ** (np.floor(np.log2(np.maximum(np.abs(want).astype(np.float64), 1e-300))) - precision)
        if storage == "f16":
            half = np.maximum(half, 2.0 ** -25)   # subnormal halves
        bad = off > half + 2.0 ** -49
        assert not bad.any(), (i, int(bad.sum()), float(np.max((off - half)[bad])))
