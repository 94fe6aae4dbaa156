"""Fields in and out of 32- and 16-bit lattices: the initial equilibrium is rounded to the storage
type as FP64 arithmetic rounds it, moments are those of FP64 sums, and nodes with non-finite values
report them as plain FP64 arithmetic does.  Odd widths leave half a pair of nodes at the row's end."""

import pytest

torch = pytest.importorskip("torch")
np = pytest.importorskip("numpy")

pytestmark = pytest.mark.gpu

EX, EY = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)
PRECISION = {"f32": 24, "f16": 11, "bf16": 8}
SHAPES = [(3, 3), (67, 37), (64, 20), (257, 5)]


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2002_05265_gb300 import lbm
    return lbm


def _phi(s, u):
    return 2.0 / 3.0 - u * u if s == 0 else 0.5 * (u * u + s * u + 1.0 / 3.0)


def _fields(nx, ny, amp, seed):
    g = np.random.Generator(np.random.Philox(seed))
    rho, ux, uy = 1.0 + 0.1 * amp * g.uniform(-1, 1, (ny, nx)), amp * g.uniform(-1, 1, (ny, nx)), amp * g.uniform(-1, 1, (ny, nx))
    ux[0, 0] = uy[0, 0] = 0.0
    rho[0, :] = 1.0
    return rho, ux, uy


def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _lattice(L, shape, storage, shift):
    lat = L.Lattice(shape[0], shape[1], "chm", (1.9, 1.2, 0.9), storage=L.STORAGES[storage])
    if shift != (0.0, 0.0):
        lat.set_shift_velocity(*shift)
    return lat


def _populations(lat):
    f = torch.empty((9, lat.ny, lat.nx), dtype=torch.float64, device="cuda")
    lat.get_populations(f)
    return f.cpu().numpy()


@pytest.mark.parametrize("shift", [(0.0, 0.0), (0.1, -0.04)])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("amp", [1e-5, 0.1, 0.95])
def test_initial_equilibrium_is_rounded_from_fp64(L, shape, storage, shift, amp):
    """Every stored g_i = f^eq_i - s_i lies within half a unit in the last place of the storage type
    of its FP64 value (2^-52 allowed for that value's own rounding and for reading f back)."""
    rho, ux, uy = _fields(*shape, amp, seed=7)
    lat = _lattice(L, shape, storage, shift)
    lat.init_equilibrium(_cuda(rho), _cuda(ux), _cuda(uy))
    f = _populations(lat)
    lat.close()
    for i in range(9):
        s = _phi(EX[i], shift[0]) * _phi(EY[i], shift[1])
        want = (rho * _phi(EX[i], ux) * _phi(EY[i], uy)).astype(np.longdouble) - s
        got = f[i].astype(np.longdouble) - s
        half = 2.0 ** (np.floor(np.log2(np.maximum(np.abs(want), 1e-300).astype(np.float64))) - PRECISION[storage])
        if storage == "f16":
            half = np.maximum(half, 2.0 ** -25)   # subnormal halves
        assert np.all(np.abs(got - want) <= half * (1 + 2.0 ** -10) + 2.0 ** -52), (i, float(np.max(np.abs(got - want) / half)))


@pytest.mark.parametrize("shift", [(0.0, 0.0), (0.1, -0.04)])
@pytest.mark.parametrize("storage", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("shape", SHAPES)
def test_moments_are_fp64_sums(L, shape, storage, shift):
    """rho, u and Pi of the stored state against long double sums of its populations: each of the
    nine populations read back carries up to 2^-54 of rounding, the result's own rounding is 2^-53 of
    about 1, together below 5e-16."""
    lat = _lattice(L, shape, storage, shift)
    lat.init_equilibrium(*[_cuda(v) for v in _fields(*shape, 0.1, seed=9)])
    lat.step(5)
    f = _populations(lat).astype(np.longdouble)
    out = [torch.empty((shape[1], shape[0]), dtype=torch.float64, device="cuda") for _ in range(6)]
    lat.moments(*out)
    lat.close()
    m = lambda p, q: sum(EX[i] ** p * EY[i] ** q * f[i] for i in range(9))
    rho = m(0, 0)
    for got, want in zip(out, (rho, m(1, 0) / rho, m(0, 1) / rho, m(2, 0), m(1, 1), m(0, 2))):
        assert float(np.max(np.abs(got.cpu().numpy() - want))) <= 5e-16


@pytest.mark.parametrize("storage", ["f64", "f32", "f16", "bf16"])
def test_moments_of_non_finite_nodes(L, storage):
    """Infinite and undefined populations and an empty node: rho and u are non-finite where plain
    FP64 sums over all nine populations are, and of the same kind."""
    nx, ny = 33, 6
    lat = _lattice(L, (nx, ny), storage, (0.0, 0.0))
    f = np.array([[[_phi(EX[i], 0.0) * _phi(EY[i], 0.0)]] for i in range(9)]) * np.ones((9, ny, nx))
    f[3, 1, 4] = np.inf
    f[0, 2, 32] = -np.inf
    f[1, 3, 9], f[3, 3, 9] = np.inf, -np.inf
    f[5, 4, 0] = np.nan
    f[:, 5, 17] = 0.0
    lat.set_populations(_cuda(f))
    out = [torch.empty((ny, nx), dtype=torch.float64, device="cuda") for _ in range(3)]
    lat.moments(*out)
    stored = _populations(lat)
    lat.close()
    with np.errstate(invalid="ignore", divide="ignore"):
        g = [stored[i] - _phi(EX[i], 0.0) * _phi(EY[i], 0.0) for i in range(9)]
        rho = 1.0 + sum(g)
        ux, uy = sum(EX[i] * g[i] for i in range(9)) / rho, sum(EY[i] * g[i] for i in range(9)) / rho
    rho[5, 17] = np.nan   # (0 or a rounding of it: nothing is asked of u there)
    for got, want in zip(out, (rho, ux, uy)):
        got = got.cpu().numpy()
        got[5, 17] = want[5, 17] = 0.0
        assert np.array_equal(np.isnan(got), np.isnan(want))
        assert np.array_equal(np.isposinf(got), np.isposinf(want)) and np.array_equal(np.isneginf(got), np.isneginf(want))
        fin = np.isfinite(want)
        assert float(np.max(np.abs(got[fin] - want[fin]))) <= 5e-16
