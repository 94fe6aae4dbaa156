"""Time-fused launches of large lattices: whole waves of tall marches, four steps each, in the unrolled
form (one model) and the rolled one (several), over even and odd rows, against the register-staged
kernels, bit for bit.  No tolerance is involved."""

import pytest

torch = pytest.importorskip("torch")
np = pytest.importorskip("numpy")

from paper_2002_05265_gb300 import flows

pytestmark = pytest.mark.gpu

MODELS = ["bgk", "rm", "hm", "cm", "chm", "k", "pr", "rr"]
RATES = (1.9, 1.3, 0.9)


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2002_05265_gb300 import lbm
    return lbm


_FIELDS = {}


def _fields(nx, ny):
    if (nx, ny) not in _FIELDS:
        _FIELDS.clear()
        noise = flows.random_populations_perturbation((3, ny, nx), 0.01, nx + ny)
        _FIELDS[nx, ny] = [torch.from_numpy(np.ascontiguousarray(f + d)).cuda()
                           for f, d in zip(flows.vortex(nx, ny, Ma=0.2, seed=nx), noise)]
    return _FIELDS[nx, ny]


def _lattices(L, shape, models, storage, shift, path):
    out = []
    for m in models:
        lat = L.Lattice(shape[0], shape[1], m, RATES, storage=L.STORAGES[storage])
        if shift:
            lat.set_shift_velocity(0.1, -0.02)
        lat.set_kernel_path(path)
        lat.init_equilibrium(*_fields(*shape))
        out.append(lat)
    return out


def _same(a, b):
    shape = (9, a.ny, a.nx)
    f, g = (torch.empty(shape, dtype=torch.float64, device="cuda") for _ in range(2))
    a.get_populations(f)
    b.get_populations(g)
    return torch.equal(f, g)


@pytest.mark.parametrize("shift", [False, True])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("models", [["k"], ["bgk"], ["chm", "rr"]])
@pytest.mark.parametrize("shape", [(2048, 2100), (2049, 2100)])
def test_tall_marches_of_four_steps(L, shape, models, storage, shift):
    """77,700 strip-rows a lattice: one wave of resident warps that march 32 rows for one lattice,
    two for two lattices of different models.  Recorded runs of four steps take one launch each."""
    fused = _lattices(L, shape, models, storage, shift, L.LBM_PATH_AUTO)
    plain = _lattices(L, shape, models, storage, shift, L.LBM_PATH_VECTOR)
    g = L.lbm_group_create([x.ctx for x in fused], graph_steps=4)
    L.lbm_group_set_timing(g)
    done = 0
    for n in (4, 7, 37):
        L.lbm_group_step(g, n)
        done += n
        for lat in plain:
            lat.step(n)
        for m, a, b in zip(models, fused, plain):
            assert _same(a, b), (m, done)
            assert a.status() == (L.LBM_OK, -1, done)
    _, lattice_steps, launches = L.lbm_group_timing(g)
    assert lattice_steps == 44 * len(models) and launches == 11
    L.lbm_group_destroy(g)
    for lat in fused + plain:
        lat.close()
