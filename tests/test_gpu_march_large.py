"""Time-fused launches of large lattices: whole waves of tall marches, four steps each, in the unrolled
form (one model) and the rolled one (several), over even and odd rows -- against the register-staged
kernels, bit for bit -- and the copy-engine launches that the library's own choice took before it
marched.  No tolerance is involved."""

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


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("models", [MODELS, ["bgk", "rm", "hm", "pr"]])
def test_copy_engine_group_of_1024_lattices(L, models, storage):
    """The benchmark's group of 1024 x 1024 lattices in one copy-engine launch a step."""
    staged = _lattices(L, (1024, 1024), models, storage, False, L.LBM_PATH_BULK)
    plain = _lattices(L, (1024, 1024), models, storage, False, L.LBM_PATH_VECTOR)
    g = L.lbm_group_create([x.ctx for x in staged], graph_steps=8)
    assert L.lbm_group_describe(g)["family"] == L.LBM_PATH_BULK
    L.lbm_group_step(g, 21)
    for m, a, b in zip(models, staged, plain):
        b.step(21)
        assert _same(a, b), m
        assert a.status() == (L.LBM_OK, -1, 21)
    L.lbm_group_destroy(g)
    for lat in staged + plain:
        lat.close()


@pytest.mark.parametrize("storage", ["f16", "bf16"])
def test_copy_engine_at_16384(L, storage):
    """The 16384 x 16384 16-bit lattice, one copy-engine launch a step: rho and u of every node."""
    n = 16384
    x = torch.arange(n, device="cuda", dtype=torch.float64) * (2 * np.pi / n)
    ux = 0.1 + 0.05 * torch.sin(3 * x)[:, None] * torch.cos(5 * x)[None, :]
    uy = 0.04 * torch.cos(2 * x)[:, None] * torch.sin(7 * x)[None, :]
    rho = torch.ones_like(ux)
    out = []
    for path in (L.LBM_PATH_BULK, L.LBM_PATH_VECTOR):
        lat = L.Lattice(n, n, "chm", RATES, storage=L.STORAGES[storage])
        lat.set_shift_velocity(0.1, 0.0)
        lat.set_kernel_path(path)
        lat.init_equilibrium(rho, ux, uy)
        lat.step(8)
        assert lat.status()[0] == L.LBM_OK
        fields = [torch.empty_like(ux) for _ in range(3)]
        lat.moments(*fields)
        lat.close()
        out.append(fields)
    for a, b in zip(*out):
        assert torch.equal(a, b)
    del out, fields, rho, ux, uy
    torch.cuda.empty_cache()


@pytest.mark.parametrize("shape,storage,launches", [
    ((3, 30000), "f16", 4), ((3, 30000), "f32", 4), ((21, 30000), "f32", 4), ((15, 30000), "f16", 4),
    ((1000001, 4), "f16", 4), ((701, 699), "f16", 4),
    ((8, 100000), "f16", 1), ((24, 30000), "f32", 1), ((52, 30000), "f32", 1), ((2001, 1999), "f16", 1)])
def test_narrow_and_flat_lattices_are_not_fused(L, shape, storage, launches):
    """Launches of a recorded run of four steps, by shape, and the state they leave."""
    nx, ny = shape
    x, y = (torch.arange(n, device="cuda", dtype=torch.float64) * (2 * np.pi / n) for n in (nx, ny))
    f = [1 + 0 * y[:, None] + 0 * x[None, :], 0.05 * torch.sin(y)[:, None] * torch.cos(x)[None, :],
         0.04 * torch.cos(2 * y)[:, None] + 0 * x[None, :]]
    lats = []
    for path in (L.LBM_PATH_AUTO, L.LBM_PATH_VECTOR):
        lat = L.Lattice(nx, ny, "k", RATES, storage=L.STORAGES[storage])
        lat.set_kernel_path(path)
        lat.init_equilibrium(*[v.contiguous() for v in f])
        lats.append(lat)
    g = L.lbm_group_create([lats[0].ctx], graph_steps=4)
    L.lbm_group_set_timing(g)
    L.lbm_group_step(g, 12)
    lats[1].step(12)
    assert _same(*lats)
    _, steps, n = L.lbm_group_timing(g)
    assert (steps, n) == (12, 3 * launches)
    L.lbm_group_destroy(g)
    for lat in lats:
        lat.close()
