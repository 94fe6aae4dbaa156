"""Time-fused launches (several time steps of every lattice in one launch): each node update does
the arithmetic of the one-step kernels, value for value, so the states agree bit for bit with the
register-staged kernels whatever the lattice, the number of steps and how the launches split them.
No tolerance is involved.  Sizes cover strips with and without remainder (56 stored columns at
four steps), odd widths (no paired loads), lattices narrower than a strip and of few rows, and more
rows than warps."""

import pytest

torch = pytest.importorskip("torch")
np = pytest.importorskip("numpy")

from paper_2002_05265_gb300 import flows

pytestmark = pytest.mark.gpu

MODELS = ["bgk", "rm", "hm", "cm", "chm", "k", "pr", "rr"]


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2002_05265_gb300 import lbm
    return lbm


def _fields(nx, ny, seed):
    rho, ux, uy = flows.vortex(nx, ny, Ma=0.2, seed=seed)
    noise = flows.random_populations_perturbation((3, ny, nx), 0.01, seed)
    return [torch.from_numpy(np.ascontiguousarray(f + d)).cuda() for f, d in zip((rho, ux, uy), noise)]


def _state(lat):
    f = torch.empty((9, lat.ny, lat.nx), dtype=torch.float64, device="cuda")
    lat.get_populations(f)
    return f


def _lattice(L, shape, model, storage, shift, path):
    rates = (1.9, 1.3, 0.9)
    lat = L.Lattice(shape[0], shape[1], model, rates, storage=L.STORAGES[storage])
    if shift:
        lat.set_shift_velocity(0.1, -0.02)
    lat.set_kernel_path(path)
    lat.init_equilibrium(*_fields(*shape, seed=sum(shape)))
    return lat


@pytest.mark.parametrize("shift", [False, True])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("shape", [(3, 3), (4, 5), (56, 40), (57, 41), (112, 9), (130, 300), (1001, 64), (2300, 70)])
def test_fused_steps_equal_single_steps(L, shape, storage, shift):
    for model in MODELS:
        for calls in ((2,), (7, 3), (37,)):
            fused = _lattice(L, shape, model, storage, shift, L.LBM_PATH_AUTO)
            plain = _lattice(L, shape, model, storage, shift, L.LBM_PATH_VECTOR)
            for n in calls:
                fused.step(n)
                plain.step(n)
            assert torch.equal(_state(fused), _state(plain)), (model, calls)
            assert fused.status()[2] == sum(calls)
            fused.close()
            plain.close()


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("models", [MODELS, ["k", "k", "k"]])
def test_fused_group_of_unequal_lattices(L, models, storage):
    """One launch over lattices of unequal sizes, of one model and of all, with checks between
    recorded graphs: every lattice as if stepped alone."""
    shapes = [(64 + 37 * k, 40 + 11 * k) for k in range(len(models))]
    lats = [_lattice(L, s, m, storage, False, L.LBM_PATH_AUTO) for s, m in zip(shapes, models)]
    for k, lat in enumerate(lats):
        lat.set_check(10 + k)
    g = L.lbm_group_create([x.ctx for x in lats], graph_steps=6)
    for n in (53, 1, 24):
        L.lbm_group_step(g, n)
    for lat, s, m in zip(lats, shapes, models):
        alone = _lattice(L, s, m, storage, False, L.LBM_PATH_VECTOR)
        alone.step(78)
        assert torch.equal(_state(lat), _state(alone)), (m, s)
        assert lat.status() == (L.LBM_OK, -1, 78)
        alone.close()
    L.lbm_group_destroy(g)
    for lat in lats:
        lat.close()


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("check", [0, 7, 50])
def test_fused_batch_equals_lattices(L, storage, check):
    """Instances of a sweep, fused between checks, against lattices of the register-staged kernels
    stored around the same mean flow: narrow, odd, wide and flat ones, every model, bit for bit."""
    shapes = [(32, 33), (57, 3), (61, 140), (64, 64), (113, 200), (256, 17), (3, 256), (200, 35)]
    u = [(0.05 + 0.01 * k, 0.02 - 0.01 * k) for k in range(len(shapes))]
    descs = [dict(nx=nx, ny=ny, model=m, rates=(1.9, 1.3, 0.9), ux_ref=a, uy_ref=b)
             for (nx, ny), m, (a, b) in zip(shapes, MODELS, u)]
    fields = [_fields(nx, ny, nx + ny) for nx, ny in shapes]
    b = L.lbm_batch_create(descs, storage=L.STORAGES[storage])
    L.lbm_batch_init_equilibrium(b, *[torch.cat([f[i].flatten() for f in fields]) for i in range(3)])
    for target in (41, 42, 103):
        L.lbm_batch_run(b, target, check_every=check, growth=1e12)
    status, _, steps, _ = L.lbm_batch_status(b, len(descs))
    assert list(status) == [0] * len(descs) and list(steps) == [103] * len(descs)
    for k, ((nx, ny), m) in enumerate(zip(shapes, MODELS)):
        lat = L.Lattice(nx, ny, m, (1.9, 1.3, 0.9), storage=L.STORAGES[storage])
        lat.set_shift_velocity(*u[k])
        lat.set_kernel_path(L.LBM_PATH_VECTOR)
        lat.init_equilibrium(*fields[k])
        lat.step(103)
        got = torch.empty((9, ny, nx), dtype=torch.float64, device="cuda")
        L.lbm_batch_get_populations(b, k, got)
        assert torch.equal(got, _state(lat)), (m, nx, ny)
        lat.close()
    L.lbm_batch_destroy(b)
