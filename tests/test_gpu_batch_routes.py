"""Sweeps whose instances march between checks, step one at a time, or do both side by side, by size,
number, check interval and kernel shape: every instance against its lattice in the register-staged
kernels, bit for bit.  120 x 130 and 192 x 150 march where many are at work, 193 x 151 has odd rows,
16 x 16 and 5 x 90 never march."""

import pytest

torch = pytest.importorskip("torch")
np = pytest.importorskip("numpy")

pytestmark = pytest.mark.gpu

MODELS = ["bgk", "rm", "hm", "cm", "chm", "k", "pr", "rr"]
RATES = (1.9, 1.3, 0.9)


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2002_05265_gb300 import lbm
    return lbm


def _fields(nx, ny):
    x, y = (torch.arange(n, device="cuda", dtype=torch.float64) * (2 * np.pi / n) for n in (nx, ny))
    u = 0.05 + 0.04 * torch.sin(y)[:, None] * torch.cos(x)[None, :]
    return [torch.ones_like(u), u, 0.03 * torch.cos(2 * y)[:, None] + 0 * u]


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("block", [None, 128, 256, 512])
@pytest.mark.parametrize("sizes", [[(16, 16)] * 40 + [(5, 90)] * 8,
                                   [(192, 150)] * 152 + [(193, 151)] * 8 + [(120, 130)] * 8 + [(16, 16)] * 8],
                         ids=["small", "mixed"])
def test_every_route_steps_alike(L, sizes, block, storage):
    descs = [dict(nx=nx, ny=ny, model=MODELS[k % 8], rates=RATES, ux_ref=0.05, uy_ref=0.0) for k, (nx, ny) in enumerate(sizes)]
    b = L.lbm_batch_create(descs, storage=L.STORAGES[storage])
    f = {s: _fields(*s) for s in set(sizes)}
    L.lbm_batch_init_equilibrium(b, *[torch.cat([f[s][i].flatten() for s in sizes]) for i in range(3)])
    if block:
        L.lbm_batch_set_shape(b, 4 if storage == "f32" or block < 512 else 8, block)
    for target, check in ((9, 0), (23, 100), (31, 2), (47, 5), (48, 1)):   # one kernel and another
        L.lbm_batch_run(b, target, check_every=check, growth=1e12)
    status, _, steps, _ = L.lbm_batch_status(b, len(descs))
    assert not status.any() and (steps == 48).all()
    picked = list(range(8)) + list(range(len(sizes) - 24, len(sizes)))
    for k in picked:
        nx, ny = sizes[k]
        lat = L.Lattice(nx, ny, MODELS[k % 8], RATES, storage=L.STORAGES[storage])
        lat.set_shift_velocity(0.05, 0.0)
        lat.set_kernel_path(L.LBM_PATH_VECTOR)
        lat.init_equilibrium(*f[sizes[k]])
        lat.step(48)
        got, want = (torch.empty((9, ny, nx), dtype=torch.float64, device="cuda") for _ in range(2))
        L.lbm_batch_get_populations(b, k, got)
        lat.get_populations(want)
        lat.close()
        assert torch.equal(got, want), (k, nx, ny)
    L.lbm_batch_destroy(b)
