"""Performance cases of the D2Q9 library: what a user of it has it do, through its public calls.

A lattice case is one simulation as a program runs it: the initial equilibrium from (rho, u), the
time steps, the macroscopic fields at the end.  A group case advances the lattices of a model
comparison together with their blow-up checks; a restart case resumes a checkpoint, advances it and
writes the next one; a sweep case is a numerical-stability study of many small lattices; an adjoint
case is a gradient of a run's misfit; a linear-stability case is a map of growth rates.

Flows are those of the method's paper (convected vortex, double shear layer, uniform flow), their
position, strength or phase drawn from the seed.  Viscosities and Mach numbers lie where the flow's
digits are reproducible: a flow that blows up amplifies its own rounding.  The fields of a run come
back in the type its populations are stored in, FP64 for FP64.
"""

import math

import numpy as np
import torch

from paper_2002_05265_gb300 import lbm
from paper_2002_05265_gb300.adjoint import LBMRun

CS = 1.0 / math.sqrt(3.0)
MODELS = ("bgk", "rm", "hm", "cm", "chm", "k", "pr", "rr")
# FP32 operations of one node's stream-and-collide update (multiply, add; a fused pair counts as two)
UPDATE_FLOPS = {"bgk": 109, "rm": 109, "hm": 113, "cm": 129, "chm": 133, "k": 141, "pr": 104, "rr": 126}
FIELD_TYPE = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
GROUP_CHECK = 100
GRAPH_STEPS = 100
SWEEP_CHECK = 100


def listed():
    return [
        # the smallest call: a few steps of a ragged lattice of the unit-test kind, latency only
        dict(name="ragged_67x37_f64", kind="lattice", nx=67, ny=37, model="chm", preset="reg", storage="f64",
             nu=1e-3, ma=0.2, steps=20, shift=False, check=0),
        # the paper's convected vortex on its small lattice in full precision: a validation run
        dict(name="vortex_128_f64", kind="lattice", nx=128, ny=128, model="bgk", preset="srt", storage="f64",
             nu=1e-4, ma=0.1, steps=1000, shift=False, check=0),
        # the long-distance transport study at L = 256, stored around the mean flow, watched for blow-up
        dict(name="transport_256_f32", kind="lattice", nx=256, ny=256, model="rr", preset="srt", storage="f32",
             nu=1e-3, ma=0.3, steps=1000, shift=True, check=100),
        # an odd-sized lattice whose rows no copy engine can take
        dict(name="ragged_1001x777_f32", kind="lattice", nx=1001, ny=777, model="k", preset="reg", storage="f32",
             nu=1e-4, ma=0.2, steps=200, shift=False, check=0),
        # the model comparison: the eight models on the 1024 x 1024 double shear layer, checked as they run
        dict(name="shear_1024_x8_f32", kind="group", n=1024, models="all", storage="f32", nu=1e-5, ma=0.1, steps=200),
        # reduced-precision storage on a lattice of ordinary size
        dict(name="vortex_2048_f16", kind="lattice", nx=2048, ny=2048, model="rr", preset="srt", storage="f16",
             nu=1e-4, ma=0.2, steps=200, shift=True, check=0),
        dict(name="vortex_4096_bf16", kind="lattice", nx=4096, ny=4096, model="chm", preset="reg", storage="bf16",
             nu=1e-5, ma=0.2, steps=200, shift=False, check=0),
        # resume a checkpoint, advance, write the next checkpoint and the run's diagnostics
        dict(name="restart_2048_f32", kind="restart", nx=2048, ny=2048, model="cm", preset="reg", storage="f32",
             nu=1e-4, ma=0.1, steps=100),
        # the largest lattice: the throughput run of vortex convection
        dict(name="vortex_16384_f32", kind="lattice", nx=16384, ny=16384, model="k", preset="reg", storage="f32",
             nu=1e-6, ma=0.2, steps=96, shift=False, check=0),
        # the numerical-stability study: lattices of uneven sizes 32..256, every model, both rate presets
        dict(name="sweep_1024_f32", kind="sweep", instances=1024, steps=1000, storage="f32"),
        # gradient of a run's misfit with respect to the initial velocity and the rates
        dict(name="adjoint_512_f32", kind="adjoint", nx=512, ny=512, model="chm", storage="f32", nu=1e-4, ma=0.1,
             steps=1000),
        # growth rates over a wavenumber grid for several mean flows
        dict(name="growth_16x64x64", kind="growth", model="k", preset="reg", nu=1e-3, flows=16, nk=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lattice"] * 5 + ["group", "group", "restart", "sweep", "adjoint", "growth"])
    model = rng.choice(MODELS)
    preset = "srt" if model in ("bgk", "rr") else "reg"
    ma = round(rng.uniform(0.05, 0.2), 3)
    nu = float("%.3g" % math.exp(rng.uniform(math.log(1e-4), math.log(1e-2))))
    if kind in ("lattice", "restart"):
        # areas over 2^11 .. 2^28 (2^24 for a restart) with aspect ratios up to 2; a multiple of
        # 32 in x half of the time, any width otherwise; the steps keep the work below the largest listed
        area = math.exp(rng.uniform(math.log(2.0 ** 11), math.log(2.0 ** (28 if kind == "lattice" else 24))))
        aspect = 2.0 ** rng.uniform(-1.0, 1.0)
        nx = max(32, int(math.sqrt(area * aspect)))
        if rng.random() < 0.5:
            nx = nx // 32 * 32
        ny = max(32, min(int(area / nx), 2 ** 28 // nx))
        storage = rng.choice(["f32", "f32", "f32", "f16", "bf16", "f64"])
        most = (1e9 if storage == "f64" else 8e9) / (nx * ny)
        steps = max(2, min(_log_int(rng, 16, 1000), int(most)))
        case = dict(kind=kind, nx=nx, ny=ny, model=model, preset=preset, storage=storage, nu=nu, ma=ma, steps=steps)
        if kind == "lattice":
            case.update(shift=rng.random() < 0.4, check=rng.choice([0, 0, 50]))
        return case
    if kind == "group":
        n = rng.choice([64, 96, 200, 256, 384, 500, 512, 768, 1000, 1024, 1536])
        return dict(kind="group", n=n, models=rng.choice(["all", "bgk,rm,hm,pr", "cm,chm,k,rr", "chm,k"]),
                    storage=rng.choice(["f32", "f32", "f16", "bf16"]), nu=nu, ma=ma,
                    steps=min(_log_int(rng, 50, 800), int(3e9 / (8 * n * n))))
    if kind == "sweep":
        instances = _log_int(rng, 64, 1024)
        return dict(kind="sweep", instances=instances, steps=min(_log_int(rng, 100, 2000), 1000000 // instances),
                    storage="f32")
    if kind == "adjoint":
        nx, ny = rng.randint(64, 512), rng.randint(64, 512)
        return dict(kind="adjoint", nx=nx, ny=ny, model=model, storage=rng.choice(["f32", "f32", "f64"]), nu=nu, ma=ma,
                    steps=_log_int(rng, 50, 600))
    return dict(kind="growth", model=model, preset=preset, nu=nu, flows=rng.randint(1, 16), nk=rng.randint(8, 64))


def _rates(nu, preset):
    w = 1.0 / (3.0 * nu + 0.5)
    return (w, w, w) if preset == "srt" else (w, 1.0, 1.0)


def _rng(seed):
    return np.random.Generator(np.random.Philox(seed))


def _vortex(nx, ny, ma, xc, yc, beta, radius):
    """Convected vortex (Sec. 5a) centred at (xc, yc), with periodic images folded to the nearest."""
    u0 = ma * CS
    eps = beta * u0
    x = torch.arange(nx, dtype=torch.float64, device="cuda") - xc
    y = torch.arange(ny, dtype=torch.float64, device="cuda") - yc
    x = ((x + 0.5 * nx) % nx - 0.5 * nx)[None, :] / radius
    y = ((y + 0.5 * ny) % ny - 0.5 * ny)[:, None] / radius
    bell = torch.exp(-0.5 * x * x) * torch.exp(-0.5 * y * y)
    rho = 1.0 - (eps * eps / (2.0 * CS * CS)) * bell * bell
    ux = u0 - eps * y * bell
    uy = eps * x * bell
    return [rho.contiguous(), ux.contiguous(), uy.contiguous()]


def _seeded_vortex(case, seed):
    g = _rng(seed)
    nx, ny = case["nx"], case["ny"]
    return _vortex(nx, ny, case["ma"], g.uniform(0, nx), g.uniform(0, ny), g.uniform(0.4, 0.6), 0.1 * min(nx, ny))


def _shear_layer(n, ma, phase, delta):
    """Periodic double shear layer (App. C) of width n / 80, its transverse wave at `phase`."""
    u0, kappa = ma * CS, 80.0 / n
    y = torch.arange(n, dtype=torch.float64, device="cuda")[:, None]
    x = torch.arange(n, dtype=torch.float64, device="cuda")[None, :]
    prof = torch.where(y <= 0.5 * n, torch.tanh(kappa * (y - 0.25 * n)), torch.tanh(kappa * (0.75 * n - y)))
    ux = (u0 * prof).expand(n, n).contiguous()
    uy = (delta * u0 * torch.sin(2.0 * math.pi * (x / n + phase))).expand(n, n).contiguous()
    return [torch.ones_like(ux), ux, uy]


def _group_models(case):
    return MODELS if case["models"] == "all" else tuple(case["models"].split(","))


def _model_preset(model):
    return "srt" if model in ("bgk", "rr") else "reg"


def _shear_seed(case, seed):
    g = _rng(seed)
    return _shear_layer(case["n"], case["ma"], g.uniform(0, 1), g.uniform(0.04, 0.06))


def _sweep_instances(case, seed):
    """Sizes (the study's, whatever the seed), models, rates and vortices of a stability study,
    and its concatenated fields."""
    g, sizes = _rng(seed), _rng(4).integers(32, 257, (case["instances"], 2))
    descs, fields = [], []
    for k in range(case["instances"]):
        nx, ny = (int(v) for v in sizes[k])
        model = MODELS[k % len(MODELS)]
        preset = "srt" if (k // len(MODELS)) % 2 == 0 else "reg"
        ma, nu = float(g.uniform(0.05, 0.3)), float(np.exp(g.uniform(np.log(1e-2), np.log(1e-1))))
        descs.append(dict(nx=nx, ny=ny, model=model, rates=_rates(nu, preset), ux_ref=ma * CS, uy_ref=0.0))
        fields.append([float(v) for v in (nx, ny, ma, g.uniform(0, nx), g.uniform(0, ny), 0.5, 0.1 * min(nx, ny))])
    # all instances' vortices at once, node by node
    p = torch.tensor(fields, dtype=torch.float64, device="cuda")
    count = torch.tensor([d["nx"] * d["ny"] for d in descs], device="cuda")
    node = torch.repeat_interleave(torch.arange(len(descs), device="cuda"), count)
    local = torch.arange(node.numel(), device="cuda") - (torch.cumsum(count, 0) - count)[node]
    nx, ny, ma, xc, yc, beta, r = (p[:, k][node] for k in range(7))
    x, y = local.double() % nx, torch.div(local, nx.long(), rounding_mode="floor").double()
    x = ((x - xc + 0.5 * nx) % nx - 0.5 * nx) / r
    y = ((y - yc + 0.5 * ny) % ny - 0.5 * ny) / r
    u0 = ma * CS
    eps = beta * u0
    bell = torch.exp(-0.5 * (x * x + y * y))
    return descs, [1.0 - eps * eps / (2.0 * CS * CS) * bell * bell, u0 - eps * y * bell, eps * x * bell]


def _adjoint_inputs(case, seed):
    g = _rng(seed)
    nx, ny = case["nx"], case["ny"]
    u0, xc, yc = case["ma"] * CS, g.uniform(0, nx), g.uniform(0, ny)
    radius = 0.1 * min(nx, ny)
    start = _vortex(nx, ny, case["ma"], xc, yc, 0.5, radius)
    # the target: a stronger vortex that the mean flow carried along, seen with measurement noise
    _, tx, ty = _vortex(nx, ny, case["ma"], xc + u0 * case["steps"], yc, 0.7, radius)
    noise = torch.from_numpy(g.normal(0.0, 1e-2 * u0, size=(2, ny, nx))).cuda()
    return start, [tx + noise[0], ty + noise[1]]


def _growth_inputs(case, seed):
    g = _rng(seed)
    ang = g.uniform(0.0, 0.25 * math.pi, case["flows"])
    mach = g.uniform(0.05, 0.5, case["flows"])
    flows = np.stack([np.ones(case["flows"]), mach * CS * np.cos(ang), mach * CS * np.sin(ang)], 1)
    k = math.pi * (np.arange(case["nk"]) + g.uniform(0.2, 0.8)) / case["nk"]
    kx, ky = np.meshgrid(k, k, indexing="ij")
    return torch.from_numpy(flows).cuda(), torch.from_numpy(np.stack([kx.ravel(), ky.ravel()], 1)).cuda()


class _Group:
    def __init__(self, lattices):
        self.lattices = lattices
        self.handle = lbm.lbm_group_create([x.ctx for x in lattices], graph_steps=GRAPH_STEPS)

    def __del__(self):
        lbm.lbm_group_destroy(self.handle)


class _Batch:
    def __init__(self, descs, storage):
        self.handle = lbm.lbm_batch_create(descs, storage=storage)

    def __del__(self):
        lbm.lbm_batch_destroy(self.handle)


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind in ("lattice", "restart"):
        nx, ny = case["nx"], case["ny"]
        lat = lbm.Lattice(nx, ny, case["model"], _rates(case["nu"], case["preset"]), storage=lbm.STORAGES[case["storage"]])
        s["lattice"] = lat
        s["fields"] = _seeded_vortex(case, seed)
        if kind == "restart":
            # the checkpoint in hand: a state a few steps into a run
            s["checkpoint"] = torch.empty((9, ny, nx), dtype=torch.float64, device="cuda")
            lat.init_equilibrium(*s.pop("fields"))
            lat.step(8)
            lat.get_populations(s["checkpoint"])
            s["next"] = torch.empty_like(s["checkpoint"])
            s["sums"] = torch.empty(8, dtype=torch.float64, device="cuda")
        else:
            if case["shift"]:
                lat.set_shift_velocity(case["ma"] * CS, 0.0)
            if case["check"]:
                lat.set_check(case["check"], uref=(case["ma"] * CS, 0.0))
            s["out"] = [torch.empty((ny, nx), dtype=torch.float64, device="cuda") for _ in range(3)]
    elif kind == "group":
        n = case["n"]
        lattices = []
        for m in _group_models(case):
            lat = lbm.Lattice(n, n, m, _rates(case["nu"], _model_preset(m)), storage=lbm.STORAGES[case["storage"]])
            lat.set_check(GROUP_CHECK)
            lattices.append(lat)
        s["group"] = _Group(lattices)
        s["fields"] = _shear_seed(case, seed)
        s["out"] = [torch.empty((3, n, n), dtype=torch.float64, device="cuda") for _ in lattices]
    elif kind == "sweep":
        descs, s["fields"] = _sweep_instances(case, seed)
        s["sizes"] = [(d["nx"], d["ny"]) for d in descs]
        s["batch"] = _Batch(descs, lbm.STORAGES[case["storage"]])
        s["out"] = torch.empty(9 * sum(x * y for x, y in s["sizes"]), dtype=torch.float64, device="cuda")
    elif kind == "adjoint":
        s["start"], s["target"] = _adjoint_inputs(case, seed)
        s["rates"] = torch.tensor(_rates(case["nu"], "reg"), dtype=torch.float64)
    else:
        s["flows"], s["k"] = _growth_inputs(case, seed)
        n = s["flows"].shape[0], s["k"].shape[0]
        s["growth"] = torch.empty(n, dtype=torch.float64, device="cuda")
    return s


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "lattice":
        lat = state["lattice"]
        lat.init_equilibrium(*state["fields"])
        lat.step(case["steps"])
        lat.moments(*state["out"])
        out = {k: v.to(FIELD_TYPE[case["storage"]]) for k, v in zip(("rho", "ux", "uy"), state["out"])}
        if case["check"]:
            out["status"] = lat.status()
        return out
    if kind == "restart":
        lat = state["lattice"]
        lat.set_populations(state["checkpoint"])
        lat.step(case["steps"])
        lat.reduce(state["sums"])
        lat.get_populations(state["next"])
        return {"sums": state["sums"].to(FIELD_TYPE[case["storage"]]),
                "populations": state["next"].to(FIELD_TYPE[case["storage"]])}
    if kind == "group":
        lattices = state["group"].lattices
        for lat in lattices:
            lat.init_equilibrium(*state["fields"])
        lbm.lbm_group_step(state["group"].handle, case["steps"])
        for lat, out in zip(lattices, state["out"]):
            lat.moments(out[0], out[1], out[2])
        return {"fields": [v.to(FIELD_TYPE[case["storage"]]) for v in state["out"]],
                "status": [lat.status() for lat in lattices]}
    if kind == "sweep":
        b = state["batch"].handle
        lbm.lbm_batch_init_equilibrium(b, *state["fields"])
        lbm.lbm_batch_run(b, case["steps"], check_every=SWEEP_CHECK)
        status, blowup, steps, diag = lbm.lbm_batch_status(b, len(state["sizes"]))
        at = 0
        for i, (nx, ny) in enumerate(state["sizes"]):
            lbm.lbm_batch_get_populations(b, i, state["out"][at:at + 9 * nx * ny])
            at += 9 * nx * ny
        return {"status": status, "blowup": blowup, "steps": steps, "diag": diag.astype(np.float32),
                "populations": state["out"].float()}
    if kind == "adjoint":
        rho, ux, uy = state["start"]
        ux, uy = ux.detach().requires_grad_(), uy.detach().requires_grad_()
        rates = state["rates"].detach().requires_grad_()
        loss = LBMRun.apply(ux, uy, rates, rho, case["steps"], lbm.MODELS[case["model"]],
                            lbm.STORAGES[case["storage"]], 0, *state["target"])
        loss.backward()
        t = FIELD_TYPE[case["storage"]]
        return {"loss": loss.detach().to(t), "ux": ux.grad.to(t), "uy": uy.grad.to(t), "rates": rates.grad.to(t)}
    lbm.lbm_lsa_growth(case["model"], _rates(case["nu"], case["preset"]), state["flows"], state["k"], state["growth"])
    return {"growth": state["growth"]}


def work(case):
    """Inputs read once, outputs written once, and the collision arithmetic of every update (a
    state that stays on the chip needs no memory traffic of its own)."""
    kind = case["kind"]
    if kind == "lattice":
        n = case["nx"] * case["ny"]
        return {"bytes": 48.0 * n, "flops": float(n) * case["steps"] * UPDATE_FLOPS[case["model"]]}
    if kind == "restart":
        n = case["nx"] * case["ny"]
        return {"bytes": 144.0 * n, "flops": float(n) * case["steps"] * UPDATE_FLOPS[case["model"]]}
    if kind == "group":
        n, models = case["n"] ** 2, _group_models(case)
        return {"bytes": 24.0 * n * (1 + len(models)),
                "flops": float(n) * case["steps"] * sum(UPDATE_FLOPS[m] for m in models)}
    if kind == "sweep":
        # sizes average 144^2 nodes; every model takes part equally
        n = case["instances"] * 144.0 * 144.0
        return {"bytes": (24.0 + 72.0) * n, "flops": n * case["steps"] * sum(UPDATE_FLOPS.values()) / len(UPDATE_FLOPS)}
    if kind == "adjoint":
        # one forward run and a transposed update of about twice its arithmetic per step
        n = case["nx"] * case["ny"]
        return {"bytes": 56.0 * n, "flops": 3.0 * n * case["steps"] * UPDATE_FLOPS[case["model"]]}
    # Hessenberg reduction and QR eigenvalues of a 9 x 9 complex matrix: about (10/3 + 20/3) n^3
    # complex multiply-adds of 8 operations
    n = case["flows"] * float(case["nk"]) ** 2
    return {"bytes": 8.0 * n + 16.0 * case["nk"] ** 2, "flops": n * 8 * 10.0 * 9 ** 3}


# ---- the same results in plain FP64 torch ---------------------------------------------------
EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)


def _factor(s, u):
    """One-dimensional factor of the extended equilibrium for velocity component s."""
    return 2.0 / 3.0 - u * u if s == 0 else 0.5 * (u * u + s * u + 1.0 / 3.0)


def _equilibrium(rho, ux, uy):
    px, py = {s: _factor(s, ux) for s in (0, 1, -1)}, {s: _factor(s, uy) for s in (0, 1, -1)}
    return [rho * px[EX[i]] * py[EY[i]] for i in range(9)]


def _macro(f):
    rho = f[0] + f[1] + f[2] + f[3] + f[4] + f[5] + f[6] + f[7] + f[8]
    ux = (f[1] - f[3] + f[5] - f[6] - f[7] + f[8]) / rho
    uy = (f[2] - f[4] + f[5] + f[6] - f[7] - f[8]) / rho
    return rho, ux, uy


def _collide(f, model, w, w3, w4):
    """Post-collision populations of App. B's models from the pre-collision ones."""
    rho, ux, uy = _macro(f)
    eq = _equilibrium(rho, ux, uy)
    n = [a - b for a, b in zip(f, eq)]
    if model == "bgk":
        return [a - w * b for a, b in zip(f, n)]
    cs2 = 1.0 / 3.0
    # moments of the non-equilibrium part (orders 0 and 1 vanish)
    diag = n[5] + n[6] + n[7] + n[8]
    m20, m02, m11 = n[1] + n[3] + diag, n[2] + n[4] + diag, n[5] - n[6] + n[7] - n[8]
    m21, m12, m22 = n[5] + n[6] - n[7] - n[8], n[5] - n[6] - n[7] + n[8], diag
    p20, p02, p11 = (1.0 - w) * m20, (1.0 - w) * m02, (1.0 - w) * m11
    if model == "rm":
        p21, p12, p22 = (1.0 - w3) * m21, (1.0 - w3) * m12, (1.0 - w4) * m22
    elif model in ("hm", "pr", "rr"):
        if model == "rr":
            a21, a12 = 2.0 * ux * m11 + uy * m20, 2.0 * uy * m11 + ux * m02
            a22 = uy * uy * m20 + ux * ux * m02 + 4.0 * ux * uy * m11
        else:
            a21, a12, a22 = m21, m12, m22 - cs2 * (m20 + m02)
        r3, r4 = (0.0, 0.0) if model == "pr" else (1.0 - w3, 1.0 - w4)
        p21, p12, p22 = r3 * a21, r3 * a12, r4 * a22 + cs2 * (p20 + p02)
    else:
        # central moments, shifted by u, relaxed, shifted back
        k21, k12 = m21 - 2.0 * ux * m11 - uy * m20, m12 - 2.0 * uy * m11 - ux * m02
        k22 = m22 - 2.0 * ux * m12 - 2.0 * uy * m21 + ux * ux * m02 + uy * uy * m20 + 4.0 * ux * uy * m11
        q21, q12 = (1.0 - w3) * k21, (1.0 - w3) * k12
        if model == "cm":
            q22 = (1.0 - w4) * k22
        elif model == "chm":
            q22 = (1.0 - w4) * (k22 - cs2 * (m20 + m02)) + cs2 * (p20 + p02)
        else:
            # fourth cumulant of the full central moments, equilibrium part rho c_s^2 removed again
            c22 = k22 - cs2 * (m20 + m02) - (m20 * m02 + 2.0 * m11 * m11) / rho
            q22 = (1.0 - w4) * c22 + cs2 * (p20 + p02) + (p20 * p02 + 2.0 * p11 * p11) / rho
        p21, p12 = q21 + 2.0 * ux * p11 + uy * p20, q12 + 2.0 * uy * p11 + ux * p02
        p22 = q22 + 2.0 * ux * q12 + 2.0 * uy * q21 + ux * ux * p02 + uy * uy * p20 + 4.0 * ux * uy * p11
    back = [p22 - p20 - p02,
            0.5 * (p20 - p12 - p22), 0.5 * (p02 - p21 - p22), 0.5 * (p20 + p12 - p22), 0.5 * (p02 + p21 - p22),
            0.25 * (p22 + p11 + p12 + p21), 0.25 * (p22 - p11 - p12 + p21),
            0.25 * (p22 + p11 - p12 - p21), 0.25 * (p22 - p11 + p12 - p21)]
    return [a + b for a, b in zip(eq, back)]


def _step(f, model, rates):
    return [torch.roll(v, (EY[i], EX[i]), (0, 1)) for i, v in enumerate(_collide(f, model, *rates))]


def _exact_lattice(f, model, rates, steps):
    for _ in range(steps):
        f = _step(f, model, rates)
    return f


def _exact_sweep(case, seed):
    descs, (rho, ux, uy) = _sweep_instances(case, seed)
    n, count = len(descs), torch.tensor([d["nx"] * d["ny"] for d in descs], device="cuda")
    first = torch.cumsum(count, 0) - count
    node = torch.repeat_interleave(torch.arange(n, device="cuda"), count)
    wide = torch.tensor([d["nx"] for d in descs], device="cuda")[node]
    high = torch.tensor([d["ny"] for d in descs], device="cuda")[node]
    local = torch.arange(node.numel(), device="cuda") - first[node]
    x, y = local % wide, torch.div(local, wide, rounding_mode="floor")
    pull = [first[node] + (y - EY[i]) % high * wide + (x - EX[i]) % wide for i in range(9)]
    rates = torch.tensor([d["rates"] for d in descs], dtype=torch.float64, device="cuda")[node]
    kind = torch.tensor([MODELS.index(d["model"]) for d in descs], device="cuda")[node]
    own = [(m, torch.nonzero(kind == k).flatten()) for k, m in enumerate(MODELS) if bool((kind == k).any())]
    own = [(m, idx, [rates[idx, k] for k in range(3)]) for m, idx in own]
    f = _equilibrium(rho, ux, uy)
    ref = torch.tensor([d["ux_ref"] for d in descs], dtype=torch.float64, device="cuda")[node]
    diag = torch.zeros((n, 4), dtype=torch.float64, device="cuda")
    mean = lambda v: torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, node, v) / count
    for t in range(case["steps"]):
        if t % SWEEP_CHECK == 0:
            r, vx, vy = _macro(f)
            diag[:, 0], diag[:, 1] = mean((vx - ref) ** 2 + vy ** 2), mean(vx ** 2 + vy ** 2)
            diag[:, 2] = torch.full((n,), math.inf, dtype=torch.float64, device="cuda").scatter_reduce(0, node, r, "amin")
            if t == 0:
                diag[:, 3] = diag[:, 0]
        g = [torch.empty_like(v) for v in f]
        for m, idx, w in own:
            for v, h in zip(g, _collide([a[idx] for a in f], m, *w)):
                v[idx] = h
        f = [v[pull[i]] for i, v in enumerate(g)]
    blocks = torch.empty(9 * node.numel(), dtype=torch.float64, device="cuda")
    for i, v in enumerate(f):   # instance by instance, [9][ny][nx] each
        blocks[9 * first[node] + i * count[node] + local] = v
    return {"status": None, "blowup": None, "steps": None, "diag": diag, "populations": blocks}


def _exact_adjoint(case, seed):
    (rho, ux, uy), (tx, ty) = _adjoint_inputs(case, seed)
    ux, uy = ux.requires_grad_(), uy.requires_grad_()
    rates = [torch.tensor(v, dtype=torch.float64, device="cuda", requires_grad=True) for v in _rates(case["nu"], "reg")]

    f = torch.stack(_equilibrium(rho, ux, uy))
    with torch.no_grad():   # a state every few steps, then backwards stretch by stretch
        kept, g, every = [], f.detach(), 20
        for t in range(case["steps"]):
            if t % every == 0:
                kept.append(g)
            g = torch.stack(_step(list(g), case["model"], rates))
    g = g.requires_grad_()
    _, vx, vy = _macro(list(g))
    loss = 0.5 * ((vx - tx) ** 2 + (vy - ty) ** 2).sum()
    lam, = torch.autograd.grad(loss, g)
    grad = [torch.zeros((), dtype=torch.float64, device="cuda") for _ in rates]
    for q in reversed(range(len(kept))):
        start = kept[q].detach().requires_grad_()
        h = start
        for _ in range(min(every, case["steps"] - q * every)):
            h = torch.stack(_step(list(h), case["model"], rates))
        got = torch.autograd.grad(h, [start] + rates, lam, allow_unused=True)
        lam = got[0]
        grad = [a if b is None else a + b for a, b in zip(grad, got[1:])]
    gx, gy = torch.autograd.grad(f, [ux, uy], lam)
    return {"loss": loss.detach(), "ux": gx, "uy": gy, "rates": torch.stack(grad)}


def _exact_growth(case, seed):
    flows, k = _growth_inputs(case, seed)
    rates = _rates(case["nu"], case["preset"])
    k = k.cpu().numpy()
    shift = np.exp(-1j * (k[:, 0, None] * np.array(EX) + k[:, 1, None] * np.array(EY)))
    growth = np.empty((flows.shape[0], k.shape[0]))
    for i, (rho, ux, uy) in enumerate(flows.cpu()):
        f = torch.stack(_equilibrium(rho, ux, uy))
        jac = torch.autograd.functional.jacobian(lambda v: torch.stack(_collide(list(v), case["model"], *rates)), f)
        lam = np.linalg.eigvals(shift[:, :, None] * jac.numpy()[None])
        growth[i] = np.log(np.abs(lam)).max(1)
    return {"growth": growth}


def exact(case, seed):
    kind = case["kind"]
    if kind == "sweep":
        return _exact_sweep(case, seed) if case["instances"] * case["steps"] <= 1100000 else None
    if kind == "adjoint":
        return _exact_adjoint(case, seed) if case["steps"] <= 1000 else None
    if kind == "growth":
        return _exact_growth(case, seed)
    with torch.no_grad():
        if kind == "group":
            start = _equilibrium(*_shear_seed(case, seed))
            fields = []
            for m in _group_models(case):
                f = _exact_lattice(start, m, _rates(case["nu"], _model_preset(m)), case["steps"])
                fields.append(torch.stack(_macro(f)))
            return {"fields": fields, "status": None}
        f = _equilibrium(*_seeded_vortex(case, seed))
        # a step costs about 0.6 ns a node here, and 1 ms at least
        if case["steps"] * max(1e-3, 6e-10 * case["nx"] * case["ny"]) > 20.0:
            return None
        rates = _rates(case["nu"], case["preset"])
        if kind == "restart":
            f = _exact_lattice(f, case["model"], rates, 8 + case["steps"])
            rho, ux, uy = _macro(f)
            u2 = ux * ux + uy * uy
            sums = [rho.sum(), (rho * ux).sum(), (rho * uy).sum(), 0.5 * (rho * u2).sum(), u2.mean(), u2.mean(),
                    rho.min(), torch.zeros((), dtype=torch.float64, device="cuda")]
            return {"sums": torch.stack(sums), "populations": torch.stack(f)}
        rho, ux, uy = _macro(_exact_lattice(f, case["model"], rates, case["steps"]))
        return {"rho": rho, "ux": ux, "uy": uy, "status": None}
