"""What the speed of this framework is measured on: passes of its public entry points, from the
smallest column to the full two-phase domain, in each storage precision and wall type.

Kinds of case and the use they stand for:

* ``domain``  - one lattice handle: a kept state is set (the paper's equilibrate-then-change
                protocol), advanced by a block of steps, and its populations and density are read.
* ``thermal`` - the same with the temperature field and the energy equation.
* ``slab``    - the multi-GPU path's step on one slab that is the whole domain (caller-owned
                populations, mass partials handed from step to step).
* ``batch``   - thousands of independent liquid columns: created from their density profiles,
                run for a block of steps, and read; the whole life of a batch.
* ``train``   - the warm-start network's training: minibatch gather, forward, backward, Adam.
* ``predict`` - the network's inference over the rows of many columns.

States are what a run meets: a liquid layer under vapour at the coexistence densities of its
temperature, a slightly wavy interface with noise, and a weak flow. Populations of FP32 runs are
returned as float32 (the library reads them out as doubles), those of FP64 and double-float
runs as float64.
"""
import math

import numpy as np
import torch

from paper_2301_12869_gb300 import lbm

A, B, R, G, SIGMA = 0.25, 4.0, 1.0, -1.0, 1.385
C_V, KAPPA = 5.0, 0.02
CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
WGT = (4 / 9, 1 / 9, 1 / 9, 1 / 9, 1 / 9, 1 / 36, 1 / 36, 1 / 36, 1 / 36)
FLOPS_NODE = 150        # of one isothermal node step (densities, potential, force, collision)
FLOPS_NODE_THERMAL = 230  # with the energy equation's two stages
MLP_ROW_FLOPS = 2 * (6 * 128 + 2 * 128 * 128 + 128)


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the paper's 1-D column on its own: 800 nodes, where a step's latency is all there is
        dict(name="column 4x200 fp64", kind="domain", precision="fp64", nx=4, ny=200, form=1, wall=0,
             Tr=0.85, gy=-2e-5, steps=1000),
        # the benchmark's two-phase domain with the gravity form that needs the mean density
        dict(name="domain 1024x4096 fp32", kind="domain", precision="fp32", nx=1024, ny=4096, form=2, wall=0,
             Tr=0.80, gy=-1e-4, steps=100),
        # the same domain in the precision that comparisons are made against
        dict(name="domain 1024x4096 fp64", kind="domain", precision="fp64", nx=1024, ny=4096, form=2, wall=0,
             Tr=0.80, gy=-1e-4, steps=10),
        # a size that no tile divides, plain gravity
        dict(name="domain 772x1003 fp32", kind="domain", precision="fp32", nx=772, ny=1003, form=1, wall=0,
             Tr=0.82, gy=-2e-5, steps=150),
        # the paper's own walls (Zou-He wet nodes) on a mid-sized domain
        dict(name="wet walls 256x768 fp32", kind="domain", precision="fp32", nx=256, ny=768, form=2, wall=1,
             Tr=0.85, gy=-2e-5, steps=200),
        # one step after the other on caller-owned populations, as a rank of the multi-GPU path does
        dict(name="slab 1024x2048 fp32", kind="slab", precision="fp32", nx=1024, ny=2048, form=2, wall=0,
             Tr=0.80, gy=-1e-4, steps=20),
        # the benchmark's heated column with the energy equation
        dict(name="thermal 512x2048 fp32", kind="thermal", precision="fp32", nx=512, ny=2048, form=1, wall=0,
             Tr=0.875, gy=-2e-5, steps=100),
        # the benchmark's 1024 short columns: the FP32 phase of the way to a steady state
        dict(name="batch 1024 cols fp32", kind="batch", precision="fp32", cols=1024, heights="64,128", wall=0,
             steps=1500),
        # its finishing phase in double-float arithmetic
        dict(name="batch 1024 cols dd", kind="batch", precision="dd", cols=1024, heights="64,128", wall=0,
             steps=600),
        # the full range of heights in plain FP64
        dict(name="batch 320 cols fp64", kind="batch", precision="fp64", cols=320, heights="64,128,256,512,1024",
             wall=0, steps=150),
        # training of the warm-start network at the benchmark's minibatch
        dict(name="train 8192", kind="train", rows=200000, batch=8192, iters=40),
        # the rows of the columns that one warm start covers (not a multiple of a tile)
        dict(name="predict 157003", kind="predict", rows=157003),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["domain", "domain", "domain", "thermal", "slab", "batch", "batch", "batch", "train", "predict"])
    if kind in ("domain", "thermal", "slab"):
        precision = rng.choice(["fp32", "fp32", "fp64"])
        nx = 4 * max(1, int(_log(rng, 4, 1024) / 4))
        ny = int(_log(rng, 24, 4096 if kind == "domain" else 2048))
        form, wall = rng.choice([1, 2]), rng.choice([0, 0, 0, 1])
        if kind == "slab":
            precision = "fp32"
        nodes = nx * ny
        # a block of steps, shorter on large lattices and in FP64
        steps = int(min(600, max(10, (2e8 if precision == "fp32" else 2e7) / nodes)) * rng.uniform(0.5, 1.0)) + 1
        if kind == "slab":
            steps = min(steps, 20)
        return dict(kind=kind, precision=precision, nx=nx, ny=ny, form=form, wall=wall,
                    Tr=round(rng.uniform(0.80, 0.90), 4), gy=-round(min(5e-5, 0.02 / ny) * rng.uniform(0.2, 1.0), 9),
                    steps=steps)
    if kind == "batch":
        precision = rng.choice(["fp32", "fp32", "dd", "fp64"])
        cols = int(_log(rng, 24, 1024))
        hs = sorted({int(_log(rng, 16, 1024)) for _ in range(rng.randint(1, 3))})
        mean = sum(hs) / len(hs)
        budget = {"fp32": 1.2e8, "dd": 5e7, "fp64": 1.6e7}[precision]  # rows x steps
        most = {"fp32": 1500, "dd": 600, "fp64": 400}[precision]
        steps = int(min(most, max(50, budget / (cols * mean))) * rng.uniform(0.5, 1.0))
        return dict(kind=kind, precision=precision, cols=cols, heights=",".join(map(str, hs)),
                    wall=rng.choice([0, 0, 0, 1]), steps=steps)
    if kind == "train":
        batch = 2 * int(_log(rng, 64, 8192))
        return dict(kind=kind, rows=int(_log(rng, 20000, 500000)), batch=batch,
                    iters=int(min(40, 8192 * 40 / batch) * rng.uniform(0.5, 1.0)) + 1)
    return dict(kind=kind, rows=int(_log(rng, 500, 1.2e6)))


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) % (1 << 62))


_COEX = {}


def _coexistence(Tr):
    """rho_v, rho_l at the reduced temperature Tr (a table of the Maxwell rule, interpolated)."""
    if not _COEX:
        _, Tc, _ = lbm.lbm_critical_point(A, B, R)
        t = np.linspace(0.68, 0.97, 59)
        v = np.array([lbm.lbm_coexistence(A, B, R, x * Tc)[:2] for x in t])
        _COEX.update(t=t, v=v, Tc=Tc)
    return np.interp(Tr, _COEX["t"], _COEX["v"][:, 0]), np.interp(Tr, _COEX["t"], _COEX["v"][:, 1])


def _tc():
    _coexistence(0.8)
    return _COEX["Tc"]


def _feq(rho, ux, uy):
    u2 = ux * ux + uy * uy
    f = torch.empty((9,) + tuple(rho.shape), dtype=torch.float64, device=rho.device)
    for i in range(9):
        cu = CX[i] * ux + CY[i] * uy
        f[i] = WGT[i] * rho * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * u2)
    return f


def _field(case, seed):
    """Density and populations of a liquid layer below vapour: a wavy interface with noise and a
    weak smooth flow."""
    g = _gen(seed)
    nx, ny = case["nx"], case["ny"]
    rv, rl = (float(x) for x in _coexistence(case["Tr"]))
    r = torch.rand(8, generator=g, device="cuda", dtype=torch.float64)
    x = torch.arange(nx, device="cuda", dtype=torch.float64)[None, :]
    y = torch.arange(ny, device="cuda", dtype=torch.float64)[:, None]
    y0 = (0.4 + 0.2 * r[0]) * ny + min(2.0, ny / 32.0) * torch.sin(2 * math.pi * (x / nx + r[1]))
    rho = 0.5 * (rl + rv) - 0.5 * (rl - rv) * torch.tanh(2.0 * (y - y0) / 5.0)
    noise = 1e-3 * (2.0 * torch.rand((ny, nx), generator=g, device="cuda", dtype=torch.float64) - 1.0)
    rho = rho + torch.where((y - y0).abs() <= 10.0, noise * (rho / rl), torch.zeros_like(rho))
    kx, ky = 2 * math.pi / nx, math.pi / ny
    ux = 2e-3 * (0.5 + r[2]) * torch.cos(kx * x + 6.3 * r[3]) * torch.sin(ky * (y + 0.5))
    uy = 2e-3 * (0.5 + r[4]) * torch.sin(kx * x + 6.3 * r[5]) * torch.sin(ky * (y + 0.5))
    return rho.contiguous(), _feq(rho, ux, uy)


def _temperatures(case):
    Tc = _tc()
    return (case["Tr"] + 0.03) * Tc, (case["Tr"] - 0.03) * Tc


def _temperature_field(case, seed):
    """The conduction profile with small smooth variations."""
    g = _gen(seed + 7919)
    nx, ny = case["nx"], case["ny"]
    Tb, Tt = _temperatures(case)
    x = torch.arange(nx, device="cuda", dtype=torch.float64)[None, :]
    y = torch.arange(ny, device="cuda", dtype=torch.float64)[:, None]
    if case["wall"]:
        T = Tb + (Tt - Tb) * y / (ny - 1)
        s = torch.sin(math.pi * y / (ny - 1))
    else:
        T = Tb + (Tt - Tb) * (y + 0.5) / ny
        s = torch.sin(math.pi * (y + 0.5) / ny)
    r = torch.rand(2, generator=g, device="cuda", dtype=torch.float64)
    return (T + 5e-3 * Tb * (r[0] - 0.5) * s * torch.cos(2 * math.pi * (x / nx + r[1]))).contiguous()


def _columns(case, seed):
    """Column descriptors (host) and their concatenated initial densities (device)."""
    g = np.random.default_rng(int(seed) % (1 << 63))
    hs = [int(h) for h in case["heights"].split(",")]
    n, Tc = case["cols"], _tc()
    ny = np.array(hs)[np.arange(n) % len(hs)]
    Tr = g.uniform(0.75, 0.95, n)
    gy = -np.exp(g.uniform(np.log(1e-6), np.log(np.minimum(1e-4, 2.5e-3 / ny))))
    form = g.integers(1, 3, n)
    frac = g.uniform(0.35, 0.65, n)
    rv, rl = _coexistence(Tr)
    cols = [dict(ny=int(ny[c]), T=float(Tr[c] * Tc), gx=0.0, gy=float(gy[c]), form=int(form[c])) for c in range(n)]
    rho = np.concatenate([
        np.repeat(0.5 * (rl[c] + rv[c])
                  - 0.5 * (rl[c] - rv[c]) * np.tanh(2.0 * (np.arange(ny[c]) - frac[c] * ny[c]) / 5.0), 4)
        for c in range(n)])
    return cols, torch.from_numpy(rho).cuda()


def _features(rows, seed):
    """Column descriptors as the network meets them, and a smooth density target."""
    g = _gen(seed)
    u = torch.rand((rows, 6), generator=g, device="cuda", dtype=torch.float64)
    x = torch.stack([0.70 + 0.25 * u[:, 0], -6.0 + 2.0 * u[:, 1], 1.0 + torch.round(u[:, 2]), 0.6 + 1.2 * u[:, 3],
                     u[:, 4], 6.0 + torch.round(u[:, 5])], dim=1)
    front = (x[:, 3] - 0.3) / 1.8
    t = 1.3 - 1.1 * torch.tanh((x[:, 4] - front) * torch.exp2(x[:, 5]) / 8.0) * (1.6 - x[:, 0])
    return x.float().contiguous(), t.float().contiguous()


def _network(seed):
    """Packed parameters with weights of the usual initial scale and small biases."""
    g = np.random.default_rng(int(seed) % (1 << 63))
    fan = {"W1": (6, 128), "W2": (128, 128), "W3": (128, 128), "w4": (128, 1)}
    P = {k: g.uniform(-1, 1, (128,) if k == "w4" else (b, a)) * math.sqrt(6.0 / (a + b)) for k, (a, b) in fan.items()}
    P.update(b1=0.1 * g.standard_normal(128), b2=0.1 * g.standard_normal(128), b3=0.1 * g.standard_normal(128),
             b4=np.array([0.5]))
    return lbm.mlp_pack(P)


# ------------------------------------------------------------------ prepare and run
class _Owned:
    """A network handle that is released with its state."""

    def __init__(self, h):
        self.h = h

    def __del__(self):
        lbm.lbm_mlp_destroy(self.h)


def _params(case, **kw):
    return lbm.make_params(case["nx"], case["ny"], case["Tr"] * _tc(), case["precision"], a=A, b=B, R=R,
                           form=case["form"], g=(0.0, case["gy"]), wall=case["wall"], **kw)


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind in ("domain", "thermal"):
        rho0, s["f0"] = _field(case, seed)
        kw = {}
        if kind == "thermal":
            Tb, Tt = _temperatures(case)
            kw = dict(thermal=1, T_bot=Tb, T_top=Tt, c_v=C_V, kappa=KAPPA)
            s["T0"] = _temperature_field(case, seed)
        s["lat"] = lbm.Lattice(_params(case, **kw), rho0)
        s["f"] = torch.empty_like(s["f0"])
    elif kind == "slab":
        rho0, f0 = _field(case, seed)
        ny, nx = rho0.shape
        p = _params(case, rho_ref=float(rho0.mean()))
        slab = lbm.make_slab(0, ny)
        n = lbm.lbm_slab_partials(p, slab)
        buf = [torch.zeros((9, ny + 2 * lbm.LBM_SLAB_HALO, nx), dtype=torch.float32, device="cuda") for _ in range(3)]
        buf[0][:, 2:-2] = (f0 - p.rho_ref * _weights(f0)).float()
        s.update(p=p, slab=slab, buf=buf, part=[torch.zeros(n, dtype=torch.float64, device="cuda") for _ in range(2)],
                 status=torch.zeros(1, dtype=torch.int32, device="cuda"))
    elif kind == "batch":
        s["cols"], s["rho0"] = _columns(case, seed)
        s["p"] = lbm.make_params(4, 8, 0.8 * _tc(), case["precision"], a=A, b=B, R=R, wall=case["wall"])
        s["stream"] = torch.cuda.Stream()  # a batch captures a graph: not on the legacy default stream
        s["stream"].wait_stream(torch.cuda.current_stream())
    else:
        s["x"], s["t"] = _features(case["rows"], seed)
        s["P"] = _network(seed)
        cap = 128 * (-(-case.get("batch", 128) // 128))
        s["net"] = _Owned(lbm.lbm_mlp_create(s["P"], cap))
        s["seed"] = int(seed) & 0xFFFFFFFF
        s["y"] = torch.empty(case["rows"], dtype=torch.float32, device="cuda")
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind in ("domain", "thermal"):
        lat, f = s["lat"], s["f"]
        lbm.lbm_set_state(lat.h, s["f0"])
        if kind == "thermal":
            lbm.lbm_set_temperature(lat.h, s["T0"])
        lat.step(case["steps"])
        lbm.lbm_get_state(lat.h, f)
        rho = torch.empty(f.shape[1:], dtype=torch.float64, device=f.device)
        lbm.lbm_moments(lat.h, rho)
        out = [f, rho] if kind == "domain" else [f, rho, lat.temperature()]
        return [v.float() for v in out] if case["precision"] == "fp32" else out
    if kind == "slab":
        a, (p0, p1), buf = s["p"], s["part"], s["buf"]
        lbm.lbm_slab_mass(a, s["slab"], buf[0], p0)
        src, dst, spare = buf
        for k in range(case["steps"]):
            lbm.lbm_slab_step(a, s["slab"], src, dst, p0, p1, s["status"])
            src, dst = dst, (spare if k == 0 else src)
            p0, p1 = p1, p0
        return [src]
    if kind == "batch":
        with torch.cuda.stream(s["stream"]):
            b = lbm.lbm_batch_init(s["p"], s["cols"], s["rho0"], s["stream"].cuda_stream)
            lbm.lbm_batch_run(b, 0.0, case["steps"], 100)
            steps, _, _ = lbm.lbm_batch_results(b, case["cols"])
            n = s["rho0"].numel()
            f = torch.empty(9 * n, dtype=torch.float64, device="cuda")
            rho = torch.empty(n, dtype=torch.float64, device="cuda")
            lbm.lbm_batch_get_state(b, f)
            lbm.lbm_batch_moments(b, rho)
            lbm.lbm_batch_destroy(b)
            if case["precision"] == "fp32":
                f, rho = f.float(), rho.float()
        return [f, rho, steps]
    if kind == "train":
        lbm.lbm_mlp_set_params(s["net"].h, s["P"])
        lbm.lbm_mlp_train(s["net"].h, s["x"], s["t"], case["batch"], case["iters"], 3e-4, s["seed"], record=False)
        return [lbm.lbm_mlp_get_params(s["net"].h)]
    lbm.lbm_mlp_predict(s["net"].h, s["x"], s["y"])
    return [s["y"]]


def work(case):
    kind = case["kind"]
    real = 4 if case.get("precision") == "fp32" else 8
    if kind in ("domain", "thermal"):
        n = case["nx"] * case["ny"]
        th = kind == "thermal"
        return dict(bytes=n * ((9 + th) * 8 + (10 + th) * real),
                    flops=case["steps"] * n * (FLOPS_NODE_THERMAL if th else FLOPS_NODE))
    if kind == "slab":  # every step's populations are the caller's: read and written
        n = case["nx"] * case["ny"]
        return dict(bytes=case["steps"] * n * 72, flops=case["steps"] * n * FLOPS_NODE)
    if kind == "batch":
        hs = [int(h) for h in case["heights"].split(",")]
        n = sum(4 * hs[c % len(hs)] for c in range(case["cols"]))
        return dict(bytes=n * (8 + 10 * real), flops=case["steps"] * n * FLOPS_NODE)
    if kind == "train":
        rows = case["batch"] * case["iters"]
        return dict(bytes=rows * 28 + 2 * 4 * lbm.MLP_NPARAMS, flops=3 * rows * MLP_ROW_FLOPS)
    return dict(bytes=case["rows"] * 28 + 4 * lbm.MLP_NPARAMS, flops=case["rows"] * MLP_ROW_FLOPS)


# ------------------------------------------------------------------ the same in plain 64 bits
def _weights(f):
    return torch.tensor(WGT, dtype=torch.float64, device=f.device).view((9,) + (1,) * (f.dim() - 1))


def _pulled(f, wall, gy, form, mean):
    """Streamed populations, x periodic, walls at the ends of the second-to-last axis."""
    q = torch.empty_like(f)
    for i in range(9):
        s = torch.roll(f[i], CX[i], dims=-1)
        if CY[i] == 0:
            q[i] = s
        elif CY[i] == 1:
            q[i][..., 1:, :] = s[..., :-1, :]
            q[i][..., 0, :] = f[OPP[i]][..., 0, :]
        else:
            q[i][..., :-1, :] = s[..., 1:, :]
            q[i][..., -1, :] = f[OPP[i]][..., -1, :]
    if wall:
        for row, sg in ((0, 1.0), (-1, -1.0)):
            w = [q[i][..., row, :] for i in range(9)]
            up, dn = ((2, 5, 6), (4, 7, 8)) if sg > 0 else ((4, 7, 8), (2, 5, 6))
            K = w[0] + w[1] + w[3] + 2.0 * (w[dn[0]] + w[dn[1]] + w[dn[2]])
            g2, m2 = gy.squeeze(-1), mean.squeeze(-1)
            rho = torch.where(form.squeeze(-1) == 1, K, K + sg * 0.5 * m2 * g2) / (1.0 + sg * 0.5 * g2)
            Fy = torch.where(form.squeeze(-1) == 1, rho, rho - m2) * g2
            d = 0.5 * (w[1] - w[3])
            new = (w[4], w[7] - d - 0.25 * Fy, w[8] + d - 0.25 * Fy) if sg > 0 else \
                  (w[2], w[5] + d + 0.25 * Fy, w[6] - d + 0.25 * Fy)
            for i, v in zip(up, new):
                q[i][..., row, :] = v
    return q


def _macro(f, T, gy, form, wall):
    """Streamed populations, rho, the potential's stencil sum, force and velocity."""
    mean = f.sum(dim=0).mean(dim=(-2, -1), keepdim=True)
    q = _pulled(f, wall, gy, form, mean)
    rho = q.sum(dim=0)
    e = B * rho / 4.0
    p = rho * R * T * (1.0 + e + e * e - e ** 3) / (1.0 - e) ** 3 - A * rho * rho
    psi = torch.sqrt(torch.clamp(2.0 * (p - rho / 3.0) / G, min=0.0))
    W_, E_ = torch.roll(psi, 1, dims=-1), torch.roll(psi, -1, dims=-1)
    Sx, Sy = torch.zeros_like(psi), torch.zeros_like(psi)
    dx, ax = E_ - W_, E_ + W_
    Sx[..., 1:-1, :] = dx[..., 1:-1, :] / 3.0 + (dx[..., 2:, :] + dx[..., :-2, :]) / 12.0
    Sy[..., 1:-1, :] = (psi[..., 2:, :] - psi[..., :-2, :]) / 3.0 + (ax[..., 2:, :] - ax[..., :-2, :]) / 12.0
    Fx = -G * psi * Sx
    Fy = -G * psi * Sy + torch.where(form == 1, rho, rho - mean) * gy
    ux = ((q[1] - q[3] + q[5] - q[6] - q[7] + q[8]) + 0.5 * Fx) / rho
    uy = ((q[2] - q[4] + q[5] + q[6] - q[7] - q[8]) + 0.5 * Fy) / rho
    return q, rho, (Sx, Sy), (Fx, Fy), (ux, uy)


_M = np.array([[1, 1, 1, 1, 1, 1, 1, 1, 1], [-4, -1, -1, -1, -1, 2, 2, 2, 2], [4, -2, -2, -2, -2, 1, 1, 1, 1],
               [0, 1, 0, -1, 0, 1, -1, -1, 1], [0, -2, 0, 2, 0, 1, -1, -1, 1], [0, 0, 1, 0, -1, 1, 1, -1, -1],
               [0, 0, -2, 0, 2, 1, 1, -1, -1], [0, 1, -1, 1, -1, 0, 0, 0, 0], [0, 0, 0, 0, 0, 1, -1, 1, -1]], float)


def _step(f, T, gy, form, wall):
    """One step with every relaxation time 1: m* = m_eq + S/2."""
    _, rho, (Sx, Sy), (Fx, Fy), (ux, uy) = _macro(f, T, gy, form, wall)
    jx, jy, u2 = rho * ux, rho * uy, ux * ux + uy * uy
    uF, s = ux * Fx + uy * Fy, SIGMA / 0.5 * G * G * (Sx * Sx + Sy * Sy)
    m = torch.stack([rho, -2 * rho + 3 * rho * u2 + 3 * uF + 0.5 * s, rho - 3 * rho * u2 - 3 * uF - 0.5 * s,
                     jx + 0.5 * Fx, -jx - 0.5 * Fx, jy + 0.5 * Fy, -jy - 0.5 * Fy,
                     rho * (ux * ux - uy * uy) + ux * Fx - uy * Fy, rho * ux * uy + 0.5 * (ux * Fy + uy * Fx)])
    Mi = torch.from_numpy(np.linalg.inv(_M)).to(f.device)
    return (Mi @ m.reshape(9, -1)).reshape(f.shape), rho, ux, uy


def _rate(T, rho, ux, uy, wall, Tb, Tt):
    def pad(v, lo, hi):
        return torch.cat([lo(v[:1]), v, hi(v[-1:])])

    if wall:
        Tp = pad(T, lambda r: r, lambda r: r)
    else:
        Tp = pad(T, lambda r: 2 * Tb - r, lambda r: 2 * Tt - r)
    uxp, uyp = (pad(v, lambda r: -r, lambda r: -r) for v in (ux, uy))
    ny = T.shape[0]

    def nb(v, i):
        return torch.roll(v[1 + CY[i]:1 + CY[i] + ny], -CX[i], dims=1)

    gx = 3 * sum(WGT[i] * CX[i] * nb(Tp, i) for i in range(9))
    gy = 3 * sum(WGT[i] * CY[i] * nb(Tp, i) for i in range(9))
    lap = 6 * sum(WGT[i] * (nb(Tp, i) - T) for i in range(9))
    div = 3 * sum(WGT[i] * (CX[i] * nb(uxp, i) + CY[i] * nb(uyp, i)) for i in range(9))
    e = B * rho / 4.0
    z = (1 + e + e * e - e ** 3) / (1 - e) ** 3
    k = -(ux * gx + uy * gy) + KAPPA / (rho * C_V) * lap - T * R * z / C_V * div
    if wall:
        k[0] = 0
        k[-1] = 0
    return k


def _rounded(f, case, rho_ref):
    """A float32 run's populations as it holds them."""
    w = rho_ref * _weights(f)
    return (f - w).float().double() + w if case["precision"] == "fp32" else f


def _exact_lattice(case, seed):
    rho0, f = _field(case, seed)
    ref = float(rho0.mean())
    f = _rounded(f, case, ref)
    dev = f.device
    form, gy = (torch.full((1, 1), float(v), dtype=torch.float64, device=dev) for v in (case["form"], case["gy"]))
    wall, T = case["wall"], case["Tr"] * _tc()
    if case["kind"] == "thermal":
        Tb, Tt = _temperatures(case)
        T = _temperature_field(case, seed)
        T = T.float().double() if case["precision"] == "fp32" else T
    for _ in range(case["steps"]):
        f, rho, ux, uy = _step(f, T, gy, form, wall)
        if case["kind"] == "thermal":
            k1 = _rate(T, rho, ux, uy, wall, Tb, Tt)
            k2 = _rate(T + k1, rho, ux, uy, wall, Tb, Tt)
            T = T + 0.5 * (k1 + k2)
            if wall:
                T[0], T[-1] = Tb, Tt
    if case["kind"] == "slab":
        return [torch.nn.functional.pad(f - ref * _weights(f), (0, 0, 2, 2))]
    rho = _macro(f, T, gy, form, wall)[1]
    return [f, rho] if case["kind"] == "domain" else [f, rho, T]


def _exact_batch(case, seed):
    cols, rho0 = _columns(case, seed)
    ny = np.array([c["ny"] for c in cols])
    off = np.concatenate([[0], np.cumsum(4 * ny)])
    F = torch.empty(9 * int(off[-1]), dtype=torch.float64, device="cuda")
    D = torch.empty(int(off[-1]), dtype=torch.float64, device="cuda")
    for h in np.unique(ny):
        ids = np.flatnonzero(ny == h)
        at = torch.from_numpy(off[ids][:, None] + np.arange(4 * h)[None, :]).cuda()
        rho = rho0[at].view(len(ids), h, 4)
        z = torch.zeros_like(rho)
        f = _feq(rho, z, z)
        f = _rounded(f, case, rho.mean(dim=(1, 2), keepdim=True))

        def per(key):
            return torch.tensor([float(cols[c][key]) for c in ids], dtype=torch.float64, device="cuda").view(-1, 1, 1)

        T, gy, form = per("T"), per("gy"), per("form")
        for _ in range(case["steps"]):
            f = _step(f, T, gy, form, case["wall"])[0]
        D[at] = _macro(f, T, gy, form, case["wall"])[1].reshape(len(ids), -1)
        at9 = torch.from_numpy(9 * off[ids][:, None] + np.arange(36 * h)[None, :]).cuda()
        F[at9] = f.permute(1, 0, 2, 3).reshape(len(ids), -1)
    return [F, D, None]


def _unpack(packed):
    P, o = {}, 0
    for name, shape in (("W1", (128, 16)), ("b1", (128,)), ("W2", (128, 128)), ("b2", (128,)), ("W3", (128, 128)),
                        ("b3", (128,)), ("w4", (128,)), ("b4", (1,))):
        n = int(np.prod(shape))
        P[name] = torch.from_numpy(np.asarray(packed[o:o + n], dtype=np.float64).reshape(shape)).cuda()
        o += n
    return P


def _forward(P, x):
    c = torch.tensor([0.825, -5.0, 1.5, 1.4, 0.5, 8.0], dtype=torch.float64, device=x.device)
    d = torch.tensor([0.125, 1.0, 0.5, 1.1, 0.5, 2.0], dtype=torch.float64, device=x.device)
    h = torch.nn.functional.pad((x.double() - c) / d, (0, 10))
    for k in "123":
        h = torch.nn.functional.silu(h @ P["W" + k].T + P["b" + k])
    return h @ P["w4"] + P["b4"]


def _minibatch(rows, batch, step, seed):
    """SplitMix64(seed; step * batch + i) mod rows."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + (np.uint64(step * batch) + np.arange(1, batch + 1, dtype=np.uint64)) * np.uint64(
            0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return torch.from_numpy((z % np.uint64(rows)).astype(np.int64)).cuda()


def _exact_train(case, seed):
    x, t = _features(case["rows"], seed)
    P = {k: v.requires_grad_(True) for k, v in _unpack(_network(seed)).items()}
    m = {k: torch.zeros_like(v) for k, v in P.items()}
    v2 = {k: torch.zeros_like(v) for k, v in P.items()}
    for it in range(case["iters"]):
        i = _minibatch(case["rows"], case["batch"], it, int(seed) & 0xFFFFFFFF)
        loss = ((_forward(P, x[i]) - t[i].double()) ** 2).mean()
        grads = torch.autograd.grad(loss, list(P.values()))
        with torch.no_grad():
            for (k, p), g in zip(P.items(), grads):
                m[k] = 0.9 * m[k] + 0.1 * g
                v2[k] = 0.999 * v2[k] + 0.001 * g * g
                p -= 3e-4 * (m[k] / (1 - 0.9 ** (it + 1))) / (torch.sqrt(v2[k] / (1 - 0.999 ** (it + 1))) + 1e-8)
    return [torch.cat([p.detach().reshape(-1) for p in P.values()])]


def exact(case, seed):
    if case["kind"] in ("domain", "thermal", "slab"):
        return _exact_lattice(case, seed)
    if case["kind"] == "batch":
        return _exact_batch(case, seed)
    if case["kind"] == "train":
        return _exact_train(case, seed)
    x, _ = _features(case["rows"], seed)
    P = _unpack(_network(seed))
    return [torch.cat([_forward(P, c) for c in x.split(65536)])]
