"""Performance cases of the framework, through its public Python entry points.

Four kinds of work, with the sizes of this repository's workloads, tests and benchmark:

* "cavity": one cavity from caller fields, a stretch of time steps, then its state, its fields
  and its diagnostics (Cavity.init / step / state_get / fields / diagnostics);
* "sweep":  a batch of uneven cavities stepped together (Batch.step / nusselt, Cavity.fields);
* "net":    the warm-start network, inference (WarmNet.forward) or the loss and its gradient, the
  body of a training step (WarmNet.loss_grad);
* "gemm":   the tensor-core product behind the network's convolutions (gemm_bf16).

exact() restates the model and the network in float64 torch without the library.
"""
import math

import numpy as np
import torch

import workloads
from paper_1511_04552_gb300 import binding as B
from paper_1511_04552_gb300 import warmstart as WS

DEV = "cuda"
STORAGE = {"f32": B.STORE_F32, "f16": B.STORE_F16, "bf16": B.STORE_BF16}
FIELDS = B.UX | B.UY | B.THETA | B.PHI
SWEEP_STEPS = 64
WEIGHTS = "paper_1511_04552_gb300/weights/warmnet_256.npz"


def listed():
    return [
        # the smallest workload (the oracle's 32 x 32 cavity): launches and latency
        _cavity("cavity 32x32", 32, 32, 1e3, 0.01, 20e-9, 200),
        # a small cavity of odd sizes, taller than the tiles divide, with some slip forces off
        _cavity("cavity 130x67 some forces", 130, 67, 3e4, 0.02, 30e-9, 100,
                mask=B.F_ALL & ~(B.F_SAFFMAN | B.F_MAGNUS)),
        # Eq 19 taken literally, two thermal sets, on the size of the ablation studies
        _cavity("cavity 128x128 two sets", 128, 128, 1e5, 0.03, 30e-9, 100, sets=2),
        # the benchmark's cavity and its 1000-step check interval
        _cavity("cavity 256x256", 256, 256, 1e5, 0.03, 30e-9, 1000),
        # the precision configuration, state beyond L2: FP32 and FP16 (stochastic rounding)
        _cavity("cavity 1024x1024", 1024, 1024, 1e6, 0.02, 50e-9, 40),
        _cavity("cavity 1024x1024 fp16", 1024, 1024, 1e6, 0.02, 50e-9, 40, storage="f16"),
        # the largest single cavity, not square, BF16 rounded to nearest
        _cavity("cavity 1500x1000 bf16", 1500, 1000, 1e6, 0.02, 50e-9, 40, storage="bf16",
                nearest=True),
        # the parametric sweep of 80 uneven cavities
        dict(name="sweep 80", kind="sweep", n=0, low=0, high=0, storage="f32"),
        # inference for one warm start with the shipped weights
        dict(name="net forward 1", kind="net", grad=False, shipped=True, ny=256, nx=256, c0=16,
             hidden=64, batch=1),
        # one training batch of the shipped network's size
        dict(name="net gradient 16", kind="net", grad=True, shipped=False, ny=256, nx=256, c0=16,
             hidden=64, batch=16),
        # a small network, not square, odd batch and MLP width
        dict(name="net gradient small", kind="net", grad=True, shipped=False, ny=48, nx=64, c0=8,
             hidden=7, batch=3),
        # the library's GEMM on a square of its own benchmark
        dict(name="gemm 4096", kind="gemm", M=4096, N=4096, K=4096, a_k=True, b_k=True, splits=1),
    ]


def _cavity(name, nx, ny, Ra, phi, d_p, steps, storage="f32", nearest=False, sets=1,
            mask=B.F_ALL):
    return dict(name=name, kind="cavity", nx=nx, ny=ny, Ra=Ra, phi=phi, d_p=d_p, steps=steps,
                storage=storage, nearest=nearest, sets=sets, mask=mask)


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["cavity"] * 5 + ["net"] * 3 + ["sweep", "gemm"])
    if kind == "cavity":
        sets = 2 if rng.random() < 0.15 else 1
        hi = 256 if sets == 2 else 1200
        nx, ny = _log(rng, 24, hi), _log(rng, 24, hi)
        storage = rng.choice(["f32", "f32", "f16", "bf16"])
        c = _cavity("", nx, ny, 10.0 ** rng.uniform(3.0, 5.0 if ny < 64 else 6.0),
                    rng.choice([0.0, 0.01, 0.02, 0.03, 0.04]), rng.uniform(10e-9, 100e-9),
                    rng.randint(20, max(20, min(1000, 40 * 1000000 // (nx * ny)))), storage,
                    rng.random() < 0.3, sets,
                    # the ablations switch off any force but the drag that holds the others
                    B.F_ALL if rng.random() < 0.75 else B.F_ALL & ~rng.choice(
                        [B.F_BROWNIAN, B.F_THERMOPHORESIS, B.F_SAFFMAN, B.F_MAGNUS, B.F_GRAVITY,
                         B.F_BUOYANCY]))
    elif kind == "sweep":
        low = _log(rng, 32, 128)
        c = dict(kind="sweep", n=_log(rng, 4, 60), low=low, high=rng.randint(low, 512),
                 storage=rng.choice(["f32", "f32", "f16"]))
    elif kind == "net":
        c = dict(kind="net", grad=rng.random() < 0.5, shipped=False,
                 ny=16 * _log(rng, 2, 16), nx=16 * _log(rng, 2, 16), c0=rng.choice([8, 16, 16]),
                 hidden=_log(rng, 7, 64), batch=_log(rng, 1, 16))
    else:
        M, N, K = _log(rng, 64, 65536), _log(rng, 4, 4096), _log(rng, 12, 4096)
        while 2.0 * M * N * K > 2.0 * 4096 ** 3 or M * N > 4096 ** 2:
            M //= 2
        c = dict(kind="gemm", M=M, N=N, K=K, a_k=rng.random() < 0.7, b_k=rng.random() < 0.7,
                 splits=rng.choice([1, 1, 2, 8]))
    c.pop("name", None)
    return c


# ---- inputs ------------------------------------------------------------------------------------

def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _modes(g, n, ny, nx):
    """n smooth random fields [n][ny][nx] of order one: six cosine modes each."""
    k = torch.randint(0, 4, (n, 6, 2), device=DEV, generator=g).float() * math.pi
    a = torch.rand(n, 6, 1, device=DEV, generator=g) - 0.5
    y = torch.cos(k[..., :1] * (torch.arange(ny, device=DEV) + 0.5) / ny)
    x = torch.cos(k[..., 1:] * (torch.arange(nx, device=DEV) + 0.5) / nx)
    return torch.bmm((a * y).transpose(1, 2), x)


def _warm(g, nx, ny, phi):
    """Fields a warm start meets: a convection roll on the conduction profile with smooth
    departures of the temperature and the particles, and noise of the workloads' amplitude."""
    x = (torch.arange(nx, device=DEV) + 0.5) / nx
    y = (torch.arange(ny, device=DEV)[:, None] + 0.5) / ny
    sx, sy = torch.sin(math.pi * x), torch.sin(math.pi * y)
    m = _modes(g, 2, ny, nx)
    ux = 0.02 * sx ** 2 * torch.sin(2 * math.pi * y)
    uy = -0.02 * torch.sin(2 * math.pi * x) * sy ** 2
    w = torch.stack([ux, uy, 0.5 - x + 0 * y + 0.1 * sx * m[0], phi * (1 + 0.01 * m[1])])
    noise = 2 * torch.rand(4, ny, nx, device=DEV, generator=g) - 1
    amp = torch.tensor([1e-3, 1e-3, 1e-3, 1e-3 * phi], device=DEV)[:, None, None]
    return (w + amp * noise).float().contiguous()


def _conditions(n, seed):
    """(Ra, phi, d_p) of the training draw's ranges, as the network's entry points take them."""
    return WS.sample_conditions(n, seed).astype(np.float32)


def _sweep_cavities(case, seed):
    if case["n"] == 0:
        return workloads.sweep80()
    r = np.random.default_rng(7)  # sizes and parameters belong to the case, fields to the seed
    lo, hi = math.log(case["low"]), math.log(case["high"] + 1)
    return [dict(nx=int(math.exp(r.uniform(lo, hi))), ny=int(math.exp(r.uniform(lo, hi))),
                 Ra=10.0 ** r.uniform(3.0, 5.0), Pr=6.2, phi=0.01 * int(r.integers(0, 5)),
                 d_p=r.uniform(10e-9, 100e-9)) for _ in range(case["n"])]


def _net_inputs(case, seed):
    g = _generator(seed)
    ny, nx, b = case["ny"], case["nx"], case["batch"]
    cond = torch.from_numpy(_conditions(b, seed))
    if not case["grad"]:
        return dict(cond=cond.to(DEV), target=None)
    # training fields: smooth, with the spreads of the shipped network's normaliser
    spread = torch.tensor([0.02, 0.02, 0.3, 3e-4, 2e-3], device=DEV)[None, :, None, None]
    t = spread * _modes(g, b * 5, ny, nx).reshape(b, 5, ny, nx)
    phi = cond[:, 1].to(DEV)[:, None, None]
    t[:, 3] += phi
    t[:, 4] += 1 - phi
    return dict(cond=cond.to(DEV), target=t.contiguous())


def _net_params(case, seed):
    """(parameters, mean, scale): the shipped ones, or He-scaled random ones."""
    if case["shipped"]:
        d = np.load(WEIGHTS)
        return torch.from_numpy(d["params"]), d["mean"], d["scale"]
    g, out = torch.Generator().manual_seed(int(seed)), []
    for size, fan, scale in _net_segments(case["c0"], case["hidden"]):
        u = 2 * torch.rand(size, generator=g) - 1
        out.append(u * (scale * math.sqrt(6.0 / fan) if fan else 0.05))
    return (torch.cat(out).float(), np.array([0.0, 0.0, 0.01, 1e-6, -1e-5]),
            np.array([0.02, 0.02, 0.3, 3e-4, 2e-3]))


def _gemm_inputs(case, seed):
    g = _generator(seed)
    M, N, K = case["M"], case["N"], case["K"]
    a = torch.randn((M, K) if case["a_k"] else (K, M), device=DEV, generator=g).bfloat16()
    b = torch.randn((N, K) if case["b_k"] else (K, N), device=DEV, generator=g).bfloat16()
    return a, b


def _k_per_split(case):
    return ((case["K"] + case["splits"] - 1) // case["splits"] + 63) // 64 * 64


def prepare(case, seed):
    kind = case["kind"]
    if kind == "cavity":
        nx, ny = case["nx"], case["ny"]
        cav = B.Cavity(nx, ny, case["Ra"], 6.2, case["phi"], case["d_p"], device=DEV,
                       storage=STORAGE[case["storage"]], thermal_sets=case["sets"],
                       force_mask=case["mask"],
                       rounding=B.ROUND_NEAREST if case["nearest"] else B.ROUND_STOCHASTIC)
        return dict(kind=kind, cav=cav, warm=_warm(_generator(seed), nx, ny, case["phi"]),
                    steps=case["steps"],
                    state=torch.empty(cav.np, ny, nx, device=DEV),
                    fields=torch.empty(4, ny, nx, device=DEV))
    if kind == "sweep":
        g, cavs, warm = _generator(seed), [], []
        for c in _sweep_cavities(case, seed):
            cav = B.Cavity(c["nx"], c["ny"], c["Ra"], c["Pr"], c["phi"], c["d_p"], device=DEV,
                           storage=STORAGE[case["storage"]])
            warm.append(_warm(g, c["nx"], c["ny"], c["phi"]))
            cavs.append(cav.init(warm=warm[-1]))
        batch = B.Batch(cavs)
        batch.tune(64)
        out = torch.empty(sum(4 * c.nx * c.ny for c in cavs), device=DEV)
        views, at = [], 0
        for c in cavs:
            views.append(out[at:at + 4 * c.nx * c.ny].view(4, c.ny, c.nx))
            at += 4 * c.nx * c.ny
        return dict(kind=kind, batch=batch, cavs=cavs, warm=warm, out=out, views=views)
    if kind == "net":
        params, mean, scale = _net_params(case, seed)
        net = WS.WarmNet(case["ny"], case["nx"], case["c0"], case["hidden"], case["batch"],
                         device=DEV)
        net.set_params(params).set_normalizer(mean, scale)
        return dict(kind=kind, net=net, **_net_inputs(case, seed))
    a, b = _gemm_inputs(case, seed)
    return dict(kind=kind, a=a, b=b, a_k=case["a_k"], b_k=case["b_k"], splits=case["splits"],
                kps=_k_per_split(case))


def run(state):
    kind = state["kind"]
    if kind == "cavity":
        cav = state["cav"]
        cav.init(warm=state["warm"])
        cav.step(state["steps"])
        d = cav.diagnostics()
        return dict(state=cav.state_get(out=state["state"]),
                    fields=cav.fields(FIELDS, out=state["fields"]), **d)
    if kind == "sweep":
        for c, w in zip(state["cavs"], state["warm"]):
            c.init(warm=w)
        state["batch"].step(SWEEP_STEPS)
        hot, cold = state["batch"].nusselt()
        for c, v in zip(state["cavs"], state["views"]):
            c.fields(FIELDS, out=v)
        return dict(fields=state["out"], hot=hot.astype(np.float32), cold=cold.astype(np.float32))
    if kind == "net":
        if state["target"] is None:
            return dict(fields=state["net"].forward(state["cond"]))
        loss, grad = state["net"].loss_grad(state["cond"], state["target"])
        return dict(loss=loss, grad=grad)
    return dict(d=WS.gemm_bf16(state["a"], state["b"], state["a_k"], state["b_k"],
                               splits=state["splits"], k_per_split=state["kps"]))


def work(case):
    """Bytes and operations of one pass. A time step reads and writes its state once (27 or 36
    populations per node, the unit of every MLUPS figure here) and does about 600 operations per
    node; the network's inputs, parameters and results move once around its convolutions."""
    kind = case["kind"]
    if kind == "cavity":
        nodes = case["nx"] * case["ny"]
        elem = 4 if case["storage"] == "f32" else 2
        planes = 9 * (2 + case["sets"])
        return {"bytes": nodes * (case["steps"] * 2 * planes * elem + 4 * (4 + 4 + planes)),
                "flops": 600.0 * nodes * case["steps"]}
    if kind == "sweep":
        nodes = sum(c["nx"] * c["ny"] for c in _sweep_cavities(case, 0))
        elem = 4 if case["storage"] == "f32" else 2
        return {"bytes": nodes * (SWEEP_STEPS * 2 * 27 * elem + 4 * (4 + 4)),
                "flops": 600.0 * nodes * SWEEP_STEPS}
    if kind == "net":
        params = sum(s for s, _, _ in _net_segments(case["c0"], case["hidden"]))
        fields = 5 * case["batch"] * case["ny"] * case["nx"]
        flops = WS.conv_flops(case["ny"], case["nx"], case["c0"], case["batch"])
        return {"bytes": 4 * (fields + params * (2 if case["grad"] else 1)),
                "flops": flops * (3 if case["grad"] else 1)}
    M, N, K, z = case["M"], case["N"], case["K"], case["splits"]
    return {"bytes": 2 * (M + N) * K + 4 * z * M * N, "flops": 2.0 * M * N * K}


# ---- float64 restatements ------------------------------------------------------------------------

EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
W9 = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
MIR = (0, 1, 4, 3, 2, 8, 7, 6, 5)


def _constants(c):
    """Scales, ratios and relaxation times (Eqs 7-11, 22-24) of one cavity, FP64."""
    KB, ny, phi, d, Ra, Pr = 1.380649e-23, c["ny"], c["phi"], c["d_p"], c["Ra"], 6.2
    rf, cpf, kf, bf, mu, rp, cpp, kp, bp = (997.1, 4179.0, 0.613, 2.1e-4, 8.9e-4, 3970.0, 765.0,
                                            40.0, 0.85e-5)
    T0, dT, g, lf = 298.15, 10.0, 9.81, 0.17e-9
    U0 = 0.1 / math.sqrt(3.0)
    nu = U0 * ny * math.sqrt(Pr / Ra)
    al = nu / Pr
    rho_r, rhocp_r = phi * rp / rf + 1 - phi, phi * rp * cpp / (rf * cpf) + 1 - phi
    beta_r = phi * bp / bf + 1 - phi
    ReT = rf * KB * T0 / (3 * math.pi * mu * mu * lf)
    k_r = 1 + 64.7 * phi ** 0.764 * (lf / d) ** 0.369 * (kf / kp) ** 0.7476 * Pr ** 0.995 * \
        ReT ** 1.2321
    mu_r = 1 + 4.93 * phi + 222.4 * phi * phi
    rw0, rp0 = 1 - phi, phi * rp / rf
    Yw, Yp = rw0 / (rw0 + rp0), rp0 / (rw0 + rp0)
    tw, ttw = 3 * nu + 0.5, 3 * al + 0.5
    tp = (3 * nu * mu_r / rho_r + 0.5 - Yw * tw) / Yp if phi > 0 else tw
    ttp = (3 * al * k_r / rhocp_r + 0.5 - Yw * ttw) / Yp if phi > 0 else ttw
    nuf = mu / rf
    H = (Ra * nuf * nuf / Pr / (g * bf * dT)) ** (1 / 3)
    dx = H / ny
    dt = nu * dx * dx / nuf
    CF, vel = dt * dt / (rf * dx), dx / dt
    mun, rhon, kn = mu * mu_r, rf * rho_r, kf * k_r
    nun, bSt, Vp, Ap = mun / rhon, 18 * mun / (rp * d * d), math.pi * d ** 3 / 6, math.pi * d * d
    Kn, ks = lf / d, kn / kp
    KT = 6 * math.pi * 1.17 * (ks + 2.18 * Kn) / ((1 + 3 * 1.14 * Kn) * (1 + 2 * ks + 4.36 * Kn))
    return dict(rw0=rw0, rp0=rp0, tw=tw, tp=tp, ttw=ttw, ttp=ttp, k_r=k_r,
                buoy=beta_r * U0 * U0 / ny, gG=(1 - rf / rp) * g * dt * dt / dx, t_r=dT / T0,
                # lattice force per unit lattice moment: n_p = rho^p (rho_f / rho_p) / V_p
                cB=CF * (rf / rp) / Vp * rp * (2 * KB * T0 / (3 * math.pi * mun * d)) * Ap *
                (2 * KB * T0 / (math.pi * mun * d * d)) * (rf / rp) / dx,
                cT=CF * rf * bSt * KT * nun * dT / (dx * T0),
                cS=CF * (rf / rp) / Vp * 0.25 * 81.2 * mun * d * d * vel *
                math.sqrt(rhon * 8 * vel / (H * mun)),
                cM=CF * rf * bSt * 0.34 * 0.25 * vel * vel * H / nun * (d / H) ** 2.84,
                bdt=bSt * dt, cRe=rp * d * vel / mun, r_cp=cpp / cpf, phi_per=rf / rp)


class _Exact:
    """The twin-component step (Eqs 18-36, Table 1) of B cavities of one size in float64."""

    def __init__(self, cavs, warm, sets=1, mask=B.F_ALL):
        self.nx, self.ny, self.sets, self.mask = cavs[0]["nx"], cavs[0]["ny"], sets, mask
        cs = [_constants(c) for c in cavs]
        self.k = {n: torch.tensor([c[n] for c in cs], dtype=torch.float64,
                                  device=DEV)[:, None, None] for n in cs[0]}
        w = torch.stack(warm).double()
        ux, uy, th, phi = w[:, 0], w[:, 1], w[:, 2], w[:, 3]
        f = [self.equilibrium(r, ux, uy) for r in (1 - phi, phi / self.k["phi_per"], th)]
        self.f = f + ([f[2].clone()] if sets == 2 else [])
        self.then = None

    @staticmethod
    def equilibrium(rho, ux, uy):
        uu = 1.5 * (ux * ux + uy * uy)
        eu = [EX[q] * ux + EY[q] * uy for q in range(9)]
        return torch.stack([W9[q] * rho * (1 + 3 * eu[q] + 4.5 * eu[q] ** 2 - uu)
                            for q in range(9)], 1)

    def pull(self, f, thermal):
        out = torch.empty_like(f)
        for q in range(9):
            ex, ey = EX[q], EY[q]
            xs = slice(max(ex, 0), self.nx + min(ex, 0))
            xf = slice(max(-ex, 0), self.nx + min(-ex, 0))
            ys = slice(max(ey, 0), self.ny + min(ey, 0))
            yf = slice(max(-ey, 0), self.ny + min(-ey, 0))
            if thermal:
                if ex:
                    out[:, q] = -f[:, OPP[q]] + W9[q] * ex  # 2 W_q T_wall, T_wall = e_qx / 2
                out[:, q, :, xs] = f[:, MIR[q], :, xf]
            else:
                out[:, q] = f[:, OPP[q]]
            out[:, q, ys, xs] = f[:, q, yf, xf]
        return out

    def moments(self):
        p = [self.pull(f, s >= 2) for s, f in enumerate(self.f)]
        mx = lambda a: a[:, 1] - a[:, 3] + a[:, 5] - a[:, 6] - a[:, 7] + a[:, 8]  # noqa: E731
        my = lambda a: a[:, 2] - a[:, 4] + a[:, 5] + a[:, 6] - a[:, 7] - a[:, 8]  # noqa: E731
        rw, rp, th = p[0].sum(1), p[1].sum(1), p[2].sum(1)
        if self.sets == 2:
            c = self.k["r_cp"] * rp
            th = (rw * th + c * p[3].sum(1)) / (rw + c)
        return p, rw, rp, th, mx(p[0]), my(p[0]), mx(p[1]), my(p[1])

    def step(self):
        k, m = self.k, self.mask
        p, rw, rp, th, mwx, mwy, mpx, mpy = self.moments()
        rho = rw + rp
        Yw, Yp = rw / rho, rp / rho
        ux, uy = (mwx + mpx) / rho, (mwy + mpy) / rho
        has = rp > 1e-30
        rps = torch.where(has, rp, torch.ones_like(rp))
        uwx, uwy = mwx / rw, mwy / rw
        upx, upy = torch.where(has, mpx / rps, uwx), torch.where(has, mpy / rps, uwy)
        wx, wy = uwx - upx, uwy - upy

        def grad(a, thermal):
            w, e = a[..., :1], a[..., -1:]
            x = torch.cat([1 - w if thermal else w, a, -1 - e if thermal else e], -1)
            y = torch.cat([a[:, :1], a, a[:, -1:]], 1)
            return 0.5 * (x[..., 2:] - x[..., :-2]), 0.5 * (y[:, 2:] - y[:, :-2])

        (tx, ty), (rx, ry) = grad(th, True), grad(rp, False)
        T = 1 + th * k["t_r"]
        fx, fy = torch.zeros_like(rw), torch.zeros_like(rw)
        if m & B.F_BROWNIAN:
            c = -k["cB"] * rp * T * T
            fx, fy = fx + c * rx, fy + c * ry
        if m & B.F_THERMOPHORESIS:
            c = -k["cT"] * rp / T
            fx, fy = fx + c * tx, fy + c * ty
        if m & B.F_SAFFMAN:
            c = k["cS"] * rp * (upx ** 2 + upy ** 2) ** 0.25
            fx, fy = fx - c * wy, fy + c * wx
        if m & B.F_MAGNUS:
            i = torch.arange(self.nx, device=DEV, dtype=torch.float64)[None, :].expand_as(rw[0])
            j = torch.arange(self.ny, device=DEV, dtype=torch.float64)[:, None].expand_as(rw[0])
            z, s = torch.stack([i + 0.5, self.nx - i - 0.5, j + 0.5, self.ny - j - 0.5]).min(0)
            zh = 2 * z / self.ny
            c = k["cM"] * rp * ((uwx + upx) ** 2 + (uwy + upy) ** 2) * zh * (0.63 - zh)
            fx = fx + c * ((s == 0).double() - (s == 1).double())
            fy = fy + c * ((s == 2).double() - (s == 3).double())
        buoy = rho * k["buoy"] * th if m & B.F_BUOYANCY else torch.zeros_like(rw)
        gG = k["gG"] if m & B.F_GRAVITY else 0 * k["gG"]
        zero = torch.zeros_like(rw)
        fx, fy = torch.where(has, fx, zero), torch.where(has, fy, zero)
        Fpx, Fpy, Fwx, Fwy = fx, fy - rp * gG, -fx, buoy + k["rp0"] * gG - fy
        if m & B.F_DRAG:
            w = torch.sqrt(wx * wx + wy * wy)
            a = k["bdt"] * (1 + 0.15 * (k["cRe"] * w) ** 0.687) * (1 + rp / rw)
            E = -torch.expm1(-a)
            relax = 1 - Yp / k["tw"] - Yw / k["tp"]
            for x in (0, 1):
                b = (Fwx / rw - Fpx / rps, Fwy / rw - Fpy / rps)[x]
                J = rw * rp / rho * (E * relax * (wx, wy)[x] + (1 - E / a) * b)
                J = torch.where(has, J, zero)
                if x == 0:
                    Fpx, Fwx = Fpx + J, Fwx - J
                else:
                    Fpy, Fwy = Fpy + J, Fwy - J
        taus = [k["tw"], k["tp"]]
        taus += [k["ttw"], k["ttp"]] if self.sets == 2 else [Yw * k["ttw"] + Yp * k["ttp"]]
        force = [(Fwx, Fwy), (Fpx, Fpy)]
        for s, tau in enumerate(taus):
            eq = self.equilibrium((rw, rp, th, th)[s], ux, uy)
            out = p[s] - (p[s] - eq) / tau[:, None]
            if s < 2:
                out += torch.stack([3 * W9[q] * (EX[q] * force[s][0] + EY[q] * force[s][1])
                                    for q in range(9)], 1)
            self.f[s] = out

    def fields(self):
        _, rw, rp, th, mwx, mwy, mpx, mpy = self.moments()
        rho = rw + rp
        return torch.stack([(mwx + mpx) / rho, (mwy + mpy) / rho, th, rp * self.k["phi_per"]], 1)

    def nusselt(self, th):
        s = self.k["k_r"][:, 0, 0] * self.nx
        hot = ((4 - 9 * th[..., 0] + th[..., 1]) / 3).mean(1) * s
        cold = ((9 * th[..., -1] - th[..., -2] + 4) / 3).mean(1) * s
        return hot, cold

    def state(self):
        """Deviations from the conduction state, [B][planes][ny][nx]."""
        w = torch.tensor(W9, dtype=torch.float64, device=DEV)[None, :, None, None]
        tc = 0.5 - (torch.arange(self.nx, device=DEV, dtype=torch.float64) + 0.5) / self.nx
        rest = [self.k["rw0"][:, None], self.k["rp0"][:, None], tc, tc]
        return torch.cat([f - w * r for f, r in zip(self.f, rest)], 1)


def _exact_cavity(case, seed):
    e = _Exact([case], [_warm(_generator(seed), case["nx"], case["ny"], case["phi"])],
               case["sets"], case["mask"])
    then = e.fields()[0]
    for _ in range(case["steps"]):
        e.step()
    now = e.fields()[0]
    hot, cold = e.nusselt(now[None, 2])
    n2 = lambda a: float(a.square().sum().sqrt())  # noqa: E731
    r = max(n2(now[s] - then[s]) / (case["steps"] * n2(now[s])) if n2(now[s]) else 0.0
            for s in (slice(0, 2), slice(2, 3), slice(3, 4)))
    return dict(state=e.state()[0], fields=now, nu_hot=float(hot), nu_cold=float(cold),
                mass_w=float(e.f[0].sum()), mass_p=float(e.f[1].sum()), residual=r)


def _exact_sweep(case, seed):
    cavs, g = _sweep_cavities(case, seed), _generator(seed)
    warm = [_warm(g, c["nx"], c["ny"], c["phi"]) for c in cavs]
    sizes = {}
    for i, c in enumerate(cavs):
        sizes.setdefault((c["nx"], c["ny"]), []).append(i)
    if len(sizes) > 16:
        return None  # one pass per size: too slow in plain torch
    out, hot, cold = [None] * len(cavs), [0.0] * len(cavs), [0.0] * len(cavs)
    for ids in sizes.values():
        e = _Exact([cavs[i] for i in ids], [warm[i] for i in ids])
        for _ in range(SWEEP_STEPS):
            e.step()
        f = e.fields()
        h, c = e.nusselt(f[:, 2])
        for n, i in enumerate(ids):
            out[i], hot[i], cold[i] = f[n].reshape(-1), float(h[n]), float(c[n])
    return dict(fields=torch.cat(out), hot=np.array(hot), cold=np.array(cold))


def _net_layers(c0):
    """(channels in, channels out, stride, FiLM) in parameter order: e0..e4, d3..d0, out."""
    a, b, c, d = c0, 2 * c0, 4 * c0, 8 * c0
    return [(4, a, 1, 0), (a, b, 2, 0), (b, c, 2, 0), (c, d, 2, 0), (d, d, 2, 1),
            (2 * d, d, 1, 1), (d + c, c, 1, 1), (c + b, b, 1, 1), (b + a, a, 1, 1), (a, 5, 1, 0)]


def _net_segments(c0, hidden):
    """(size, fan-in or 0 for a bias, scale) of the flat parameter vector's parts."""
    out = []
    for cin, cout, _, _ in _net_layers(c0):
        out += [(cout * cin * 9, 9 * cin, 1.0), (cout, 0, 1.0)]
    F = 2 * sum(co for _, co, _, film in _net_layers(c0) if film)
    return out + [(3 * hidden, 3, 1.0), (hidden, 0, 1.0), (F * hidden, hidden, 0.1), (F, 0, 1.0)]


def _net_output(p, cond, ny, nx, c0, hidden):
    """The network's normalised output [b][5][ny][nx] from flat parameters, in p's type."""
    F = torch.nn.functional
    parts = torch.split(p, [s for s, _, _ in _net_segments(c0, hidden)])
    conv, (W1, b1, W2, b2) = parts[:-4], parts[-4:]
    c = torch.stack([(torch.log10(cond[:, 0]) - 4.5) / 1.5, (cond[:, 1] - 0.025) / 0.025,
                     (cond[:, 2] * 1e9 - 55) / 45], 1)
    r = F.silu(c @ W1.view(hidden, 3).T + b1) @ W2.view(-1, hidden).T + b2
    xi = ((torch.arange(nx, device=p.device, dtype=p.dtype) + 0.5) / nx - 0.5).expand(ny, nx)
    eta = ((torch.arange(ny, device=p.device, dtype=p.dtype) + 0.5) / ny - 0.5)[:, None]
    X = torch.stack([torch.ones_like(xi), xi, eta.expand(ny, nx), 4 * xi * eta])
    y, skip, at = X.expand(cond.shape[0], 4, ny, nx), [], 0
    for n, (cin, cout, stride, film) in enumerate(_net_layers(c0)):
        if 5 <= n < 9:
            y = torch.cat([y.repeat_interleave(2, 2).repeat_interleave(2, 3), skip[8 - n]], 1)
        y = F.conv2d(y, conv[2 * n].view(cout, cin, 3, 3), conv[2 * n + 1], stride, 1)
        if film:
            y = (1 + r[:, at:at + cout, None, None]) * y + r[:, at + cout:at + 2 * cout, None, None]
            at += 2 * cout
        y = F.silu(y) if n < 9 else y
        skip.append(y)
    return y


def _exact_net(case, seed):
    params, mean, scale = _net_params(case, seed)
    i = _net_inputs(case, seed)
    p = params.to(DEV).double().requires_grad_(case["grad"])
    cond = i["cond"].double()
    m, s = (torch.tensor(v, dtype=torch.float64, device=DEV)[None, :, None, None]
            for v in (mean, scale))
    phi = cond[:, 1, None, None]
    base = torch.zeros(case["batch"], 5, 1, 1, dtype=torch.float64, device=DEV)
    base[:, 3], base[:, 4] = phi, 1 - phi
    out = _net_output(p, cond, case["ny"], case["nx"], case["c0"], case["hidden"])
    if case["grad"]:
        loss = (out - (i["target"].double() - base - m) / s).square().mean()
        loss.backward()
        return dict(loss=float(loss.detach()), grad=p.grad)
    dev = m + s * out
    dev[:, 3:] -= dev[:, 3:].mean((2, 3), keepdim=True)  # the cavity's masses are kept
    return dict(fields=base + dev)


def exact(case, seed):
    kind = case["kind"]
    if kind == "cavity":
        return _exact_cavity(case, seed)
    if kind == "sweep":
        return _exact_sweep(case, seed)
    if kind == "net":
        with torch.set_grad_enabled(case["grad"]):
            return _exact_net(case, seed)
    a, b = _gemm_inputs(case, seed)
    a, b = (a if case["a_k"] else a.T).double(), (b if case["b_k"] else b.T).double()
    k, d = _k_per_split(case), []
    for z in range(case["splits"]):
        d.append(a[:, z * k:(z + 1) * k] @ b[:, z * k:(z + 1) * k].T)
    return dict(d=torch.stack(d))
