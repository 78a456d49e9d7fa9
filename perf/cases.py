"""What the library is measured on: the calls its users' programs make, from one step on a
small grid to adaptive runs at 2048^2, an ensemble, standalone transforms and the network.

A case is a dict of plain values. listed() gives the fixed ones, draw() more of the same
ranges; prepare() makes a case's inputs and handles on the GPU from a seed, run() makes one
pass through the public binding, work() says what a pass cannot do without, and exact()
gives what run() returns as plain torch computes it in 64 bits (the paper's formulas on
full real transforms, written here independently of the library).

Grids are powers of two (the library takes no others); the odd sizes are batches, step and
trial counts and member lists. Adaptive runs keep the zero-stability cap on the step ratio:
without it the first jumps from k_min follow rounding noise, and no two programs' runs can
be compared.
"""
import functools
import math

import numpy as np
import torch

from paper_2006_04784_gb300 import fch

L = 4.0 * math.pi
EPS = 0.1
PREC = {"f64": fch.FCH_FP64, "f32": fch.FCH_MIXED, "f32x2": fch.FCH_FP32X2}
RTYPE = {"f64": torch.float64, "f32": torch.float32, "f32x2": torch.float64}


# ------------------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest call: one step on a small grid and the diagnostics printed beside it
        dict(name="step_64_f64", kind="fixed", n=64, prec="f64", scheme="imex", field="circle", q=0.0, eta2=3.0, dt=1e-3, steps=1, diag=True),
        # fixed steps of the 128^2 circular bilayer (the plain double-precision workload)
        dict(name="fixed_128_f64", kind="fixed", n=128, prec="f64", scheme="imex", field="circle", q=0.0, eta2=3.0, dt=1e-3, steps=100, diag=False),
        # the paper's benchmark size, super-critical strength, double-float
        dict(name="imex_256_f32x2", kind="adaptive", n=256, prec="f32x2", scheme="imex", field="curve", q=0.0, eta2=3.0, sigma=1e-5, trials=64),
        # the nonlinear solver at the same size: its iterations loop on the device
        dict(name="psd_256_f32x2", kind="adaptive", n=256, prec="f32x2", scheme="psd", field="curve", q=0.0, eta2=3.0, sigma=1e-5, trials=24),
        # the 512^2 comparison of the schemes in double precision
        dict(name="sav_512_f64", kind="adaptive", n=512, prec="f64", scheme="sav", field="curve", q=0.0, eta2=3.0, sigma=1e-5, trials=32),
        # the regularised well (q > 0, sech and tanh at every point) on the paper's 512^2 benchmark
        dict(name="foot_512_f32x2", kind="adaptive", n=512, prec="f32x2", scheme="imex", field="curve", q=0.5, eta2=3.0, sigma=1e-5, trials=32),
        # the benchmark workload: 1024^2 bilayer network, critical strength
        dict(name="imex_1024_f32x2", kind="adaptive", n=1024, prec="f32x2", scheme="imex", field="network", q=0.0, eta2=1.5, sigma=1e-5, trials=48),
        # the same at the largest grid the library takes
        dict(name="imex_2048_f32x2", kind="adaptive", n=2048, prec="f32x2", scheme="imex", field="network", q=0.0, eta2=1.5, sigma=1e-5, trials=32),
        # a sweep over schemes and strengths on uneven grids, advanced as one graph
        dict(name="sweep_11_f32x2", kind="ensemble", sizes="256,256,512,256,512,256,256,512,256,1024,256", schemes="imex,sav,etd", prec="f32x2",
             field="curve", q=0.0, sigma=1e-5, rounds=8, launches=3),
        # standalone batched transforms there and back, single precision
        dict(name="fft_1024_f32_b16", kind="fft", n=1024, prec="f32", batch=16),
        # one inference of the trained-size network at 1024^2 on the tensor cores
        dict(name="fno_1024_tc", kind="fno", n=1024, batch=1, mode=2, train=False),
        # one optimiser step of the network on its training grid
        dict(name="fno_train_128_b8", kind="fno", n=128, batch=8, mode=0, train=True),
    ]


def draw(rng):
    fixed = [{k: v for k, v in c.items() if k != "name"} for c in listed()]
    while True:
        case = _draw(rng)
        if case not in fixed:
            return case


def _draw(rng):
    kind = rng.choice(["fixed", "adaptive", "adaptive", "adaptive", "ensemble", "fft", "fft", "fno"])
    q, eta2 = rng.choice([(0.0, 3.0), (0.0, 1.5), (0.0, 3.0), (0.2, 3.0), (0.5, 3.0)])
    field = rng.choice(["circle", "curve", "network"])
    if kind == "fixed":
        n = 2 ** rng.randint(4, 10)
        prec, scheme = rng.choice(["f64", "f32", "f32x2"]), rng.choice(["imex", "imex", "sav", "psd"])
        if prec == "f32" and scheme == "psd":
            scheme = "imex"  # its tolerance lies below single precision
        most = 100 if n <= 256 else 24
        most = max(1, most // 12) if scheme == "psd" else most
        return dict(kind=kind, n=n, prec=prec, scheme=scheme, field=field, q=0.0, eta2=eta2, dt=round(1e-4 * 10 ** rng.random(), 6),
                    steps=max(1, int(round(most ** rng.random()))), diag=rng.random() < 0.5)
    if kind == "adaptive":
        prec = rng.choice(["f64", "f32x2", "f32x2"])
        n = 2 ** rng.randint(6, 10 if prec == "f64" else 11)
        scheme = rng.choice(["imex", "imex", "sav", "etd", "psd"])
        if n == 2048 or q > 0 and scheme == "psd":
            scheme = rng.choice(["imex", "sav"])
        most = {"imex": 48, "sav": 48, "etd": 32, "psd": 24}[scheme]
        if n >= 1024:
            most = {"f64": 12, "f32x2": 24}[prec]
        return dict(kind=kind, n=n, prec=prec, scheme=scheme, field=field, q=q, eta2=eta2, sigma=rng.choice([1e-4, 1e-5, 1e-6]),
                    trials=rng.randint(most // 2, most))
    if kind == "ensemble":
        m = rng.randint(3, 13)
        return dict(kind=kind, sizes=",".join(str(2 ** rng.choice([7, 8, 8, 9])) for _ in range(m)),
                    schemes=rng.choice(["imex", "imex,sav", "imex,sav,etd"]), prec=rng.choice(["f64", "f32x2", "f32x2"]), field=field, q=0.0, sigma=1e-5,
                    rounds=8, launches=rng.randint(1, 2))
    if kind == "fft":
        n = 2 ** rng.randint(4, 11)
        most = min(33, max(2, (1 << 24) // (n * n)))
        return dict(kind=kind, n=n, prec=rng.choice(["f64", "f32", "f32"]), batch=max(1, int(round(most ** rng.random()))))
    if rng.random() < 0.4:
        return dict(kind="fno", n=rng.choice([64, 128]), batch=rng.randint(1, 8), mode=0, train=True)
    return dict(kind="fno", n=2 ** rng.randint(6, 10), batch=rng.randint(1, 3), mode=rng.choice([0, 1, 2, 2]), train=False)


# ------------------------------------------------------------------------------ inputs
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


@functools.lru_cache(maxsize=1)
def _stream():
    return torch.cuda.Stream()  # one stream for everything a program runs


def _field(kind, n, seed):
    """An initial field of the paper's kind: a bilayer of half-width R along the zero set of
    phi (a circle with noise, a closed curve with random modes, or a random network)."""
    dev, g = _device(), np.random.default_rng(seed)
    c = torch.arange(n, dtype=torch.float64, device=dev) * (L / n) - 0.5 * L
    X, Y = c[None, :], c[:, None]
    R, d, noise = 0.14725, 0.2, None
    if kind == "circle":
        phi = torch.sqrt(X * X + Y * Y) - 2.0
        gen = torch.Generator(device=dev)
        gen.manual_seed(int(seed))
        noise = 1e-3 * (2.0 * torch.rand((n, n), dtype=torch.float64, device=dev, generator=gen) - 1.0)
    elif kind == "curve":
        amp, ph = 0.5 * EPS * g.random(7), 2.0 * math.pi * g.random(7)
        th = torch.atan2(Y.expand(n, n), X.expand(n, n))
        rho = 3.0
        for m in range(2, 9):
            rho = rho + amp[m - 2] * torch.cos(m * (th - ph[m - 2]))
        phi = torch.sqrt(X * X + Y * Y) - rho
    else:
        d = 0.75
        ms = [(a, b) for a in range(-6, 7) for b in range(0, 7) if 4 <= a * a + b * b <= 36 and (b > 0 or a > 0)]
        cm, th = g.standard_normal(len(ms)), 2.0 * math.pi * g.random(len(ms))
        cm = cm / math.sqrt(sum(0.5 * v * v * 0.25 * (a * a + b * b) for v, (a, b) in zip(cm, ms)))
        phi = torch.zeros((n, n), dtype=torch.float64, device=dev)
        for v, t, (a, b) in zip(cm, th, ms):
            ax, ay = 0.5 * a * X + float(t), 0.5 * b * Y
            phi = phi + float(v) * (torch.cos(ax) * torch.cos(ay) - torch.sin(ax) * torch.sin(ay))
    u = -1.0 + torch.tanh((phi + R) / EPS) - torch.tanh((phi - R) / EPS) + EPS * d / 1.7 ** 2
    return (u if noise is None else u + noise).contiguous()


def _well(q, u):
    """(W, W', W'') of the regularised well W_q on a tensor"""
    v, w = u + 1.0, u - 1.0
    A, A1, A2 = 0.5 * v * v, v, torch.ones_like(u)
    if q:
        x = v / EPS
        e = torch.exp(-x.abs())
        sech, th = 2.0 * e / (1.0 + e * e), torch.tanh(x)
        A, A1, A2 = A + q * EPS * (1.0 - sech), A1 + q * sech * th, A2 + q / EPS * sech * (2.0 * sech * sech - 1.0)
    B, B1 = 0.5 * w * w + 0.1 * (u - 2.0), w + 0.1
    return A * B, A1 * B + A * B1, A2 * B + 2.0 * A1 * B1 + A


@functools.lru_cache(maxsize=None)
def _sav_constants(q, eta2):
    """(zeta, D0): above -min W'' and -min of the rest of E1, as the scheme asks"""
    W, W1, W2 = _well(q, torch.linspace(-4.0, 4.0, 600001, dtype=torch.float64))
    return float(-W2.min()) + 0.1, L * L * (max(0.0, float(-(0.5 * W1 * W1 - eta2 * W).min())) + 1.0)


def _params(case, eta1=1.45):
    eta2 = case.get("eta2", 3.0) * EPS
    zeta, D0 = _sav_constants(case["q"], eta2)
    return fch.params_default(case["q"], prec=PREC[case["prec"]], eta1=eta1 * EPS, eta2=eta2, zeta=zeta, D0=D0, zero_stab_cap=1)


def _members(case):
    """(size, scheme, eta1 / eps) of an ensemble's members: a sweep over eta1 in [1, 3]"""
    sizes, schemes = [int(s) for s in case["sizes"].split(",")], case["schemes"].split(",")
    return [(n, schemes[i % len(schemes)], 1.0 + 2.0 * i / max(1, len(sizes) - 1)) for i, n in enumerate(sizes)]


FNO = dict(width=32, layers=4, modes=16, proj=64)


def _fno_shapes():
    K, W = FNO["modes"] * (2 * FNO["modes"] - 1), FNO["width"]
    s = [("P", (W, 2)), ("bP", (W,))]
    for l in range(FNO["layers"]):
        s += [("W%d" % l, (W, W)), ("b%d" % l, (W,)), ("R%d" % l, (K, W, W, 2))]
    return s + [("Q1", (FNO["proj"], W)), ("bQ1", (FNO["proj"],)), ("Q2", (FNO["proj"],)), ("bQ2", (1,))]


def _fno_inputs(case, seed):
    """seeded weights (fan-in scaled), inputs (a state, a normalised smooth correction) and targets"""
    g, n, b = np.random.default_rng(seed), case["n"], case["batch"]
    parts = []
    for name, sh in _fno_shapes():
        size = int(np.prod(sh))
        if name[0] == "b":
            parts.append(g.uniform(-0.1, 0.1, size))
        elif name[0] == "R":
            parts.append(g.uniform(0.0, 1.0, size) / FNO["width"] ** 2)
        else:
            parts.append(g.uniform(-1.0, 1.0, size) / math.sqrt(sh[-1]))
    p = np.concatenate(parts).astype(np.float32)
    a, t = [], []
    for i in range(b):
        u = _field("curve", n, 1000 * seed + i)
        v = _field("curve", n, 1000 * seed + 500 + i) - u
        w = _field("network", n, 1000 * seed + i) - u
        a.append(torch.stack([u, v / v.square().mean().sqrt()]))
        t.append(w / w.square().mean().sqrt())
    return p, torch.stack(a).float().contiguous(), torch.stack(t).float().contiguous()


def _fft_input(case, seed):
    gen = torch.Generator(device=_device())
    gen.manual_seed(int(seed))
    n = case["n"]
    x = torch.stack([_field("curve", n, seed + i % 3) for i in range(min(3, case["batch"]))])
    x = x[torch.arange(case["batch"], device=x.device) % x.shape[0]]
    return (x + 0.5 * torch.randn(x.shape, dtype=torch.float64, device=x.device, generator=gen)).to(RTYPE[case["prec"]]).contiguous()


def prepare(case, seed):
    kind, dev = case["kind"], _device()
    s = dict(case=case)
    if kind in ("fixed", "adaptive"):
        s["u0"] = _field(case["field"], case["n"], seed).to(RTYPE[case["prec"]])
        s["out"] = torch.empty_like(s["u0"])
        s["ctx"] = fch.Context(case["n"], _params(case), L=L, stream=_stream())
    elif kind == "ensemble":
        mem = _members(case)
        s["u0"] = [_field(case["field"], n, seed + 17 * i) for i, (n, _, _) in enumerate(mem)]
        s["out"] = [torch.empty_like(u) for u in s["u0"]]
        s["ens"] = fch.Ensemble([n for n, _, _ in mem], [_params(case, e) for _, _, e in mem], L=L, stream=_stream())
    elif kind == "fft":
        s["x"] = _fft_input(case, seed)
        n = case["n"]
        s["X"] = torch.empty((case["batch"], n // 2 + 1, n), dtype=torch.complex128 if case["prec"] == "f64" else torch.complex64, device=dev)
        s["y"] = torch.empty_like(s["x"])
        s["plan"] = fch.FFTPlan(n, PREC[case["prec"]], stream=_stream())
    else:
        p, s["a"], s["t"] = _fno_inputs(case, seed)
        s["y"] = torch.empty((case["batch"], case["n"], case["n"]), dtype=torch.float32, device=dev)
        s["net"] = fch.FNO(**FNO, stream=_stream())
        s["net"].set_params(p)
        s["net"].set_bf16(case["mode"])
    torch.cuda.synchronize()  # the inputs are ready for the program's stream
    return s


# ------------------------------------------------------------------------------ one pass
def _stats(st):
    # the last error estimate itself is left out: it is a difference near rounding level whose
    # ninth digit is noise; the step sizes that it sets are here
    return {"counts": np.array([st["n_steps"], st["n_rejects"], st["n_attempts"], st["n_psd_iter"]]),
            "t": np.array([st["t"], st["k_last"]])}


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "fixed":
        ctx = s["ctx"]
        ctx.set_state_device(s["u0"])
        if case["steps"] == 1:
            ctx.step(case["scheme"], case["dt"])
        else:
            ctx.run_fixed(case["scheme"], case["dt"], case["steps"])
        ctx.get_state_device(s["out"])
        if case["diag"]:
            return {"u": s["out"], "diag": np.array([ctx.energy(), ctx.mass()])}
        ctx.synchronize()  # where a failed step is reported
        return {"u": s["out"]}
    if kind == "adaptive":
        ctx = s["ctx"]
        ctx.set_state_device(s["u0"])
        st = ctx.run_adaptive(case["scheme"], case["sigma"], 1e3, max_attempts=case["trials"], raise_on_timeout=False)
        ctx.get_state_device(s["out"])
        return {"u": s["out"], "stats": _stats(st)}
    if kind == "ensemble":
        ens, mem = s["ens"], _members(case)
        for i, u in enumerate(s["u0"]):
            ens[i].set_state_device(u)
        st = ens.run_adaptive_each([c for _, c, _ in mem], [case["sigma"]] * len(mem), 1e3, rounds=case["rounds"], max_launches=case["launches"],
                                   raise_on_timeout=False)
        for i, u in enumerate(s["out"]):
            ens[i].get_state_device(u)
        return {"u": list(s["out"]), "stats": {"counts": np.array([[x["n_steps"], x["n_rejects"], x["n_attempts"]] for x in st]),
                                               "t": np.array([[x["t"], x["k_last"]] for x in st])}}
    if kind == "fft":
        s["plan"].r2c(s["x"], s["X"])
        s["plan"].c2r(s["X"], s["y"])
        return {"X": s["X"], "y": s["y"]}
    s["net"].forward(s["a"], s["y"])
    if not case["train"]:
        return {"y": s["y"]}
    loss = s["net"].backward(s["t"])
    s["net"].adam(1e-4)
    return {"y": s["y"], "loss": loss, "grads": s["net"].grads()}


# ------------------------------------------------------------------------------ what a pass cannot do without
def _step_work(n, prec, scheme, steps, adaptive, iters=0):
    """A step reads u^n and u^{n-1} (half spectra) and writes u^{n+1}; an adaptive trial also
    reads F(u^n), F(u^{n-1}) and writes F. Transforms: four fields each way a step (twice
    that with ETD's second stage), four more for F; the solver's iterations four each."""
    h = (n // 2 + 1) * n * (8 if prec == "f32" else 16)
    ffts = {"imex": 4, "sav": 4, "etd": 8, "psd": 2 + 4 * iters}[scheme] + (4 if adaptive else 0)
    flop = 2.5 * n * n * math.log2(n * n) * ffts + 60.0 * n * n
    io = 2 * n * n * (4 if prec == "f32" else 8) + 2 * h
    return steps * (6 if adaptive else 3) * h + io, steps * flop + 4 * 2.5 * n * n * math.log2(n * n)


def work(case):
    kind = case["kind"]
    if kind == "fixed":
        b, f = _step_work(case["n"], case["prec"], case["scheme"], case["steps"], False, 10)
    elif kind == "adaptive":
        b, f = _step_work(case["n"], case["prec"], case["scheme"], case["trials"], True, 5)
    elif kind == "ensemble":
        w = [_step_work(n, case["prec"], c, case["rounds"] * case["launches"], True) for n, c, _ in _members(case)]
        b, f = sum(x for x, _ in w), sum(x for _, x in w)
    elif kind == "fft":
        n, r = case["n"], 8 if case["prec"] == "f64" else 4
        b = case["batch"] * 2 * (n * n * r + (n // 2 + 1) * n * 2 * r)
        f = case["batch"] * 2 * 2.5 * n * n * math.log2(n * n)
    else:
        W, W2, M, nl = FNO["width"], FNO["proj"], FNO["modes"], FNO["layers"]
        n, pts = case["n"], case["batch"] * case["n"] ** 2
        num = sum(int(np.prod(sh)) for _, sh in _fno_shapes())
        # the layers' channel products, the transforms along x and y restricted to the kept modes, the projection
        f = pts * (nl * (2 * W * W + 2 * 4 * W * M) + 4 * W + 2 * W * W2 + 4 * W2) + case["batch"] * nl * 2 * 8 * W * M * (2 * M - 1) * n
        b = 12 * pts + num * (2 if case["mode"] else 4)
        if case["train"]:
            f, b = 3 * f, b + 4 * pts + num * 4 * 8
    return {"bytes": float(b), "flops": float(f)}


# ------------------------------------------------------------------------------ the same in 64 bits
class _Flow:
    """The schemes, the third-order predictor and the step-size controller in float64 torch."""

    LK = [1e-6, 1e-5, 5e-5, 1e-4, 5e-4, 1e-3, 5e-3, 1e-2, 2e-2, 3e-2]
    LT = {0.0: [1, 1.07, 1.11, 1.14, 1.24, 1.34, 1.60, 1.738, 1.804, 1.855], 0.2: [1, 1.04, 1.15, 1.28, 1.50, 1.70, 1.87, 1.92, 1.95, 1.97],
          0.5: [1, 1.20, 1.32, 1.45, 1.72, 1.83, 1.965, 1.97, 1.985, 1.99]}
    NU = {0.0: (1e-3, 0.05), 0.2: (2e-5, 0.02), 0.5: (1e-6, 0.01)}

    def __init__(self, n, q, eta1, eta2, u0):
        self.n, self.q, self.e1, self.e2 = n, q, eta1, eta2
        m = torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device=u0.device)
        mh = torch.arange(n // 2 + 1, dtype=torch.float64, device=u0.device)
        self.k2 = (2.0 * math.pi / L) ** 2 * (m[:, None] ** 2 + mh[None, :] ** 2)
        self.ik2 = torch.where(self.k2 > 0, 1.0 / self.k2.clamp_min(1e-300), torch.zeros_like(self.k2))
        self.am = 1.7 * (1.0 + q / EPS)
        self.s = (EPS * EPS * self.k2 + self.am) ** 2
        self.zeta, self.D0 = _sav_constants(q, eta2)
        self.h2 = (L / n) ** 2
        self.u, self.um, self.uh, self.umh = u0, torch.zeros_like(u0), self.F_(u0), torch.zeros_like(self.F_(u0))
        self.kn, self.ktrial, self.t, self.k_last, self.e = 0.0, 0.0, 0.0, 0.0, 0.0
        self.r, self.rm = math.sqrt(self.sav(u0)[0] + self.D0), 0.0
        self.attempts = 0

    def F_(self, a):
        return torch.fft.rfft2(a)

    def R_(self, a):
        return torch.fft.irfft2(a, s=(self.n, self.n))

    def pieces(self, u):
        return (*_well(self.q, u), self.R_(-self.k2 * self.F_(u)))

    def mu(self, u):  # spectrum of delta E / delta u
        W, W1, W2, lu = self.pieces(u)
        w = EPS * EPS * lu - W1
        return -EPS * EPS * self.k2 * self.F_(w) + self.F_(-W2 * w + EPS * EPS * self.e1 * lu - self.e2 * W1)

    def rhs(self, u):
        return self.R_(-self.k2 * self.mu(u))

    def nimex(self, u):
        W, W1, W2, lu = self.pieces(u)
        a = EPS * EPS * (self.am - W2 + self.e1) * lu + W2 * W1 - self.am ** 2 * u - self.e2 * W1
        return self.F_(a) - EPS * EPS * self.k2 * self.F_(self.am * u - W1)

    def sav(self, u):
        W, W1, W2, lu = self.pieces(u)
        e1 = self.h2 * float((-EPS * EPS * lu * (W1 + self.zeta * u) + 0.5 * W1 * W1 - self.e2 * W).sum())
        v = EPS * EPS * self.k2 * self.F_(W1 + self.zeta * u) + self.F_(-EPS * EPS * (W2 + self.zeta) * lu + W1 * W2 - self.e2 * W1)
        return e1, v

    def energy(self):
        W, W1, W2, lu = self.pieces(self.u)
        w = EPS * EPS * lu - W1
        return self.h2 * float((0.5 * w * w - self.e2 * W + 0.5 * EPS * EPS * self.e1 * self.u * lu).sum())

    def bdf2(self, k):
        if self.kn <= 0:
            return 1.0 / k, -1.0 / k, 0.0, 0.0
        return 1.0 / k + 1.0 / (k + self.kn), -1.0 / k - 1.0 / self.kn, 1.0 / self.kn - 1.0 / (k + self.kn), k / self.kn

    def trial(self, scheme, k, itol):
        a, b, c, g = self.bdf2(k)
        k2, e2 = self.k2, EPS * EPS
        us = self.u + g * (self.u - self.um) if g else self.u
        r = self.r
        if scheme == "imex":
            v = (-b * self.uh - c * self.umh - k2 * self.nimex(us)) / (a + k2 * self.s)
        elif scheme == "sav":
            e1, V = self.sav(us)
            X = V / math.sqrt(e1 + self.D0)
            l0 = e2 * e2 * k2 * k2 + 2.0 * self.am * e2 * k2 + self.am ** 2
            l1 = -e2 * (self.e1 + 2.0 * self.zeta) * k2 - 2.0 * self.am * e2 * k2 - self.am ** 2
            p = (-b * self.uh - c * self.umh - k2 * l1 * self.F_(us)) / (a + k2 * l0)
            qq = -k2 * X / (a + k2 * l0)
            xr = self.R_(X)
            x1 = self.h2 * float((xr * self.R_(a * p + b * self.uh + c * self.umh)).sum())
            x2 = self.h2 * float((xr * self.R_(qq)).sum())
            r = (-b * self.r - c * self.rm + 0.5 * x1) / (a * (1.0 - 0.5 * x2))
            v = p + r * qq
        elif scheme == "etd":
            ell = -k2 * self.s - 1e-2 - 15.0 * e2 * k2
            z, lin = ell * k, 1e-2 + 15.0 * e2 * k2
            small, em = z.abs() < 1e-2, torch.expm1(z)
            zs = torch.where(small, torch.ones_like(z), z)
            t1, t2 = torch.zeros_like(z), torch.zeros_like(z)
            for j in range(11, -1, -1):
                t1, t2 = t1 * z + 1.0 / math.factorial(j + 1), t2 * z + 1.0 / math.factorial(j + 2)
            p1, p2 = torch.where(small, t1, em / zs), torch.where(small, t2, (em - zs) / (zs * zs))
            n0 = -k2 * self.nimex(self.u) + lin * self.uh
            ut = torch.exp(z) * self.uh + k * p1 * n0
            v = ut + k * p2 * (-k2 * self.nimex(self.R_(ut)) + lin * ut - n0)
        else:
            if k <= self.LK[0]:
                lam = self.LT[self.q][0]
            else:
                lam = float(np.interp(k, self.LK, self.LT[self.q]))
            y, v = us, self.F_(us)
            for _ in range(1000):
                R = self.mu(y) + (a * v + b * self.uh + c * self.umh) * self.ik2
                d = torch.where(k2 > 0, -R / (self.s + a * self.ik2), torch.zeros_like(R))
                v = v + lam * d
                y = self.R_(v)
                if float(self.R_(d).norm() / y.norm()) < itol:
                    break
        return v, r

    def accept(self, v, r, k):
        self.u, self.um, self.uh, self.umh = self.R_(v), self.u, v, self.uh
        self.r, self.rm, self.kn, self.ktrial, self.k_last = r, self.r, k, k, k
        self.t += k

    def fixed(self, scheme, dt, steps):
        for _ in range(steps):
            self.accept(*self.trial(scheme, dt, 1e-10), dt)

    def adaptive(self, scheme, sigma, trials):
        """the backward-Euler start at k_min, then `trials` trials less the start"""
        nu, kmax = self.NU[self.q]
        itol, kmax = nu * sigma, kmax if scheme == "psd" else math.inf
        Fm = self.rhs(self.u)
        self.accept(*self.trial(scheme, 1e-9, itol), 1e-9)
        Fn = self.rhs(self.u)
        for _ in range(trials - 1):
            k, kn = self.ktrial, self.kn
            v, r = self.trial(scheme, k, itol)
            y = self.R_(v)
            F, g = self.rhs(y), k / kn
            up = self.u + k / 6.0 * ((3.0 + 2.0 * g) / (1.0 + g) * F + (3.0 + g) * Fn - g * g / (1.0 + g) * Fm)
            self.e = float((y - up).norm() / up.norm())
            new = max(1e-9, min(0.9 * k * (sigma / max(self.e, 1e-16)) ** (1.0 / 3.0), (1.0 + math.sqrt(2.0)) * k, kmax))
            if self.e <= sigma or k <= 1e-9:
                self.accept(v, r, k)
                Fm, Fn = Fn, F
            self.ktrial = new


def _fno_forward(p, a):
    """the network in 64 bits on full transforms; p: name -> tensor"""
    M, n, W = FNO["modes"], a.shape[-1], FNO["width"]
    ky = [q if q < M else n - (q - M + 1) for q in range(2 * M - 1)]
    h = torch.einsum("ci,bixy->bcxy", p["P"], a) + p["bP"][None, :, None, None]
    for l in range(FNO["layers"]):
        Rc = torch.view_as_complex(p["R%d" % l].contiguous()).reshape(M, 2 * M - 1, W, W)
        X = torch.fft.rfft2(h)[:, :, ky, :M]
        Z = torch.einsum("kqoi,biqk->boqk", Rc, X)
        Y = torch.zeros((a.shape[0], W, n, n // 2 + 1), dtype=Z.dtype, device=a.device)
        Y[:, :, ky, :M] = Z
        col = Y[..., 0]
        col = 0.5 * (col + torch.conj(torch.roll(torch.flip(col, [-1]), 1, -1)))
        Y = torch.cat([col[..., None], Y[..., 1:]], dim=-1)
        h2 = torch.einsum("cj,bjxy->bcxy", p["W%d" % l], h) + p["b%d" % l][None, :, None, None] + torch.fft.irfft2(Y, s=(n, n))
        h = torch.nn.functional.gelu(h2) if l < FNO["layers"] - 1 else h2
    z = torch.nn.functional.gelu(torch.einsum("dc,bcxy->bdxy", p["Q1"], h) + p["bQ1"][None, :, None, None])
    return torch.einsum("d,bdxy->bxy", p["Q2"], z) + p["bQ2"][0]


def _one(case, seed, n, scheme, eta1, steps):
    u0 = _field(case["field"], n, seed).to(RTYPE[case["prec"]]).double()
    f = _Flow(n, case["q"], eta1 * EPS, case.get("eta2", 3.0) * EPS, u0)
    if case["kind"] == "fixed":
        f.fixed(scheme, case["dt"], steps)
    else:
        f.adaptive(scheme, case["sigma"], steps)
    return f


def exact(case, seed):
    kind = case["kind"]
    if kind == "fixed":
        f = _one(case, seed, case["n"], case["scheme"], 1.45, case["steps"])
        if case["diag"]:
            return {"u": f.u, "diag": np.array([f.energy(), 0.5 * f.h2 * float((f.u + 1.0).sum())])}
        return {"u": f.u}
    if kind == "adaptive":
        f = _one(case, seed, case["n"], case["scheme"], 1.45, case["trials"])
        return {"u": f.u, "stats": {"counts": None, "t": np.array([f.t, f.k_last])}}
    if kind == "ensemble":
        # the members' start and first trial come on top of the launches' trials
        fs = [_one(case, seed + 17 * i, n, c, e, 2 + case["rounds"] * case["launches"]) for i, (n, c, e) in enumerate(_members(case))]
        return {"u": [f.u for f in fs], "stats": {"counts": None, "t": np.array([[f.t, f.k_last] for f in fs])}}
    if kind == "fft":
        x = _fft_input(case, seed)
        X = torch.fft.rfft2(x.double()).transpose(1, 2).contiguous()
        return {"X": X, "y": x.double()}
    p, a, t = _fno_inputs(case, seed)
    w, o = {}, 0
    flat = torch.from_numpy(p).to(a.device).double().requires_grad_(case["train"])
    for name, sh in _fno_shapes():
        size = int(np.prod(sh))
        w[name] = flat[o:o + size].reshape(sh)
        o += size
    if not case["train"]:
        return {"y": _fno_forward(w, a.double())}
    y = _fno_forward(w, a.double())
    loss = (y - t.double()).square().mean()
    loss.backward()
    return {"y": y.detach(), "loss": float(loss.detach()), "grads": flat.grad.cpu().numpy()}
