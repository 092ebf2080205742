"""Timed cases of the crossbar solver, each one a call a user's program makes.

A case is a dict of plain values.  Its ``kind`` names the call:

* ``solve``   ``Solver.solve``: node voltages and output currents of a handle's crossbars;
* ``batch``   ``Batch.solve_items``: many crossbars of many shapes in one persistent launch;
* ``linear``  ``Solver.gmres_solve``: one Jacobian system of the paper's normalised regime;
* ``check``   ``Solver.residual``: the KCL residual and conductances at given voltages;
* ``warm``    the learned warm start: first Newton step, network, ``Solver.solve_from``;
* ``layer``   one convolution layer of the network in training: forward, weight gradient,
              backward data.

``prepare`` makes what a program holds before the call (handles, inputs, output buffers) on
the GPU; ``run`` is the call; ``exact`` is the same result in 64 bits from plain torch
(Newton's method with conjugate gradients in the Kronecker eigenbasis; the Jacobian is
symmetric positive definite).
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2109_07929_gb300 as mca
from paper_2109_07929_gb300 import cnn

DEV = "cuda"
F64 = torch.float64

PRECISIONS = {"split": mca.PREC_BF16_SPLIT, "fp64": mca.PREC_FP64, "mhat": mca.PREC_MHAT}
NEG_RATIO = 0.35          # a2 / a1 of the Yakopcic-form devices
BATCH_SIZES = (64, 128, 256, 512)


def _solve(name=None, rows=0, cols=0, vectors=1, maps=1, precision="split", rtol=1e-8,
           g="loguniform", device="sinh", host=False, g_wire_bot=1.0):
    c = dict(kind="solve", rows=rows, cols=cols, vectors=vectors, maps=maps,
             precision=precision, rtol=rtol, g=g, device=device, host=host,
             g_wire_bot=g_wire_bot)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one small array from host memory, as in an interactive design loop
        _solve("solve_32_host", 32, 32, 1, rtol=1e-10, host=True),
        # a programmed (bimodal) weight array: eight crossbars with one input each
        _solve("solve_256_bimodal", 256, 256, 8, maps=8, g="bimodal"),
        # the throughput workload: large crossbars, many inputs interleaved over four maps
        _solve("solve_1024", 1024, 1024, 16, maps=4, g_wire_bot=0.5),
        # the largest arrays
        _solve("solve_2048", 2048, 2048, 4, maps=4, g_wire_bot=0.5),
        # sizes that fill no tile, asymmetric devices driven with both polarities
        _solve("solve_ragged_yakopcic", 1100, 640, 4, device="yakopcic"),
        # statistical characterisation: crossbars of many shapes, 16 inputs each, one launch
        dict(name="batch_mix", kind="batch", crossbars=64, vectors=16, mix=1000, largest=512),
        # every step in FP64, for users who do not want a mixed-precision preconditioner
        _solve("solve_512_fp64", 512, 512, 4, maps=4, precision="fp64"),
        # the paper's own preconditioner (tridiagonal solves)
        _solve("solve_1024_mhat", 1024, 1024, 4, maps=4, precision="mhat", g_wire_bot=0.5),
        # one linear system of the paper's Table 1 (normalised regime, relative residual 1e-6)
        dict(name="linear_512", kind="linear", rows=512, cols=512, vectors=1, rtol=1e-6,
             precision="split"),
        # voltages from elsewhere checked against Kirchhoff's law
        dict(name="check_1024", kind="check", rows=1024, cols=1024, vectors=8),
        # the learned warm start at its training size
        dict(name="warm_256", kind="warm", size=256, vectors=8),
        # a middle layer of the network at the training batch
        dict(name="layer_256", kind="layer", size=256, images=32, dilation=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _capped(rng, rows, cols, hi, budget):
    """Input vectors for rows x cols, at most ``hi``, within ``budget`` units of
    m n (m + n) work."""
    most = int(budget / (rows * cols * (rows + cols)))
    return max(1, min(hi, _log_int(rng, 1, max(1, min(hi, most)))))


def draw(rng: random.Random):
    kind = rng.choice(["solve"] * 5 + ["fp64", "mhat", "batch", "linear", "check", "warm",
                                       "layer"])
    if kind in ("solve", "fp64", "mhat"):
        hi = {"solve": 2048, "fp64": 512, "mhat": 1024}[kind]
        rows, cols = _log_int(rng, 16, hi), _log_int(rng, 16, hi)
        budget = {"solve": 16 * 2 * 1024 ** 3, "fp64": 4 * 2 * 512 ** 3,
                  "mhat": 4 * 2 * 1024 ** 3}[kind]
        v = _capped(rng, rows, cols, 64, budget)
        c = _solve(rows=rows, cols=cols, vectors=v, maps=rng.randint(1, min(v, 8)),
                   precision="split" if kind == "solve" else kind,
                   g=rng.choice(["loguniform", "loguniform", "bimodal"]),
                   device=rng.choice(["sinh", "sinh", "yakopcic"]),
                   host=rng.random() < 0.25, g_wire_bot=rng.choice([1.0, 0.5]))
        return c
    if kind == "batch":
        return dict(kind="batch", crossbars=rng.randint(8, 64), vectors=rng.randint(4, 16),
                    mix=rng.randrange(1 << 20), largest=rng.choice([128, 256, 512]))
    if kind == "linear":
        rows, cols = _log_int(rng, 32, 768), _log_int(rng, 32, 768)
        return dict(kind="linear", rows=rows, cols=cols, vectors=rng.randint(1, 4), rtol=1e-6,
                    precision="split")
    if kind == "check":
        rows, cols = _log_int(rng, 32, 1400), _log_int(rng, 32, 1400)
        return dict(kind="check", rows=rows, cols=cols,
                    vectors=_capped(rng, rows, cols, 8, 8 * 2 * 1024 ** 3))
    if kind == "warm":
        size = _log_int(rng, 64, 320)
        return dict(kind="warm", size=size, vectors=rng.randint(1, 6))
    size = _log_int(rng, 48, 256)
    return dict(kind="layer", size=size, images=rng.randint(1, 32),
                dilation=rng.choice([1, 2, 4, 8, 16, 32]))


# ---- inputs ---------------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) & 0x7FFFFFFF)


def _uniform(gen, shape, lo, hi):
    return torch.rand(shape, generator=gen, device=DEV, dtype=F64) * (hi - lo) + lo


def _gmaps(gen, shape, dist):
    if dist == "bimodal":     # 10 % at 1e-4 S, the rest at 1e-6 S, lognormal spread 0.1
        on = torch.rand(shape, generator=gen, device=DEV) < 0.1
        spread = torch.randn(shape, generator=gen, device=DEV, dtype=F64)
        return torch.where(on, 1e-4, 1e-6).to(F64) * torch.exp(0.1 * spread)
    if dist == "normalised":  # the paper's regime: linear devices up to 0.4, wires 1
        return _uniform(gen, shape, 1e-3, 0.4)
    return torch.pow(10.0, _uniform(gen, shape, -6.0, -4.0))


def _circuit(rows, cols, device="sinh", g_wire_bot=1.0, normalised=False):
    if normalised:
        return dict(rows=rows, cols=cols, gt=1.0, gb=1.0, src=1.0, tr=1.0, bt=1.0, sense=1.0,
                    b=0.0, neg=1.0)
    return dict(rows=rows, cols=cols, gt=1.0, gb=g_wire_bot, src=0.1, tr=1e-3, bt=1e-3,
                sense=0.1, b=2.0, neg=NEG_RATIO if device == "yakopcic" else 1.0)


def _params(q, **kw):
    return mca.default_params(
        q["rows"], q["cols"], g_wire_top=q["gt"], g_wire_bot=q["gb"], g_src=q["src"],
        g_term_top_right=q["tr"], g_term_bot_top=q["bt"], g_sense=q["sense"], b=q["b"],
        neg_ratio=q["neg"],
        device_model=mca.DEVICE_YAKOPCIC if q["neg"] != 1.0 else mca.DEVICE_SINH, **kw)


def _solve_inputs(c, seed):
    gen = _gen(seed)
    g = _gmaps(gen, (c["maps"], c["rows"], c["cols"]), c["g"])
    lo = -0.3 if c["device"] == "yakopcic" else 0.0
    vin = _uniform(gen, (c["vectors"], c["rows"]), lo, 0.3)
    return _circuit(c["rows"], c["cols"], c["device"], c["g_wire_bot"]), g, vin


def _batch_inputs(c, seed):
    """(rows, cols) -> (gmaps, vin, map of each vector) of the crossbars of that shape."""
    rng = random.Random(c["mix"])
    sizes = [s for s in BATCH_SIZES if s <= c["largest"]]
    count = {}
    for _ in range(c["crossbars"]):
        shape = (rng.choice(sizes), rng.choice(sizes))
        count[shape] = count.get(shape, 0) + 1
    gen, groups = _gen(seed), {}
    for (m, n), k in sorted(count.items()):
        g = _gmaps(gen, (k, m, n), "loguniform")
        g = g * torch.exp(0.1 * torch.randn(g.shape, generator=gen, device=DEV, dtype=F64))
        vin = _uniform(gen, (k * c["vectors"], m), 0.0, 0.3)
        groups[(m, n)] = (g, vin, np.repeat(np.arange(k, dtype=np.int32), c["vectors"]))
    return groups


def _linear_inputs(c, seed):
    gen = _gen(seed)
    m, n = c["rows"], c["cols"]
    g = _gmaps(gen, (m, n), "normalised")
    vin = _uniform(gen, (c["vectors"], m), 0.0, 0.3)
    # the first Newton system: J(0) x = Y, D = g
    rhs = torch.zeros(c["vectors"], 2, m, n, dtype=F64, device=DEV)
    rhs[:, 0, :, 0] = vin
    D = g.reshape(1, m * n).expand(c["vectors"], -1).contiguous()
    return _circuit(m, n, normalised=True), g, D, rhs.reshape(c["vectors"], -1)


def _check_inputs(c, seed):
    gen = _gen(seed)
    m, n, v = c["rows"], c["cols"], c["vectors"]
    q = _circuit(m, n, g_wire_bot=0.5)
    g = _gmaps(gen, (m, n), "loguniform")
    vin = _uniform(gen, (v, m), 0.0, 0.3)
    # voltages as they fall along the wires, with some error of their own
    fall = torch.linspace(1.0, 0.8, n, device=DEV, dtype=F64)
    x = torch.empty(v, 2, m, n, dtype=F64, device=DEV)
    x[:, 0] = vin[:, :, None] * fall
    x[:, 1] = 0.05 * torch.linspace(1.0, 0.1, m, device=DEV, dtype=F64)[None, :, None]
    x += 1e-3 * torch.randn(x.shape, generator=gen, device=DEV, dtype=F64)
    return q, g, vin, x.reshape(v, -1)


def _warm_inputs(c, seed):
    gen = _gen(seed)
    s, v = c["size"], c["vectors"]
    return (_circuit(s, s), _gmaps(gen, (v, s, s), "loguniform"),
            _uniform(gen, (v, s), 0.0, 0.3))


def _bf16(x):
    return x.to(torch.bfloat16)


def _layer_inputs(c, seed):
    gen = _gen(seed)
    shape = (c["images"], c["size"], c["size"], cnn.C)
    x = torch.randn(shape, generator=gen, device=DEV)
    x = _bf16(torch.where(x > 0, x, 0.1 * x))           # activations of the layer below
    gz = _bf16(1e-4 * torch.randn(shape, generator=gen, device=DEV))
    taps = cnn.KSIZE * cnn.KSIZE
    w = torch.randn((cnn.C, cnn.C, cnn.KSIZE, cnn.KSIZE), generator=gen, device=DEV)
    return x, gz, w * math.sqrt(2.0 / (cnn.C * taps)), 0.1 * torch.randn(cnn.C, generator=gen,
                                                                         device=DEV)


# ---- prepare and run ------------------------------------------------------------------------

def _zeros(*shape, dtype=F64):
    return torch.zeros(*shape, dtype=dtype, device=DEV)


def _prepare_solve(c, seed):
    q, g, vin = _solve_inputs(c, seed)
    v, m, n = c["vectors"], c["rows"], c["cols"]
    solver = mca.Solver(_params(q, precision=PRECISIONS[c["precision"]], max_batch=min(v, 64),
                                newton_rtol=c["rtol"]), g)
    st = dict(solver=solver, map=np.arange(v, dtype=np.int32) % c["maps"])
    if c["host"]:
        st["vin"], st["out"] = vin.cpu().numpy(), (None, None, None)
    else:
        st["vin"], st["out"] = vin, (_zeros(v, m, n), _zeros(v, m, n), _zeros(v, n))
    return st


def _run_solve(st):
    return st["solver"].solve(st["vin"], *st["out"], map_index=st["map"])[:3]


def _prepare_batch(c, seed):
    groups = _batch_inputs(c, seed)
    solvers, outs, rows = [], [], []
    for k, ((m, n), (g, vin, maps)) in enumerate(groups.items()):
        q = _circuit(m, n)
        solvers.append(mca.Solver(_params(q, gmres_restart=16, max_batch=1, flags=0), g))
        v = vin.shape[0]
        outs.append((_zeros(v, m, n), _zeros(v, m, n), _zeros(v, n)))
        rows += [(k, int(maps[r]), vin[r], outs[k][0][r], outs[k][1][r], outs[k][2][r])
                 for r in range(v)]
    items = mca.Batch.items(*zip(*rows))
    return dict(batch=mca.Batch(solvers), items=items, outs=outs,
                keep=[vin for _, vin, _ in groups.values()])


def _run_batch(st):
    st["batch"].solve_items(st["items"])
    return st["outs"]


def _prepare_linear(c, seed):
    q, g, D, rhs = _linear_inputs(c, seed)
    v = c["vectors"]
    solver = mca.Solver(_params(q, precision=PRECISIONS[c["precision"]], max_batch=v), g)
    a = D.mean(dim=1).cpu().numpy()
    return dict(solver=solver, D=D, a=a, rhs=rhs, dx=_zeros(v, rhs.shape[1]), rtol=c["rtol"])


def _run_linear(st):
    st["solver"].gmres_solve(st["D"], st["a"], st["rhs"], st["dx"], st["rtol"], max_iters=300)
    return st["dx"]


def _prepare_check(c, seed):
    q, g, vin, x = _check_inputs(c, seed)
    v, mn = c["vectors"], c["rows"] * c["cols"]
    return dict(solver=mca.Solver(_params(q, max_batch=v), g), vin=vin, x=x,
                F=_zeros(v, 2 * mn), D=_zeros(v, mn))


def _run_check(st):
    norm, _ = st["solver"].residual(st["x"], st["vin"], st["F"], st["D"])
    return st["F"], st["D"], norm


def _prepare_warm(c, seed):
    q, g, vin = _warm_inputs(c, seed)
    s, v = c["size"], c["vectors"]
    maps = np.arange(v, dtype=np.int32)
    return dict(lin=mca.Solver(_params(q, max_newton=1, max_batch=v), g),
                full=mca.Solver(_params(q, max_batch=v), g), net=cnn.WarmStartCNN().load(),
                g=g, vin=vin, map=maps, map_dev=torch.as_tensor(maps, device=DEV), size=s,
                vlin=(_zeros(v, s, s), _zeros(v, s, s)), io=_zeros(v, s),
                out=(_zeros(v, s, s), _zeros(v, s, s)))


def _run_warm(st):
    net, s, v = st["net"], st["size"], st["vin"].shape[0]
    vlt, vlb = st["vlin"]
    st["lin"].solve(st["vin"], vlt, vlb, st["io"], map_index=st["map"], allow_not_converged=True)
    x = net.features(st["g"], st["map_dev"], st["vin"], vlt, vlb, s, s)
    _, pred = net.forward(x, v, s, s)
    guess = net.state(pred, vlt, vlb, s, s)
    vlin = net.state(None, vlt, vlb, s, s)
    vt, vb, io, _ = st["full"].solve_from(st["vin"], guess, *st["out"], st["io"],
                                          map_index=st["map"], fallback=vlin)
    return vt, vb, io


def _prepare_layer(c, seed):
    x, gz, w, bias = _layer_inputs(c, seed)
    n, s, taps = c["images"], c["size"], cnn.KSIZE * cnn.KSIZE
    lib = mca.load()
    wf = torch.empty(taps, cnn.C, cnn.C, dtype=torch.int16, device=DEV)
    wb = torch.empty_like(wf)
    if lib.mca_cnn_prep_weights(w.data_ptr(), cnn.C, cnn.C, cnn.KSIZE, cnn.C, wf.data_ptr(),
                                wb.data_ptr(), None):
        raise RuntimeError("mca_cnn_prep_weights")
    scratch = torch.empty(int(lib.mca_cnn_wgrad_scratch(n, s, s, cnn.KSIZE)),
                          dtype=torch.float32, device=DEV)
    return dict(lib=lib, x=x, gz=gz, wf=wf, wb=wb, bias=bias, scratch=scratch, n=n, s=s,
                d=c["dilation"], out=torch.empty_like(x), gx=torch.empty_like(x),
                gw=torch.empty_like(w), gb=torch.empty_like(bias))


def _run_layer(st):
    lib, n, s, d, k, ch = st["lib"], st["n"], st["s"], st["d"], cnn.KSIZE, cnn.C
    p = {key: st[key].data_ptr() for key in ("x", "gz", "wf", "wb", "bias", "scratch", "out",
                                             "gx", "gw", "gb")}
    rc = [lib.mca_cnn_conv(p["x"], n, s, s, p["wf"], k, d, ch, ch, p["bias"], 1, 0, None,
                           p["out"], None, None),
          lib.mca_cnn_conv_wgrad(p["x"], p["gz"], n, s, s, k, d, ch, ch, p["scratch"], p["gw"],
                                 p["gb"], None),
          lib.mca_cnn_conv(p["gz"], n, s, s, p["wb"], k, d, ch, ch, None, 1, 1, p["x"], p["gx"],
                           None, None)]
    if any(rc):
        raise RuntimeError(f"layer: {rc}")
    return st["out"], st["gw"], st["gb"], st["gx"]


def prepare(case, seed):
    st = {"solve": _prepare_solve, "batch": _prepare_batch, "linear": _prepare_linear,
          "check": _prepare_check, "warm": _prepare_warm,
          "layer": _prepare_layer}[case["kind"]](case, seed)
    st["run"] = case["kind"]
    return st


def run(state):
    return {"solve": _run_solve, "batch": _run_batch, "linear": _run_linear,
            "check": _run_check, "warm": _run_warm, "layer": _run_layer}[state["run"]](state)


# ---- work -----------------------------------------------------------------------------------

def _solve_work(m, n, vectors, maps, applies, outputs=True):
    """Inputs and outputs once; ``applies`` preconditioner applies of 8 m n (m + n) FLOPs per
    vector (what the eigenbasis transforms of two Newton steps take)."""
    return (8.0 * (maps * m * n + vectors * m + (vectors * (2 * m * n + n) if outputs else 0)),
            applies * 8.0 * m * n * (m + n) * vectors)


def work(case):
    kind = case["kind"]
    if kind == "solve":
        m, n, v = case["rows"], case["cols"], case["vectors"]
        by, fl = _solve_work(m, n, v, case["maps"], 6)
        if case["precision"] == "mhat":       # tridiagonal solves and stencils: O(m n)
            fl = 15 * 60.0 * m * n * v
    elif kind == "batch":
        rng, by, fl = random.Random(case["mix"]), 0.0, 0.0
        sizes = [s for s in BATCH_SIZES if s <= case["largest"]]
        for _ in range(case["crossbars"]):
            b1, f1 = _solve_work(rng.choice(sizes), rng.choice(sizes), case["vectors"], 1, 6)
            by, fl = by + b1, fl + f1
    elif kind == "linear":
        m, n, v = case["rows"], case["cols"], case["vectors"]
        by, fl = 8.0 * v * (m * n + 4 * m * n), 9 * 8.0 * m * n * (m + n) * v
    elif kind == "check":
        mn, v = case["rows"] * case["cols"], case["vectors"]
        by, fl = 8.0 * (mn + v * 5 * mn), 40.0 * mn * v
    elif kind == "warm":
        m = case["size"]
        by, fl = _solve_work(m, m, case["vectors"], case["vectors"], 6)
        chans = sum(cin * cout for cin, cout, _, _ in cnn.LAYERS)
        fl += 2.0 * chans * cnn.KSIZE ** 2 * m * m * case["vectors"]
    else:
        pix = case["images"] * case["size"] ** 2
        by = pix * cnn.C * 2.0 * 4 + 4.0 * 3 * cnn.C * cnn.C * cnn.KSIZE ** 2
        fl = 3 * 2.0 * pix * cnn.C * cnn.C * cnn.KSIZE ** 2
    return {"bytes": by, "flops": fl}


# ---- exact values ---------------------------------------------------------------------------

class _Exact:
    """One crossbar shape in FP64: F, J and P^-1 on states of shape (v, 2, m, n)."""

    def __init__(self, q):
        self.q = q
        self.mu, self.Qr = self._chain(q["cols"], q["gt"], q["src"], q["tr"])
        self.nu, self.Qc = self._chain(q["rows"], q["gb"], q["bt"], q["sense"])

    @staticmethod
    def _ends(n, g, first, last):
        d = torch.full((n,), 2.0 * g, dtype=F64, device=DEV)
        if n == 1:
            d[0] = first + last
        else:
            d[0], d[-1] = first + g, g + last
        return d

    def _chain(self, n, g, first, last):
        off = torch.full((n - 1,), -g, dtype=F64, device=DEV)
        T = torch.diag(self._ends(n, g, first, last)) + torch.diag(off, 1) + torch.diag(off, -1)
        return torch.linalg.eigh(T)

    def wires(self, x):
        q = self.q
        dt = self._ends(q["cols"], q["gt"], q["src"], q["tr"])
        db = self._ends(q["rows"], q["gb"], q["bt"], q["sense"])
        t, b = x[:, 0], x[:, 1]
        y = torch.empty_like(x)
        y[:, 0] = dt * t
        y[:, 0, :, 1:] -= q["gt"] * t[:, :, :-1]
        y[:, 0, :, :-1] -= q["gt"] * t[:, :, 1:]
        y[:, 1] = db[:, None] * b
        y[:, 1, 1:] -= q["gb"] * b[:, :-1]
        y[:, 1, :-1] -= q["gb"] * b[:, 1:]
        return y

    def device(self, g, dv):
        b = self.q["b"]
        i, D = (g * dv, g.expand_as(dv)) if b == 0.0 else (g / b * torch.sinh(b * dv),
                                                           g * torch.cosh(b * dv))
        if self.q["neg"] != 1.0:
            f = torch.where(dv < 0, self.q["neg"], 1.0)
            i, D = i * f, D * f
        return i, D

    def residual(self, g, vin, x):
        i, D = self.device(g, x[:, 0] - x[:, 1])
        F = self.wires(x)
        F[:, 0] += i
        F[:, 1] -= i
        F[:, 0, :, 0] -= self.q["src"] * vin
        return F, D

    def apply_p(self, a, r):
        """P^-1 r, per-mode 2 x 2 blocks with a1 = a2 = a (v values)."""
        h = self.Qc.T @ r @ self.Qr
        a = a[:, None, None]
        M, N = self.mu[None, None, :], self.nu[None, :, None]
        det = M * N + a * (M + N)
        t = ((N + a) * h[:, 0] + a * h[:, 1]) / det
        b = (a * h[:, 0] + (M + a) * h[:, 1]) / det
        return self.Qc @ torch.stack((t, b), 1) @ self.Qr.T

    def linear(self, D, rhs, rtol, most=60):
        """J dx = rhs by preconditioned conjugate gradients, every vector to rtol."""
        def J(z):
            w = self.wires(z)
            c = D * (z[:, 0] - z[:, 1])
            w[:, 0] += c
            w[:, 1] -= c
            return w

        def dot(p, q):
            return (p * q).sum(dim=(1, 2, 3))

        def col(s):
            return s[:, None, None, None]

        a = D.mean(dim=(1, 2))
        x, r = torch.zeros_like(rhs), rhs.clone()
        stop = rtol * dot(rhs, rhs).sqrt()
        z = self.apply_p(a, r)
        p, rz = z, dot(r, z)
        for _ in range(most):
            Jp = J(p)
            al = rz / dot(p, Jp).clamp_min(1e-300)
            x, r = x + col(al) * p, r - col(al) * Jp
            if bool((dot(r, r).sqrt() <= stop).all()):
                break
            z = self.apply_p(a, r)
            new = dot(r, z)
            p, rz = z + col(new / rz.clamp_min(1e-300)) * p, new
        return x

    def newton(self, g, vin):
        """(V_t, V_b, I_out) of every vector; g: (v, m, n)."""
        q = self.q
        x = torch.zeros(vin.shape[0], 2, q["rows"], q["cols"], dtype=F64, device=DEV)
        y = q["src"] * vin.norm(dim=1)
        for _ in range(12):
            F, D = self.residual(g, vin, x)
            rel = float((F.flatten(1).norm(dim=1) / y).max())
            if rel <= 2e-14:
                break
            x = x + self.linear(D, -F, max(1e-6 if rel < 1e-2 else 1e-4, 1e-14 / rel))
            if rel <= 1e-9:
                break
        return x[:, 0], x[:, 1], q["sense"] * x[:, 1, -1, :]


def _too_slow(m, n, v):
    return 20 * 8.0 * m * n * (m + n) * v > 1.2e13


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        if _too_slow(case["rows"], case["cols"], case["vectors"]):
            return None
        q, g, vin = _solve_inputs(case, seed)
        maps = torch.arange(vin.shape[0], device=DEV) % case["maps"]
        return _Exact(q).newton(g[maps], vin)
    if kind == "batch":
        groups = _batch_inputs(case, seed)
        if sum(20 * 8.0 * m * n * (m + n) * vin.shape[0]
               for (m, n), (_, vin, _) in groups.items()) > 1.2e13:
            return None
        return [_Exact(_circuit(m, n)).newton(g[torch.as_tensor(maps, device=DEV).long()], vin)
                for (m, n), (g, vin, maps) in groups.items()]
    if kind == "linear":
        q, g, D, rhs = _linear_inputs(case, seed)
        v, m, n = case["vectors"], case["rows"], case["cols"]
        x = _Exact(q).linear(D.reshape(v, m, n), rhs.reshape(v, 2, m, n), 1e-14, 80)
        return x.reshape(v, -1)
    if kind == "check":
        q, g, vin, x = _check_inputs(case, seed)
        v, m, n = case["vectors"], case["rows"], case["cols"]
        F, D = _Exact(q).residual(g, vin, x.reshape(v, 2, m, n))
        return F.reshape(v, -1), D.reshape(v, -1), F.flatten(1).norm(dim=1).cpu().numpy()
    if kind == "warm":
        q, g, vin = _warm_inputs(case, seed)
        return _Exact(q).newton(g, vin)
    return _exact_layer(case, seed)


def _exact_layer(case, seed):
    x, gz, w, bias = _layer_inputs(case, seed)
    K, d, s = cnn.KSIZE, case["dilation"], case["size"]
    w = _bf16(w).to(F64)                         # the operands the tensor cores multiply
    pad = d * (K // 2)
    out = torch.zeros(x.shape, dtype=F64, device=DEV)
    gx = torch.zeros_like(out)
    gw = torch.zeros_like(w)
    for im in range(x.shape[0]):
        xi, gi = x[im].to(F64), gz[im].to(F64)
        xp = torch.nn.functional.pad(xi, (0, 0, pad, pad, pad, pad))
        gp = torch.nn.functional.pad(gi, (0, 0, pad, pad, pad, pad))
        for ky in range(K):
            for kx in range(K):
                win = (slice(ky * d, ky * d + s), slice(kx * d, kx * d + s))
                out[im] += xp[win] @ w[:, :, ky, kx].T
                gw[:, :, ky, kx] += gi.reshape(-1, cnn.C).T @ xp[win].reshape(-1, cnn.C)
                gx[im] += gp[win] @ w[:, :, K - 1 - ky, K - 1 - kx]
    out += bias.to(F64)
    return (torch.where(out > 0, out, 0.1 * out), gw, gz.to(F64).sum(dim=(0, 1, 2)),
            torch.where(x.to(F64) > 0, gx, 0.1 * gx))
