"""The workloads whose speed is followed: what a user of the library has it do, through its
public entry points, on the sizes of its tests, its benchmark and its example problems.

A case is a dict of plain values; `prepare` makes the solver handle and the inputs on the GPU,
`run` is one pass, `exact` the same result in 64 bits from plain torch and numpy.

Kinds of pass
  pi     one application of the MFWH map (the unit every iteration is made of)
  fpi    a fixed-point iteration (Algorithm 1)
  gmres  one restart cycle of GMRES on (I - S) V = Pi(0), from zero, with its residual check
  batch  independent problems of uneven size solved in lockstep, one graph launch per map
  cnn    one training step of the warm-start network, then a prediction with the new weights
"""

import math

import numpy as np
import torch

import paper_2507_23613_gb300 as mfwh
from paper_2507_23613_gb300 import _lib

PRECISION = {"fp64": _lib.PREC_FP64, "fp32_kahan": _lib.PREC_FP32_KAHAN,
             "fp32_blocksum": _lib.PREC_FP32_BLOCKSUM}
FILTER = {"optimized": _lib.FILTER_OPTIMIZED, "traditional": _lib.FILTER_TRADITIONAL}


def _problem(name, nx, ny, nf, w_lo, w_hi, kind="pi", nz=0, ly=1.0, lz=1.0, precision="fp64",
             n_p=1, filter_mode="optimized", forced=False, order=2, stepping="explicit",
             time_block=0, c_hi=0.0, layer_axis=2, omega_seed=1, iters=1):
    """One wave problem: nx x ny (x nz) cells on [0, 1] x [0, ly] (x [0, lz]), nf frequencies
    spread over [w_lo, w_hi]; c_hi > 0: two layers of wave speed 1 and c_hi, split in the middle
    of axis layer_axis."""
    return dict(name=name, kind=kind, nx=nx, ny=ny, nz=nz, ly=ly, lz=lz, nf=nf, w_lo=w_lo,
                w_hi=w_hi, precision=precision, n_p=n_p, filter_mode=filter_mode, forced=forced,
                order=order, stepping=stepping, time_block=time_block, c_hi=c_hi,
                layer_axis=layer_axis, omega_seed=omega_seed, iters=iters)


def listed():
    return [
        # the smallest standard problem, 65^2 with two frequencies, solved by Algorithm 1: 40
        # short wave solves on a grid of one or two tiles, where launches and latency count
        _problem("fpi_square65", 64, 64, 2, 5.0, 10.0, kind="fpi", iters=40),
        # one Krylov cycle of the 513^2, six-frequency problems of the warm-start study: forced
        # and homogeneous wave solves, Gram-Schmidt, the residual check
        _problem("gmres_square513", 512, 512, 6, 15.0, 45.0, kind="gmres", n_p=2, iters=20),
        # the benchmark's grid: the homogeneous map that every Arnoldi step applies
        _problem("pi_square1025", 1024, 1024, 8, 10.0, 60.0, n_p=2),
        # an odd rectangle with unequal spacings, two wave speeds and more than 8 frequencies
        _problem("pi_rect_layers", 771, 530, 11, 8.0, 60.0, n_p=2, filter_mode="traditional",
                 forced=True, c_hi=1.5, layer_axis=1),
        # 3D in 64 bits, two layers: the FP64 products and residuals of the cube problems
        _problem("pi_cube129", 128, 128, 4, 8.0, 30.0, nz=128, c_hi=1.5),
        # the paper's three-frequency example with the fourth-order operator, 513^2
        _problem("pi_order4_513", 512, 512, 3, 5.0, 15.0, n_p=2, order=4),
        # the largest 2D grid of the batch workload, in FP32 wave steps
        _problem("pi32_square2049", 2048, 2048, 5, 20.0, 60.0, precision="fp32_blocksum"),
        # FP32 with Kahan sums at every step on an odd rectangle, many frequencies, forced
        _problem("pi32_kahan_rect", 611, 402, 12, 10.0, 70.0, ly=0.66, precision="fp32_kahan",
                 n_p=2, filter_mode="traditional", forced=True),
        # the 257^3 two-layer cube, FP32 wave steps at the autotuner's depth
        _problem("pi32_cube257", 256, 256, 4, 8.0, 30.0, nz=256, precision="fp32_blocksum",
                 c_hi=1.5, time_block=4),
        # uneven problems in lockstep: the batched workload, a few Arnoldi steps
        dict(name="batch_lockstep", kind="batch", problems=6, max_cells=1024, seed=3, iters=4),
        # implicit trapezoidal steps with multigrid solves
        _problem("pi_implicit_513", 512, 512, 6, 10.0, 45.0, stepping="implicit", n_p=2),
        # the warm-start network: training batch of 48 images of 129^2, then a prediction
        dict(name="cnn_train_129", kind="cnn", batch=48, height=129, width=129, layers=5,
             channels=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    most = max(work(c)["flops"] for c in listed())
    while True:
        case = _draw(rng)
        if work(case)["flops"] <= most:
            return case


def _draw(rng):
    kind = rng.choice(["fpi", "gmres", "pi64", "pi64", "pi64_3d", "order4", "pi32", "pi32",
                       "pi32_3d", "batch", "implicit", "cnn"])
    seed = rng.randrange(1, 10**6)
    if kind == "cnn":
        return dict(kind="cnn", batch=rng.randrange(8, 65), height=rng.randrange(65, 145),
                    width=rng.randrange(65, 145), layers=rng.choice([3, 4, 5]),
                    channels=rng.choice([16, 24, 32]))
    if kind == "batch":
        return dict(kind="batch", problems=rng.randrange(3, 8), max_cells=1024,
                    seed=seed, iters=rng.randrange(2, 5))
    nf = rng.randrange(1, 17) if kind in ("pi64", "pi32") else rng.randrange(1, 7)
    # many frequencies want two periods of the longest one, as the benchmark takes
    n_p = 2 if nf > 4 else rng.choice([1, 2])
    w_lo = rng.uniform(6.0, 12.0) * n_p
    layers = rng.random() < 0.4
    common = dict(w_lo=w_lo, n_p=n_p, omega_seed=seed, c_hi=1.5 if layers else 0.0,
                  forced=rng.random() < 0.3)
    if kind == "pi64_3d" or kind == "pi32_3d":
        n = [_log_int(rng, 24, 160) for _ in range(3)]
        p = _problem("", n[0], n[1], nf, w_hi=w_lo + 5.0 * nf + 6.0, nz=n[2],
                     ly=n[1] / n[0], lz=n[2] / n[0], filter_mode="traditional",
                     layer_axis=rng.randrange(3), **common)
        if kind == "pi32_3d":
            p["precision"] = rng.choice(["fp32_kahan", "fp32_blocksum"])
            p["time_block"] = rng.choice([0, 2, 4])
    elif kind == "implicit":
        nx, ny = 2 ** rng.randrange(7, 10), 2 ** rng.randrange(7, 10)
        common.update(c_hi=0.0)
        p = _problem("", nx, ny, nf, w_hi=w_lo + 35.0, ly=ny / nx,
                     stepping="implicit", filter_mode="traditional", **common)
    else:
        top = {"fpi": 200, "gmres": 400, "pi64": 1100, "order4": 600, "pi32": 1600}[kind]
        low = {"fpi": 32, "gmres": 64, "pi64": 100, "order4": 100, "pi32": 100}[kind]
        nx, ny = _log_int(rng, low, top), _log_int(rng, low, top)
        p = _problem("", nx, ny, nf, w_hi=w_lo + 5.0 * nf + 6.0,
                     ly=rng.choice([1.0, ny / nx]), filter_mode="traditional",
                     layer_axis=rng.randrange(2), **common)
        if kind == "pi32":
            p["precision"] = rng.choice(["fp32_kahan", "fp32_blocksum"])
        if kind == "order4":
            p["order"] = 4
        if kind == "fpi":
            p.update(kind="fpi", iters=rng.randrange(5, 21))
        if kind == "gmres":
            p.update(kind="gmres", iters=rng.randrange(5, 13))
    del p["name"]
    return p


# ---- inputs ----------------------------------------------------------------------------------

def _omega(case):
    """nf frequencies in [w_lo, w_hi], one in the lower half of each of nf equal cells, so that
    neighbours stay apart (the spread that the filters are designed for)."""
    u = np.random.default_rng(case["omega_seed"]).uniform(0.0, 0.5, case["nf"])
    return case["w_lo"] + (np.arange(case["nf"]) + u) * (case["w_hi"] - case["w_lo"]) / case["nf"]


def _cells(case):
    return (case["nx"], case["ny"]) + ((case["nz"],) if case["nz"] else ())


def _length(case):
    return (1.0, case["ly"]) + ((case["lz"],) if case["nz"] else ())


def _axes(case):
    """Coordinates along each axis, x first, on the GPU."""
    return [torch.arange(n + 1, dtype=torch.float64, device="cuda") * (L / n)
            for n, L in zip(_cells(case), _length(case))]


def _separable(factors):
    """The product of one function per axis (x first) on the grid, x fastest."""
    out = factors[-1]
    for f in reversed(factors[:-1]):
        out = out.unsqueeze(-1) * f
    return out


def _forcing(case, omega, seed):
    """One to four Gaussian sources exp(-b |x - x0|^2) per frequency."""
    rng = np.random.default_rng([seed, 11])
    axes = _axes(case)
    b = rng.uniform(200.0, 400.0)
    fs = []
    for _ in omega:
        f = 0.0
        for _ in range(int(rng.integers(1, 5))):
            f = f + _separable([torch.exp(-b * (x - rng.uniform(0.2, 0.8) * L) ** 2)
                                for x, L in zip(axes, _length(case))])
        fs.append(f)
    return torch.stack(fs).contiguous()


def _iterate(case, omega, seed):
    """An iterate as the solvers meet it: per frequency a sum of standing waves of about that
    wavenumber with random amplitudes, 0 on the boundary."""
    rng = np.random.default_rng([seed, 12])
    axes = _axes(case)
    vs = []
    for w in omega:
        v = 0.0
        for _ in range(6):
            d = rng.normal(size=len(axes))
            d /= np.linalg.norm(d)
            fac = []
            for x, L, n, c in zip(axes, _length(case), _cells(case), d):
                k = min(max(1, round(w * abs(c) * L / math.pi)), n - 1)
                s = torch.sin(k * math.pi / L * x)
                s[-1] = 0.0
                fac.append(s)
            fac[0] = fac[0] * (rng.normal() * 0.02)
            v = v + _separable(fac)
        vs.append(v)
    return torch.stack(vs).contiguous()


def _solver(case, omega, forcing):
    kw = {}
    if case["c_hi"]:
        kw = dict(c_lo=1.0, c_hi=case["c_hi"], layer_axis=case["layer_axis"],
                  interface=0.5 * _length(case)[case["layer_axis"]])
    return mfwh.Solver(_cells(case), _length(case), omega, forcing, n_p=case["n_p"],
                       filter_mode=FILTER[case["filter_mode"]], order=case["order"],
                       precision=PRECISION[case["precision"]], time_block=case["time_block"],
                       time_stepping=case["stepping"], **kw)


def _batch(case):
    """The problems of a batch: unit squares of 257^2, 513^2 or 1025^2 (uneven), 1 to 8
    frequencies, FP32 wave steps."""
    rng = np.random.default_rng(case["seed"])
    out = []
    for _ in range(case["problems"]):
        n = int(rng.choice([256, 512, min(1024, case["max_cells"])]))
        nf = int(rng.integers(1, 9))
        w_lo = float(rng.uniform(12.0, 20.0))
        out.append(_problem("", n, n, nf, w_lo, w_lo + 4.0 * nf + 6.0, precision="fp32_blocksum",
                            filter_mode="traditional", omega_seed=int(rng.integers(1, 10**6))))
    return out


def _network(case, seed):
    """He-normal weights, a batch of (forcing, frequency) images with their targets, the mask of
    interior points, and a second batch to predict."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    B, H, W, C = case["batch"], case["height"], case["width"], case["channels"]
    chans = [2] + [C] * (case["layers"] - 1) + [1]
    flat = []
    for cin, cout in zip(chans[:-1], chans[1:]):
        w = torch.randn(cout, cin, 3, 3, generator=g, device="cuda") * math.sqrt(2.0 / (9 * cin))
        flat += [w.reshape(-1), torch.zeros(cout, device="cuda")]
    y = torch.arange(H, device="cuda").view(1, H, 1) / (H - 1)
    x = torch.arange(W, device="cuda").view(1, 1, W) / (W - 1)

    def images(count):
        c = torch.rand(count, 2, 1, 1, generator=g, device="cuda") * 0.6 + 0.2
        w = torch.rand(count, 1, 1, generator=g, device="cuda") * 30.0 + 15.0
        f = torch.exp(-300.0 * ((x - c[:, 0]) ** 2 + (y - c[:, 1]) ** 2))
        t = torch.cos(w * torch.sqrt((x - c[:, 0]) ** 2 + (y - c[:, 1]) ** 2))
        return torch.stack([f, (w / 45.0).expand_as(f)], 1).contiguous(), t.contiguous()

    xs, ts = images(B)
    xv, _ = images(max(1, B // 4))
    mask = torch.zeros(H, W, device="cuda")
    mask[1:-1, 1:-1] = 1.0
    return torch.cat(flat), xs, ts, mask, xv, chans


def prepare(case, seed):
    if case["kind"] == "cnn":
        flat, xs, ts, mask, xv, _ = _network(case, seed)
        net = mfwh.CNN(layers=case["layers"], channels=case["channels"])
        net.set_params(flat.cpu().numpy())
        y = torch.empty(xv.shape[0], 1, *xv.shape[2:], device="cuda")
        return dict(case=case, net=net, x=xs, t=ts, mask=mask, xv=xv, y=y)
    if case["kind"] == "batch":
        solvers, vs = [], []
        for i, p in enumerate(_batch(case)):
            om = _omega(p)
            f = _forcing(p, om, seed + 1000 * i)
            solvers.append(_solver(p, om, f))
            vs.append(torch.zeros_like(f))
        return dict(case=case, solvers=solvers, vs=vs)
    om = _omega(case)
    f = _forcing(case, om, seed)
    v = torch.zeros_like(f) if case["kind"] == "gmres" else _iterate(case, om, seed)
    return dict(case=case, solver=_solver(case, om, f), v=v, out=torch.empty_like(v))


def run(state):
    case = state["case"]
    if case["kind"] == "pi":
        state["solver"].apply_Pi(state["v"], state["out"], forced=case["forced"])
        return state["out"]
    if case["kind"] == "fpi":
        state["out"].copy_(state["v"])
        state["solver"].solve_fpi(state["out"], case["iters"])
        return state["out"]
    if case["kind"] == "gmres":
        state["out"].zero_()
        info = state["solver"].solve_gmres(state["out"], restart=case["iters"], tol=1e-12,
                                           max_iters=case["iters"], raise_on_error=False)
        return dict(v=state["out"], iterations=info["iterations"],
                    history=info["history"], helmholtz=info["helmholtz_residual"])
    if case["kind"] == "batch":
        for v in state["vs"]:
            v.zero_()
        mfwh.solve_batch_graph(state["solvers"], state["vs"], restart=case["iters"], tol=1e-12,
                               max_iters=case["iters"], raise_on_error=False)
        return list(state["vs"])
    loss = state["net"].train_step(state["x"], state["t"], state["mask"], 1e-4)
    state["net"].forward(state["xv"], state["y"])
    params, grads = state["net"].get_params(grads=True)
    return dict(loss=loss, params=params, grads=grads, prediction=state["y"])


# ---- the work of a pass ------------------------------------------------------------------------

def _steps(case):
    """(N_t, dt): steps of one wave solve and the step length."""
    om, h = _omega(case), [L / n for n, L in zip(_cells(case), _length(case))]
    if case["stepping"] == "implicit":
        n_t = math.ceil(10 * case["n_p"] * om[-1] / om[0] - 1e-12)
        c = math.cos(2.0 * math.pi * case["n_p"] / n_t)
        return n_t, math.sqrt(2.0 * (1.0 - c) / c) / om[0]
    limit = 1.0 / (max(1.0, case["c_hi"]) * math.sqrt(sum(1.0 / x ** 2 for x in h)))
    if case["order"] == 4:
        limit *= math.sqrt(3.0) / 2.0
    n_t = max(2 * case["n_p"] + 1, math.ceil(case["n_p"] * 2.0 * math.pi / om[0] / (0.5 * limit)))
    return n_t, 2.0 * math.sin(math.pi * case["n_p"] / n_t) / om[0]


def _map_work(case, forced):
    """One wave solve: per point and step the stencil (2 operations for each of its points but
    the centre, 3 for the rest), an addition and a multiplication per frequency for the filter
    sums and, if forced, for the forcing; the filter solve; the iterate read and written."""
    points, interior = 1, 1
    for n in _cells(case):
        points *= n + 1
        interior *= n - 1
    dim, nf = len(_cells(case)), case["nf"]
    arms = 2 * dim * (1 if case["order"] == 2 else 2)
    n_t, _ = _steps(case)
    flops = interior * (n_t * (arms + 3 + 2 * nf * (2 if forced else 1)) + 2 * nf * nf)
    return 8 * nf * points * (3 if forced else 2), flops


def work(case):
    if case["kind"] == "cnn":
        B, H, W, C, L = (case[k] for k in ("batch", "height", "width", "channels", "layers"))
        macs = 9 * (2 * C + (L - 2) * C * C + C) * H * W
        n = B + B + max(1, B // 4)   # forward, weight gradient, prediction; input gradient below
        params = 9 * (2 * C + (L - 2) * C * C + C) + (L - 1) * C + 1
        return {"bytes": 4 * (H * W * (3 * B + 3 * max(1, B // 4) + 1) + 8 * params),
                "flops": 2 * (macs * n + 9 * ((L - 2) * C * C + C) * H * W * B)}
    if case["kind"] == "batch":
        per = [(_map_work(p, True), _map_work(p, False)) for p in _batch(case)]
        # inputs and outputs once; Pi(0) and one homogeneous map per Arnoldi step
        return {"bytes": sum(f[0] * 2 / 3 for f, _ in per),
                "flops": sum(f[1] + case["iters"] * s[1] for f, s in per)}
    if case["kind"] == "gmres":
        f, s = _map_work(case, True), _map_work(case, False)
        return {"bytes": f[0] * 2 // 3, "flops": f[1] + case["iters"] * s[1]}
    b, f = _map_work(case, case["forced"] or case["kind"] == "fpi")
    return {"bytes": b, "flops": f * case["iters"]}


# ---- the same results in 64 bits ---------------------------------------------------------------

def _filter(case):
    """(dt, omega~, weights w[n][m], B) of the discrete method."""
    om = _omega(case)
    nf, n_p = case["nf"], case["n_p"]
    n_t, dt = _steps(case)
    x2 = (om * dt) ** 2
    wt = np.arccos(1.0 / (1.0 + 0.5 * x2) if case["stepping"] == "implicit" else 1.0 - 0.5 * x2) / dt
    n_pm = np.floor(n_p * wt / wt[0] + 1e-12)
    t_fm = n_pm * 2.0 * math.pi / wt
    t = np.arange(n_t + 1) * dt

    def quadrature(step):
        s = np.zeros((n_t + 1, nf))
        for m in range(nf):
            k = min(int(math.floor(t_fm[m] / step + 1e-9)), n_t)
            r = t_fm[m] / step - k
            s[:k + 1, m] = step
            s[0, m] = s[k, m] = 0.5 * step
            if k < n_t:
                s[k, m] += step * (r - 0.5 * r * r)
                s[k + 1, m] += 0.5 * step * r * r
        return s

    sigma = quadrature(dt)
    if case["filter_mode"] == "traditional":
        par = np.stack([-np.tan(0.5 * wt * dt) / (2.0 * np.tan(wt * dt)), np.ones(nf),
                        np.zeros(nf)], 1)
    else:
        step = t_fm.max() / n_t
        tt = np.arange(n_t + 1) * step
        nu = quadrature(step) * (2.0 / t_fm)
        basis = [nu, nu * np.cos(np.outer(tt, wt)), nu * np.sin(np.outer(tt, wt))]
        a, c, s = (np.cos(np.outer(wt, tt)) @ b for b in basis)
        da, dc, ds = ((-np.sin(np.outer(wt, tt)) * tt) @ b for b in basis)
        G, H = np.block([[c, s], [dc, ds]]), np.vstack([a, da])
        z = np.concatenate([np.ones(nf), np.zeros(nf)])
        delta = wt[-1] / (2.0 * n_pm[-1])
        top = wt[-1] + 2.0 * nf * delta
        count = math.ceil(20 * top / delta - 1e-9)
        lam = (np.arange(count) + 0.5) * top / count
        ca = np.cos(np.outer(lam, tt))
        fa, fcs = ca @ basis[0], np.hstack([ca @ basis[1], ca @ basis[2]])
        xa = np.linalg.lstsq(fa - fcs @ np.linalg.solve(G, H), -(fcs @ np.linalg.solve(G, z)),
                             rcond=None)[0]
        y = np.linalg.solve(G, z - H @ xa)
        par = np.stack([xa, y[:nf], y[nf:]], 1)
    arg = np.outer(t, wt)
    w = 2.0 / t_fm * sigma * (par[:, 0] + par[:, 1] * np.cos(arg) + par[:, 2] * np.sin(arg))
    return dt, wt, w, w.T @ np.cos(arg)


class _Exact:
    """The map of one problem in 64 bits: time stepping with torch on the GPU; the implicit
    scheme in the basis of sine modes, where each step is a division."""

    def __init__(self, case, f):
        self.case, self.f = case, f
        self.omega = _omega(case)
        self.dt, self.wt, self.w, B = _filter(case)
        self.binv = torch.tensor(np.linalg.inv(B), device="cuda")
        self.h = [L / n for n, L in zip(_cells(case), _length(case))]
        self.inner = (Ellipsis,) + (slice(1, -1),) * len(self.h)
        self.c2 = 1.0
        if case["c_hi"]:
            ax = case["layer_axis"]
            x = _axes(case)[ax]
            c2 = torch.where(x < 0.5 * _length(case)[ax], 1.0, case["c_hi"] ** 2)
            self.c2 = c2[1:-1].view([-1] + [1] * ax)

    def lap(self, u):
        """c^2 Delta_h u at the interior points of the stack u, the last axes the grid's."""
        out = 0.0
        dim = len(self.h)
        for a, h in enumerate(self.h):
            d = u.dim() - 1 - a
            v = u[(Ellipsis,) + tuple(slice(None) if u.dim() - 1 - b == d else slice(1, -1)
                                      for b in reversed(range(dim)))]
            n = v.shape[d]
            if self.case["order"] == 4:
                v = torch.cat([-v.narrow(d, 1, 1), v, -v.narrow(d, n - 2, 1)], d)
                out = out + (16.0 * (v.narrow(d, 1, n - 2) + v.narrow(d, 3, n - 2))
                             - v.narrow(d, 0, n - 2) - v.narrow(d, 4, n - 2)
                             - 30.0 * v.narrow(d, 2, n - 2)) / (12.0 * h * h)
            else:
                out = out + (v.narrow(d, 0, n - 2) + v.narrow(d, 2, n - 2)
                             - 2.0 * v.narrow(d, 1, n - 2)) / (h * h)
        return self.c2 * out

    def pi(self, v, forced):
        w = torch.tensor(self.w, device="cuda")
        dt2, n_t = self.dt ** 2, self.w.shape[0] - 1
        cos = np.cos(np.outer(np.arange(n_t + 1) * self.dt, self.wt))
        f = self.f[self.inner]
        u0 = v.sum(0)
        implicit = self.case["stepping"] == "implicit"
        modes = None
        if implicit:
            cos = cos * np.cos(self.wt * self.dt)
            modes = [torch.sin(torch.outer(k, k) * (math.pi / n)) * math.sqrt(2.0 / n)
                     for n in _cells(self.case)
                     for k in [torch.arange(1, n, dtype=torch.float64, device="cuda")]]
            lam = [4.0 / h ** 2 * torch.sin(torch.arange(1, n, dtype=torch.float64, device="cuda")
                                            * math.pi / (2 * n)) ** 2
                   for n, h in zip(_cells(self.case), self.h)]
            solve = 1.0 + 0.5 * dt2 * (lam[1][:, None] + lam[0][None, :])
            f = modes[1] @ f @ modes[0]
            u = modes[1] @ u0[self.inner] @ modes[0]
        else:
            full = torch.zeros_like(u0)
            u = u0[self.inner].clone()
        q = w[0].view([-1] + [1] * u.dim()) * u
        prev, block, first = None, [], 1
        for n in range(n_t):
            F = torch.tensordot(torch.tensor(cos[n], device="cuda"), f, 1) if forced else 0.0
            if implicit:
                new = (u - 0.5 * dt2 * F) / solve if n == 0 else (2 * u - dt2 * F) / solve - prev
            else:
                full[self.inner] = u
                g = self.lap(full) - F
                new = u + 0.5 * dt2 * g if n == 0 else 2.0 * u - prev + dt2 * g
            prev, u = u, new
            block.append(new)
            if len(block) == 16 or n + 1 == n_t:
                k = len(block)
                q += torch.tensordot(w[first:first + k], torch.stack(block), ([0], [0]))
                block, first = [], first + k
        q = torch.tensordot(self.binv, q, 1)
        out = torch.zeros_like(v)
        out[self.inner] = modes[1] @ q @ modes[0] if implicit else q
        return out

    def gmres(self, iters):
        b = self.pi(torch.zeros_like(self.f), True)
        beta = b.norm()
        basis, H, history = [b / beta], np.zeros((iters + 1, iters)), []
        for j in range(iters):
            x = basis[j] - self.pi(basis[j], False)
            for _ in range(2):
                for i in range(j + 1):
                    c = torch.dot(basis[i].reshape(-1), x.reshape(-1)).item()
                    H[i, j] += c
                    x = x - c * basis[i]
            H[j + 1, j] = x.norm().item()
            basis.append(x / H[j + 1, j])
            rhs = np.zeros(j + 2)
            rhs[0] = beta.item()
            y = np.linalg.lstsq(H[:j + 2, :j + 1], rhs, rcond=None)[0]
            history.append(float(np.linalg.norm(rhs - H[:j + 2, :j + 1] @ y) / beta.item()))
        return sum(c * v for c, v in zip(y, basis)), np.array(history)

    def helmholtz(self, v):
        om2 = torch.tensor(self.omega ** 2, device="cuda").view([-1] + [1] * len(self.h))
        f = self.f[self.inner]
        r = (f - self.lap(v) - om2 * v[self.inner]).abs().flatten(1).amax(1)
        return (r / f.abs().flatten(1).amax(1)).cpu().numpy()


def _exact_network(case, seed):
    flat, xs, ts, mask, xv, chans = _network(case, seed)
    p = flat.double().requires_grad_()

    def net(x, p):
        at = 0
        for i, (cin, cout) in enumerate(zip(chans[:-1], chans[1:])):
            w = p[at:at + 9 * cin * cout].view(cout, cin, 3, 3)
            bias = p[at + 9 * cin * cout:at + 9 * cin * cout + cout]
            at += 9 * cin * cout + cout
            # a convolution as one product per tap
            xp = torch.nn.functional.pad(x, (1, 1, 1, 1))
            x = bias.view(1, -1, 1, 1) + sum(
                torch.einsum("oc,bchw->bohw", w[:, :, dy, dx],
                             xp[:, :, dy:dy + x.shape[2], dx:dx + x.shape[3]])
                for dy in range(3) for dx in range(3))
            if i + 2 < len(chans):
                x = torch.relu(x)
        return x

    count = mask.sum().item() * xs.shape[0]
    loss = 0.0
    for i in range(0, xs.shape[0], 8):
        d = (net(xs[i:i + 8].double(), p)[:, 0] - ts[i:i + 8].double()) * mask
        part = (d * d).sum() / count
        part.backward()
        loss += part.item()
    g = p.grad
    with torch.no_grad():
        new = p - 1e-4 * g / (g.abs() + 1e-8)
        y = torch.cat([net(xv[i:i + 8].double(), new) for i in range(0, xv.shape[0], 8)])
    return dict(loss=loss, params=new.cpu().numpy(), grads=g.cpu().numpy(), prediction=y)


def exact(case, seed):
    if case["kind"] == "cnn":
        return _exact_network(case, seed)
    if case["kind"] == "batch":
        out = []
        for i, p in enumerate(_batch(case)):
            out.append(_Exact(p, _forcing(p, _omega(p), seed + 1000 * i)).gmres(case["iters"])[0])
        return out
    om = _omega(case)
    e = _Exact(case, _forcing(case, om, seed))
    if case["kind"] == "gmres":
        v, history = e.gmres(case["iters"])
        return dict(v=v, iterations=None, history=history, helmholtz=e.helmholtz(v))
    v = _iterate(case, om, seed)
    for _ in range(case["iters"] if case["kind"] == "fpi" else 1):
        v = e.pi(v, case["forced"] or case["kind"] == "fpi")
    return v
