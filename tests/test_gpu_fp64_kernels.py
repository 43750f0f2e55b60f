"""The FP64 kernels of 2D problems that fixed point does not take: coefficients dt^2 c^2 / h^2 (fourth
order: / 12) below 2^-10 (spacings or speeds far apart), at least 1 or a multiple of 2^-24, and
grids that its tiles would mostly pad.  Which kernels ran is read off the number of step launches."""

import numpy as np
import pytest

import paper_2507_23613_gb300 as M
from oracle import filters as F
from oracle import wave as W
from paper_2507_23613_gb300 import _lib, build, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TOL = 1e-10   # of the FP64 maps against the oracle, as in test_gpu_parity.py

# name, cells, sides, frequencies, order, layers (axis, interface, c_hi)
PROBLEMS = [
    ("spacings", (200, 45), (1.0, 4.0), 3, 2, None),
    ("spacings_y", (45, 70), (16.0, 1.0), 2, 2, None),
    ("speeds", (40, 24), (1.0, 0.61), 2, 2, (1, 0.2, 13.0)),
    ("speeds_x", (49, 70), (1.0, 1.42), 2, 2, (0, 0.37, 13.0)),
    ("nf12", (40, 33), (1.0, 16.0), 12, 2, None),
    ("order4", (50, 40), (1.0, 0.9), 2, 4, (1, 0.3, 3.0)),
    ("order4_spacings", (48, 49), (1.0, 5.0), 5, 4, None),
]


@pytest.fixture(scope="module", autouse=True)
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    return _lib.load()


def case(name):
    _, n, length, nf, order, layer = next(p for p in PROBLEMS if p[0] == name)
    om = np.linspace(6.0, 6.0 + 2.5 * (nf - 1), nf)
    wl = inputs.gaussian_workload(name, n, nf, om, 40.0, 5, length=length)
    wl.n_p = 2 if nf > 2 else 1
    v = np.random.default_rng(6).normal(size=wl.forcing.shape) * 0.01
    v[:, [0, -1]] = 0.0
    v[:, :, [0, -1]] = 0.0
    kw = dict(n_p=wl.n_p, filter_mode=_lib.FILTER_TRADITIONAL, order=order)
    if layer:
        kw.update(c_lo=1.0, c_hi=layer[2], interface=layer[1], layer_axis=layer[0])
    return wl, v, kw, layer, order


def run(wl, v, kw, **more):
    """Pi, S, a few GMRES iterations; step launches of a map; N_t."""
    s = M.Solver(wl.n, wl.length, wl.omega, torch.from_numpy(wl.forcing).cuda(), **kw, **more)
    res = []
    vd = torch.from_numpy(v).cuda()
    for forced in (True, False):
        o = torch.full_like(vd, float("nan"))
        s.apply_Pi(vd, o, forced=forced)
        launches = s.last_timing()[1]
        res.append(o.cpu().numpy())
    x = torch.zeros_like(vd)
    s.solve_gmres(x, restart=4, tol=0.0, max_iters=6, raise_on_error=False)
    res.append(x.cpu().numpy())
    n_t = s.setup["n_t"]
    s.close()
    return res, launches, n_t


@pytest.mark.parametrize("name", [p[0] for p in PROBLEMS])
def test_depths_and_tiles_equal_one_step_and_the_oracle(name):
    wl, v, kw, layer, order = case(name)
    configs = [(1, 0)]
    if order == 2:
        configs += [(2, 1), (2, 5), (3, 4), (3, 5), (4, 0), (4, 2), (4, 5), (8, 0), (8, 1), (8, 2),
                    (8, 3)]
    ref = None
    for tb, shape in configs:
        got, launches, n_t = run(wl, v, kw, time_block=tb, tile_shape=shape)
        assert launches == -(-n_t // tb), (tb, shape)
        if ref is None:
            ref = got
        for a, b in zip(got, ref):
            assert np.array_equal(a, b), (tb, shape, np.max(np.abs(a - b)))
    # the default: the pipelined kernel, 3 steps per pass, up to 8 frequencies at second order
    got, launches, n_t = run(wl, v, kw)
    assert launches == (-(-n_t // 3) if order == 2 and len(wl.omega) <= 8 else n_t)
    for a, b in zip(got, ref):
        assert np.array_equal(a, b)
    c2 = 1.0
    if layer:
        axis, at, c = layer
        x = np.arange(wl.n[axis] + 1) * (wl.length[axis] / wl.n[axis])
        c2 = np.where(x < at, 1.0, c * c)
        c2 = np.broadcast_to(c2 if axis == 0 else c2[:, None], v.shape[1:])
    prob = W.make_problem(W.Grid(wl.n, wl.length), wl.omega, wl.forcing, c2=c2, cfl=0.5,
                          n_p=wl.n_p, filter_mode=F.FILTER_TRADITIONAL, order=order)
    for got, forced in ((ref[0], True), (ref[1], False)):
        want = W.apply_Pi(prob, v, forced=forced)
        err = np.abs(got - want).max((1, 2)) / np.abs(want).max((1, 2))
        assert np.all(err <= TOL), err
