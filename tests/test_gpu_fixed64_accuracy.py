"""Accuracy of the fixed-point 2D maps of second order against extended precision: in the maximum norm
no further off than a plain FP64 run of the scheme (two levels, FP64 sums), plus the rounding of
the result.  A quantum some bits too coarse or an increment rounded with a bias, whose error grows
with the square of the steps, is further off."""

import numpy as np
import pytest

import paper_2507_23613_gb300 as M
from paper_2507_23613_gb300 import _lib, build

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()


def scheme(T, n, length, s, w, f, v, layer, forced):
    """V in the number type T, by W^{n+1} = 2 W^n - W^{n-1} + dt^2 (c^2 Delta_h W^n - F^n)."""
    c2 = np.ones((n[1] + 1, n[0] + 1), T)
    if layer is not None:
        axis, at, c = layer
        x = np.arange(n[axis] + 1) * (length[axis] / n[axis])
        g = np.where(x < at, 1.0, c * c).astype(T)
        c2 = c2 * (g if axis == 0 else g[:, None])
    c2 = c2[1:-1, 1:-1]
    n_t, dt2 = s["n_t"], T(s["dt"]) ** 2
    ax, ay = dt2 / T(length[0] / n[0]) ** 2, dt2 / T(length[1] / n[1]) ** 2
    cos = np.cos(np.arange(n_t)[:, None] * s["dt"] * np.asarray(s["omega_tilde"])[None]).astype(T)
    w, f = w.astype(T), f.astype(T)[:, 1:-1, 1:-1]
    u = np.zeros((n[1] + 1, n[0] + 1), T)
    u[1:-1, 1:-1] = v.astype(T).sum(0)[1:-1, 1:-1]
    q = w[0][:, None, None] * u[None, 1:-1, 1:-1]
    prev = None
    for k in range(n_t):
        i = u[1:-1, 1:-1]
        inc = c2 * (ax * (u[1:-1, :-2] - 2 * i + u[1:-1, 2:]) + ay * (u[:-2, 1:-1] - 2 * i + u[2:, 1:-1]))
        if forced:
            inc = inc - dt2 * np.tensordot(cos[k], f, 1)
        new = np.zeros_like(u)
        new[1:-1, 1:-1] = i + inc / 2 if k == 0 else 2 * i - prev[1:-1, 1:-1] + inc
        prev, u = u, new
        q = q + w[k + 1][:, None, None] * u[None, 1:-1, 1:-1]
    out = np.zeros((len(w[0]),) + u.shape, T)
    out[:, 1:-1, 1:-1] = np.tensordot(np.asarray(s["B_inv"]).astype(T), q, 1)
    return out


@pytest.mark.parametrize("n,nf,layer", [((64, 49), 2, None), ((80, 60), 3, (0, 0.4, 1.5)),
                                        ((49, 97), 5, (1, 0.9, 1.2))])
@pytest.mark.parametrize("smooth", [True, False])
@pytest.mark.parametrize("forced", [True, False])
def test_no_further_off_than_fp64_steps(n, nf, layer, smooth, forced):
    if np.finfo(np.longdouble).nmant < 60:
        pytest.skip("no extended precision")
    rng = np.random.default_rng(nf)
    om = np.linspace(6.0, 6.0 + 2.5 * (nf - 1), nf) + 0.37
    length = (1.0, 1.1 * n[1] / n[0])
    shape = (nf, n[1] + 1, n[0] + 1)
    if smooth:
        sx, sy = (np.sin(np.pi * np.outer(np.arange(1, 6), np.arange(k + 1) / k)) for k in n)
        v = np.einsum("mij,iy,jx->myx", rng.normal(size=(nf, 5, 5)), sy, sx)
        f = np.einsum("mij,iy,jx->myx", rng.normal(size=(nf, 5, 5)), sy, sx) * 30.0
    else:
        v, f = rng.normal(size=shape), rng.normal(size=shape) * 30.0
    v[:, [0, -1]] = 0.0
    v[:, :, [0, -1]] = 0.0
    kw = dict(n_p=2 if nf > 4 else 1, filter_mode=_lib.FILTER_TRADITIONAL)
    if layer is not None:
        kw.update(c_lo=1.0, c_hi=layer[2], interface=layer[1], layer_axis=layer[0])
    s = M.Solver(n, length, om, torch.from_numpy(f).cuda(), **kw)
    got = torch.empty(shape, dtype=torch.float64, device="cuda")
    s.apply_Pi(torch.from_numpy(v).cuda(), got, forced=forced)
    got = got.cpu().numpy()
    setup = s.setup
    assert s.last_timing()[1] == -(-setup["n_t"] // 8)   # in fixed point
    p, keep = M.make_problem(n, length, om, None, **kw)
    w = M.plan_weights(p, setup["n_t"], nf)
    exact = scheme(np.longdouble, n, length, setup, w, f, v, layer, forced)
    fp64 = scheme(np.float64, n, length, setup, w, f, v, layer, forced)
    top = np.abs(exact).max((1, 2))
    # |V| <= |B^{-1}| sum |w| max |W|: the sums' and the filter solve's roundings
    amp = np.abs(setup["B_inv"]) @ (np.abs(w).sum(0) * np.abs(v).sum(0).max())
    err, ref = (np.abs(x - exact).max((1, 2)) for x in (got, fp64))
    assert np.all(err <= ref + 2.0 ** -50 * np.maximum(top, amp)), (err / top, ref / top)
