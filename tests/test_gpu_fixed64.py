"""The FP64 2D wave solve in fixed point against the FP64 one-step path (which a c^2 given at every
point takes) on grids around its tile edges (48 columns, 4 to 32 rows), with every number of
frequencies, equal and unequal spacings, layers along each axis, forced and homogeneous, over the
range of magnitudes and for values without a quantum."""

import numpy as np
import pytest

import paper_2507_23613_gb300 as M
from paper_2507_23613_gb300 import _lib, build, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    return _lib.load()


def maps(n, length, om, f, v, layer=None, general=False, forced=True, n_p=1, order=2):
    kw = dict(n_p=n_p, filter_mode=_lib.FILTER_TRADITIONAL, order=order)
    if layer is not None:
        axis, at, c = layer
        if general:
            x = np.arange(n[axis] + 1) * (length[axis] / n[axis])
            c2 = np.where(x < at, 1.0, c * c)
            kw["c2_field"] = np.ascontiguousarray(np.broadcast_to(
                c2 if axis == 0 else c2[:, None], (n[1] + 1, n[0] + 1)))
        else:
            kw.update(c_lo=1.0, c_hi=c, interface=at, layer_axis=axis)
    elif general:
        kw["c2_field"] = np.ones((n[1] + 1, n[0] + 1))
    s = M.Solver(n, length, om, torch.from_numpy(f).cuda(), **kw)
    out = torch.full(v.shape, float("nan"), dtype=torch.float64, device="cuda")
    s.apply_Pi(torch.from_numpy(v).cuda(), out, forced=forced)
    setup = s.setup
    s.close()
    return out.cpu().numpy(), setup


def data(n, nf, seed, scale_v=1.0, scale_f=1.0):
    rng = np.random.default_rng(seed)
    shape = (nf, n[1] + 1, n[0] + 1)
    v = rng.normal(size=shape) * scale_v
    v[:, [0, -1]] = 0.0
    v[:, :, [0, -1]] = 0.0
    return rng.normal(size=shape) * scale_f, v


def check(n, length, om, f, v, layer, forced, n_p=1, order=2):
    """Both paths are within n_t^2 / 2 roundings of a step (2^-52 of the levels, a constant bias at
    worst) of the exact levels; V = B^{-1} sum w W."""
    got, s = maps(n, length, om, f, v, layer, False, forced, n_p, order)
    # (the one-step path's sums are pairs of floats: its inputs are brought near 1 by a power of
    # two, which is exact)
    k = np.frexp(max(np.abs(v).max(), np.abs(f).max() if forced else 0.0))[1]
    want, _ = maps(n, length, om, np.ldexp(f, -k) if forced else f, np.ldexp(v, -k), layer, True,
                   forced, n_p, order)
    want = np.ldexp(want, k)
    nf, n_t, dt = len(om), s["n_t"], s["dt"]
    # the levels of the homogeneous problem are bounded by a small multiple of W^0 in the energy
    # norm; forced ones grow by t dt sum |f| at most
    level = 8.0 * np.abs(v).sum(0).max()
    if forced:
        level += n_t ** 2 * dt ** 2 * np.abs(f).sum(0).max()
    kw = {} if layer is None else dict(c_lo=1.0, c_hi=layer[2], interface=layer[1],
                                       layer_axis=layer[0])
    p, keep = M.make_problem(n, length, om, None, n_p=n_p, filter_mode=_lib.FILTER_TRADITIONAL,
                             order=order, **kw)
    w = np.abs(M.plan_weights(p, n_t, nf)).sum(0)
    bound = n_t ** 2 * 2.0 ** -52 * level * (np.abs(s["B_inv"]) @ w)
    err = np.abs(got - want).max((1, 2))
    assert np.isfinite(want).all() and np.all(err <= bound), (err, bound)
    assert np.all(got[:, [0, -1]] == 0.0) and np.all(got[:, :, [0, -1]] == 0.0)


GRIDS = [((2, 2), 1, None), ((3, 5), 1, None), ((46, 14), 2, (0, 0.4, 1.5)),
         ((47, 15), 3, None), ((48, 16), 4, (1, 0.5, 1.3)), ((49, 17), 5, None),
         ((65, 64), 6, (1, 0.93, 0.8)), ((195, 151), 16, None), ((95, 31), 7, (0, 0.01, 1.2)), ((96, 33), 9, None),
         ((97, 63), 10, None), ((33, 145), 11, (0, 0.5, 1.1)), ((200, 70), 13, None),
         ((71, 211), 14, (1, 0.3, 1.4)), ((300, 260), 8, (0, 0.6, 1.3)), ((530, 500), 12, None),
         ((1100, 640), 1, (1, 0.7, 1.2)), ((160, 161), 15, None)]


@pytest.mark.parametrize("n,nf,layer", GRIDS)
@pytest.mark.parametrize("forced", [False, True])
def test_fixed_point_map_is_the_general_one(n, nf, layer, forced):
    om = np.linspace(6.0, 6.0 + 2.5 * (nf - 1), nf) + 0.37
    f, v = data(n, nf, 1)
    for length in ((1.0, n[1] / n[0]), (1.0, 1.2 * n[1] / n[0])):   # equal and unequal spacings
        lay = None if layer is None else (layer[0], layer[1] * length[layer[0]], layer[2])
        check(n, length, om, f, v, lay, forced, n_p=2 if nf > 4 else 1)


@pytest.mark.parametrize("sv,sf", [(1e-200, 0.0), (1e200, 1e200), (0.0, 1e-180), (1.0, 1e30),
                                   (1e30, 1.0), (1e-305, 0.0), (0.0, 1e-290), (1e-300, 1e-280)])
def test_range_of_magnitudes(sv, sf):
    f, v = data((90, 50), 3, 2, sv, sf)
    for forced in (False, True):
        check((90, 50), (1.0, 0.6), np.array([6.1, 9.3, 13.0]), f, v, None, forced)


def test_zero_input_and_values_without_a_quantum():
    n, length, om = (60, 40), (1.0, 0.7), np.array([6.1, 9.3])
    f, v = data(n, 2, 3)
    out, _ = maps(n, length, om, f, 0.0 * v, forced=False)
    assert np.all(out == 0.0)
    out, _ = maps(n, length, om, 0.0 * f, 0.0 * v, forced=True)
    assert np.all(out == 0.0)
    for bad in (np.inf, -np.inf, np.nan):
        for which in (0, 1):
            g, w = f.copy(), v.copy()
            (g, w)[which][1, 20, 30] = bad
            got, _ = maps(n, length, om, g, w, forced=True)
            want, _ = maps(n, length, om, g, w, general=True, forced=True)
            assert np.array_equal(np.isfinite(got), np.isfinite(want))
            assert not np.isfinite(got).all()


def fourth_order_reference(n, length, s, w, f, v, layer, forced):
    """Extended-precision map with the fourth-order operator (odd reflection at the boundary)."""
    L = np.longdouble
    c2 = np.ones((n[1] + 1, n[0] + 1), L)
    if layer is not None:
        axis, at, c = layer
        x = np.arange(n[axis] + 1) * (length[axis] / n[axis])
        c2 = c2 * (np.where(x < at, 1.0, c * c) if axis == 0 else
                   np.where(x < at, 1.0, c * c)[:, None])
    dt, n_t = L(s["dt"]), s["n_t"]
    u = v.astype(L).sum(0)
    f = f.astype(L)
    cos = np.cos(np.arange(n_t)[:, None] * s["dt"] * np.asarray(s["omega_tilde"])[None]).astype(L)
    w = w.astype(L)
    q = w[0][:, None, None] * u[None]
    d = np.zeros_like(u)
    h = [length[a] / n[a] for a in (0, 1)]

    def second(u, axis):
        e = np.moveaxis(u, axis, 0)
        e = np.concatenate([-e[1:2], e, -e[-2:-1]])
        t = -e[:-4] + 16 * e[1:-3] - 30 * e[2:-2] + 16 * e[3:-1] - e[4:]
        out = np.zeros_like(u)
        np.moveaxis(out, axis, 0)[1:-1] = t / 12
        return out
    for k in range(n_t):
        inc = dt * dt * c2 * (second(u, 1) / L(h[0]) ** 2 + second(u, 0) / L(h[1]) ** 2)
        if forced:
            inc = inc - dt * dt * np.tensordot(cos[k], f, 1)
        inc[[0, -1]] = 0
        inc[:, [0, -1]] = 0
        d = d + (inc / 2 if k == 0 else inc)
        u = u + d
        q = q + w[k + 1][:, None, None] * u[None]
    out = np.tensordot(np.asarray(s["B_inv"]).astype(L), q, 1)
    out[:, [0, -1]] = 0
    out[:, :, [0, -1]] = 0
    return out


@pytest.mark.parametrize("n,nf,layer", [
    ((2, 3), 1, None), ((3, 2), 2, None), ((47, 15), 3, (0, 0.4, 1.5)), ((49, 17), 5, None),
    ((65, 64), 2, (1, 0.93, 0.8)), ((96, 33), 9, None), ((95, 31), 1, (1, 0.3, 1.2)),
    ((71, 47), 1, None), ((150, 60), 4, None), ((90, 62), 2, None), ((144, 65), 3, None),
    ((145, 97), 16, None)])
@pytest.mark.parametrize("forced", [False, True])
def test_fourth_order_map(n, nf, layer, forced):
    om = np.linspace(6.0, 6.0 + 2.5 * (nf - 1), nf) + 0.37
    f, v = data(n, nf, 5)
    length = (1.0, 1.1 * n[1] / n[0])
    lay = None if layer is None else (layer[0], layer[1] * length[layer[0]], layer[2])
    n_p = 2 if nf > 4 else 1
    got, s = maps(n, length, om, f, v, lay, False, forced, n_p, 4)
    kw = {} if lay is None else dict(c_lo=1.0, c_hi=lay[2], interface=lay[1], layer_axis=lay[0])
    p, keep = M.make_problem(n, length, om, None, n_p=n_p, filter_mode=_lib.FILTER_TRADITIONAL,
                             order=4, **kw)
    w = M.plan_weights(p, s["n_t"], nf)
    want = fourth_order_reference(n, length, s, w, f, v, lay, forced)
    level = 8.0 * np.abs(v).sum(0).max()
    if forced:
        level += s["n_t"] ** 2 * s["dt"] ** 2 * np.abs(f).sum(0).max()
    # as in check(); the products' coefficients are rounded to 53 bits in the map only
    bound = s["n_t"] ** 2 * 2.0 ** -52 * level * (np.abs(s["B_inv"]) @ np.abs(w).sum(0))
    err = np.abs(got - want).max((1, 2))
    assert np.isfinite(got).all() and np.all(err <= bound), (err, bound)
