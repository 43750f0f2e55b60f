"""Where device memory ends (mfwh_debug_fail_allocations stands in for it), an FP64 2D handle in
fixed point gives up its own workspace and goes on with the FP64 kernels.  What it computes then is
what a handle computes that left fixed point before its first map, bit for bit."""

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
    yield _lib.load()
    _lib.load().mfwh_debug_fail_allocations(0, 0)


def solver(n, nf, **kw):
    rng = np.random.default_rng(3)
    om = np.linspace(6.0, 6.0 + 2.5 * (nf - 1), nf) + 0.37
    f = torch.from_numpy(rng.normal(size=(nf, n[1] + 1, n[0] + 1))).cuda()
    return M.Solver(n, (1.0, n[1] / n[0]), om, f, n_p=2 if nf > 4 else 1,
                    filter_mode=_lib.FILTER_TRADITIONAL, **kw)


def drop(s):
    """The next workspace allocation fails once: the handle leaves fixed point."""
    _lib.check(_lib.load().mfwh_debug_fail_allocations(0, 1))
    s.set_graphs(True)
    s.set_graphs(False)


def results(s, v):
    out = []
    for forced in (True, False):
        o = torch.full(v.shape, float("nan"), dtype=torch.float64, device="cuda")
        s.apply_Pi(v, o, forced=forced)
        out.append(o.cpu().numpy())
    launches = s.last_timing()[1]
    x = torch.zeros_like(v)
    s.solve_gmres(x, restart=4, tol=0.0, max_iters=6, raise_on_error=False)
    return out + [x.cpu().numpy()], launches


# rows of 71 points (not a multiple of 32): the pipelined, the one-step and the fourth-order kernel
@pytest.mark.parametrize("nf,order,depth", [(3, 2, 3), (12, 2, 1), (3, 4, 1)])
@pytest.mark.parametrize("forced", [True, False])
def test_maps_after_leaving_fixed_point(nf, order, depth, forced):
    n = (70, 45)
    v = torch.from_numpy(np.random.default_rng(4).normal(size=(nf, n[1] + 1, n[0] + 1))).cuda()
    ref = solver(n, nf, order=order)
    drop(ref)
    want, launches = results(ref, v)
    assert launches == -(-ref.setup["n_t"] // depth)   # (of the last map)
    s = solver(n, nf, order=order)
    o = torch.empty_like(v)
    s.apply_Pi(v, o, forced=forced)
    assert s.last_timing()[1] == -(-s.setup["n_t"] // (4 if order == 4 else 8))
    fixed = o.cpu().numpy()
    drop(s)
    got, launches = results(s, v)
    assert launches == -(-s.setup["n_t"] // depth)
    for a, b in zip(got, want):
        assert np.array_equal(a, b)
    # and the two arithmetics agree
    scale = np.abs(fixed).max()
    assert np.abs(want[0 if forced else 1] - fixed).max() <= 1e-10 * scale


def test_krylov_basis_that_does_not_fit():
    """GMRES whose basis meets the end of memory after maps in fixed point."""
    n, nf = (70, 45), 3
    v = torch.from_numpy(np.random.default_rng(5).normal(size=(nf, n[1] + 1, n[0] + 1))).cuda()
    xs = []
    for first in (False, True):
        s = solver(n, nf)
        if first:
            s.solve_fpi(v.clone(), 3)
            _lib.check(_lib.load().mfwh_debug_fail_allocations(0, 1))
        else:
            drop(s)
        x = torch.zeros_like(v)
        s.solve_gmres(x, restart=4, tol=0.0, max_iters=6, raise_on_error=False)
        xs.append(x.cpu().numpy())
    assert np.array_equal(xs[0], xs[1])


def test_refined_solve_that_does_not_fit():
    """The FP64 residuals of an FP32 handle leave fixed point between two solves."""
    n, nf = (70, 45), 3
    xs = []
    for first in (False, True):
        s = solver(n, nf, precision=_lib.PREC_FP32_KAHAN)
        if first:
            x = torch.zeros((nf, n[1] + 1, n[0] + 1), dtype=torch.float64, device="cuda")
            s.solve_relaxed(x, restart=4, inner_tol=1e-3, max_iters=4, target=1e-3, max_refinements=1,
                            raise_on_error=False)
        drop(s)
        x = torch.zeros((nf, n[1] + 1, n[0] + 1), dtype=torch.float64, device="cuda")
        s.solve_relaxed(x, restart=6, inner_tol=1e-6, max_iters=12, target=1e-9, max_refinements=2,
                        raise_on_error=False)
        xs.append(x.cpu().numpy())
    assert np.isfinite(xs[0]).all() and np.array_equal(xs[0], xs[1])


@pytest.mark.parametrize("after", [0, 3, 14])
def test_creation_without_the_workspace_for_speed(after):
    """Memory that ends during mfwh_create: the handle is made without fixed point (its 15th
    allocation, the forcing of a launch, is the first that the FP64 kernels do without)."""
    n, nf = (70, 45), 3
    v = torch.from_numpy(np.random.default_rng(6).normal(size=(nf, n[1] + 1, n[0] + 1))).cuda()
    ref = solver(n, nf)
    drop(ref)
    want, _ = results(ref, v)
    _lib.check(_lib.load().mfwh_debug_fail_allocations(after, 1))
    s = solver(n, nf)
    _lib.check(_lib.load().mfwh_debug_fail_allocations(0, 0))
    got, launches = results(s, v)
    assert launches == -(-s.setup["n_t"] // 3)
    for a, b in zip(got, want):
        assert np.array_equal(a, b)
    _lib.check(_lib.load().mfwh_debug_fail_allocations(after, 1000))   # and where nothing helps
    with pytest.raises(_lib.MfwhError) as e:
        solver(n, nf)
    _lib.check(_lib.load().mfwh_debug_fail_allocations(0, 0))
    assert e.value.status == _lib.ERR_NOMEM


@pytest.mark.parametrize("n", [(70, 45), (3, 90), (191, 130)])
@pytest.mark.parametrize("tb", [1, 4, 16])
def test_fp32_rows_where_memory_is_short(n, tb):
    """FP32 handles made at the second attempt have rows of whole 16-byte accesses: same bits."""
    nf = 3
    v = torch.from_numpy(np.random.default_rng(7).normal(size=(nf, n[1] + 1, n[0] + 1))).cuda()
    out = []
    for short in (False, True):
        if short:
            _lib.check(_lib.load().mfwh_debug_fail_allocations(2, 1))
        s = solver(n, nf, precision=_lib.PREC_FP32_KAHAN, time_block=tb)
        res = []
        for forced in (True, False):
            o = torch.full_like(v, float("nan"))
            s.apply_Pi(v, o, forced=forced)
            res.append(o.cpu().numpy())
        out.append(res)
        s.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def cube(n, nf, tb, **kw):
    rng = np.random.default_rng(9)
    om = np.linspace(6.0, 6.0 + 2.5 * (nf - 1), nf)
    f = torch.from_numpy(rng.normal(size=(nf,) + tuple(k + 1 for k in reversed(n)))).cuda()
    return M.Solver(n, tuple(k / n[0] for k in n), om, f, n_p=2 if nf > 2 else 1, time_block=tb,
                    filter_mode=_lib.FILTER_TRADITIONAL, precision=_lib.PREC_FP32_BLOCKSUM, **kw)


@pytest.mark.parametrize("n,nf,layer", [
    ((2, 2, 2), 1, None), ((3, 30, 5), 2, 1), ((54, 7, 11), 2, None), ((55, 8, 12), 1, 0),
    ((56, 9, 13), 3, 2), ((57, 11, 15), 2, None), ((60, 12, 16), 9, 1), ((61, 13, 17), 2, 2),
    ((120, 33, 40), 4, 0)])
@pytest.mark.parametrize("tb", [2, 4])
def test_partial_sums_of_steps_and_of_blocked_launches(n, nf, layer, tb):
    """The 3D FP32 sums over 2 or 4 steps: one step per launch with an array of partial sums, and,
    where that array does not fit, the blocked kernel, at its tile edges: same bits."""
    shape = (nf,) + tuple(k + 1 for k in reversed(n))
    v = np.random.default_rng(10).normal(size=shape)
    for a in (1, 2, 3):
        v[tuple([slice(None)] * a + [[0, -1]])] = 0.0
    v = torch.from_numpy(v).cuda()
    kw = {} if layer is None else dict(c_lo=1.0, c_hi=1.4, interface=0.37 * n[layer] / n[0],
                                       layer_axis=layer)

    def maps(s):
        out = []
        for forced in (True, False):
            o = torch.full_like(v, float("nan"))
            s.apply_Pi(v, o, forced=forced)
            out.append(o.cpu().numpy())
        launches = s.last_timing()[1]   # (of the homogeneous map)
        return out, launches
    s = cube(n, nf, tb, **kw)
    want, launches = maps(s)
    n_t = s.setup["n_t"]
    assert launches == n_t
    # give the array up for a workspace that does not fit
    drop(s)
    got, launches = maps(s)
    assert launches == -(-n_t // tb)
    for a, b in zip(got, want):
        assert np.array_equal(a, b)


def test_fp32_rows_of_3d_grids_are_hardly_padded():
    """A 3D FP32 handle of 33 points a row takes about 33 / 32 of one of 32."""
    used = []
    for nx in (31, 32):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        s = cube((nx, 200, 200), 4, 4)
        torch.cuda.empty_cache()
        before = torch.cuda.mem_get_info()[0]
        s.close()
        used.append(torch.cuda.mem_get_info()[0] - before)
    assert used[0] > 0 and used[1] < 1.15 * used[0], used
