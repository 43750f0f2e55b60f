"""The FP32 blocked 3D kernel at grids around its tile edges (56 x 8 x 12 owned points at depth 4,
60 x 12 x 16 at depth 2), forced and homogeneous, with two layers along each axis: with Kahan
sums the two depths perform the same operations per point on different tiles, so their maps
are equal bit for bit, and both are within the FP32 path's error (2e-5, as in test_gpu_fp32.py) of
the FP64 map."""

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


@pytest.mark.parametrize("n,nf,layer", [
    ((2, 2, 2), 1, None), ((3, 30, 5), 2, 1), ((54, 7, 11), 2, None), ((55, 8, 12), 1, 0),
    ((56, 9, 13), 3, 2), ((57, 11, 15), 2, None), ((60, 12, 16), 9, 1), ((61, 13, 17), 2, 2),
    ((130, 40, 60), 2, None), ((120, 33, 40), 4, 0)])
def test_blocked_depths_agree_at_tile_edges(n, nf, layer):
    om = np.linspace(6.0, 6.0 + 2.5 * (nf - 1), nf)
    wl = inputs.gaussian_workload("tile", n, nf, om, 100.0, 3)
    f = torch.from_numpy(wl.forcing).cuda()
    # a smooth iterate (standing waves): the FP32 error bound is for resolved fields
    v = np.zeros_like(wl.forcing)
    axes = [np.sin(np.pi * np.arange(k + 1) / k) for k in n]
    for m in range(nf):
        v[m] = 0.01 * (m + 1) * axes[2][:, None, None] * axes[1][:, None] * axes[0]
    v = torch.from_numpy(v).cuda()
    kw = {} if layer is None else dict(c_lo=1.0, c_hi=1.4, interface=0.37, layer_axis=layer)
    outs = {}
    for key, prec, tb in (("fp64", _lib.PREC_FP64, 0), ("default", _lib.PREC_FP32_BLOCKSUM, 0),
                          (1, _lib.PREC_FP32_KAHAN, 1), (2, _lib.PREC_FP32_KAHAN, 2),
                          (4, _lib.PREC_FP32_KAHAN, 4)):
        s = M.Solver(n, wl.length, om, f, n_p=2 if nf > 2 else 1, time_block=tb, precision=prec,
                     filter_mode=_lib.FILTER_TRADITIONAL, **kw)
        res = []
        for forced in (True, False):
            o = torch.full_like(v, float("nan"))
            s.apply_Pi(v, o, forced=forced)
            res.append(o.cpu().numpy())
        s.close()
        outs[key] = res
    for key in ("default", 1, 2):
        for a, b in zip(outs[key], outs[4]):
            assert np.array_equal(a, b), (key, np.max(np.abs(a - b)))
    for a, b in zip(outs[4], outs["fp64"]):
        assert np.max(np.abs(a - b)) <= 2e-5 * np.max(np.abs(b))


@pytest.mark.parametrize("n,prec,tb,layer", [
    ((112, 128, 144), _lib.PREC_FP32_BLOCKSUM, 4, 0), ((111, 127, 143), _lib.PREC_FP32_BLOCKSUM, 4, None),
    ((119, 131, 127), _lib.PREC_FP32_BLOCKSUM, 2, 2), ((120, 132, 124), _lib.PREC_FP32_BLOCKSUM, 2, None),
    ((112, 136, 159), _lib.PREC_FP32_KAHAN, 1, 1), ((113, 135, 156), _lib.PREC_FP32_KAHAN, 2, None),
    ((167, 119, 131), _lib.PREC_FP32_KAHAN, 4, 0)])
def test_one_step_launches_give_the_bits_of_the_blocked_ones(n, prec, tb, layer):
    """Grids that fill L2 without the forcing (one step per launch, partial sums over as many steps
    as the depth) but not with it (blocked launches): with a forcing of zeros the forced map is the
    homogeneous one, bit for bit."""
    om = np.linspace(30.0, 60.0, 4)
    length = tuple(k / n[0] for k in n)
    rng = np.random.default_rng(4)
    v = np.zeros((4, n[2] + 1, n[1] + 1, n[0] + 1))
    v[:, 1:-1, 1:-1, 1:-1] = rng.normal(size=(4, n[2] - 1, n[1] - 1, n[0] - 1))
    v = torch.from_numpy(v).cuda()
    kw = {} if layer is None else dict(c_lo=1.0, c_hi=1.4, interface=0.37, layer_axis=layer)
    s = M.Solver(n, length, om, torch.zeros_like(v), n_p=1, time_block=tb, precision=prec,
                 filter_mode=_lib.FILTER_TRADITIONAL, **kw)
    out = []
    for forced in (True, False):
        o = torch.full_like(v, float("nan"))
        s.apply_Pi(v, o, forced=forced)
        out.append(o.cpu().numpy())
    s.close()
    assert np.array_equal(out[0], out[1])
