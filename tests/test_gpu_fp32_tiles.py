"""The FP32 blocked 2D kernel at grids around its tile edges (96 x 32 owned points at depth 16,
112 x 48 at depths 8 and 4; whole 4 x 4 blocks per thread), forced and homogeneous, with unequal
spacings and two layers: with Kahan sums every depth performs the one-step kernel's
operations per point, so the maps are equal bit for bit."""

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
    ((2, 2), 1, None), ((3, 90), 2, None), ((94, 30), 3, None), ((95, 31), 1, 0),
    ((96, 32), 16, None), ((97, 33), 2, 1), ((111, 47), 2, None), ((112, 48), 9, 0),
    ((113, 49), 3, 1), ((191, 130), 2, None), ((300, 200), 4, 1)])
def test_blocked_depths_equal_one_step_at_tile_edges(n, nf, layer):
    om = np.linspace(6.0, 6.0 + 2.5 * (nf - 1), nf)
    wl = inputs.gaussian_workload("tile", n, nf, om, 150.0, 3)
    f = torch.from_numpy(wl.forcing).cuda()
    v = torch.from_numpy(np.random.default_rng(4).normal(size=wl.forcing.shape) * 0.01).cuda()
    kw = {} if layer is None else dict(c_lo=1.0, c_hi=1.4, interface=0.37, layer_axis=layer)
    outs = {}
    for tb in (1, 4, 8, 16):
        s = M.Solver(n, wl.length, om, f, n_p=2 if nf > 2 else 1, time_block=tb,
                     filter_mode=_lib.FILTER_TRADITIONAL, precision=_lib.PREC_FP32_KAHAN, **kw)
        res = []
        for forced in (True, False):
            o = torch.full_like(v, float("nan"))
            s.apply_Pi(v, o, forced=forced)
            res.append(o.cpu().numpy())
        s.close()
        outs[tb] = res
    for tb in (4, 8, 16):
        for a, b in zip(outs[tb], outs[1]):
            assert np.array_equal(a, b), (tb, np.max(np.abs(a - b)))
