"""The FP32 2D kernels by grid size: k_ring2d32 on grids of few tiles, k_tb2d32 with tiles of fewer rows
where all rows would leave SMs idle, and with all.  With Kahan sums every depth performs the
one-step kernel's operations per point: equal bit for bit at the edges of their tiles."""

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


# few frequencies: k_tb2d32 at any size (4 rows owned up to 513^2); more: k_ring2d32 up to about
# 400^2 (tiles of 32 x 32 and 32 x 16), then k_tb2d32
@pytest.mark.parametrize("n,nf,layer", [
    ((119, 55), 2, None), ((120, 56), 1, 0), ((121, 57), 3, 1), ((255, 131), 2, None),
    ((401, 520), 2, 0), ((1000, 640), 1, 1), ((31, 15), 5, None), ((32, 16), 6, 0),
    ((33, 33), 4, 1), ((63, 31), 16, None), ((64, 32), 13, 0), ((95, 97), 8, None),
    ((257, 255), 12, 1), ((330, 200), 7, None), ((450, 510), 16, None), ((640, 300), 5, 0)])
def test_depths_equal_one_step(n, nf, layer):
    rng = np.random.default_rng(nf)
    om = np.linspace(9.0, 9.0 + 2.5 * (nf - 1), nf)
    shape = (nf, n[1] + 1, n[0] + 1)
    f, v = rng.normal(size=shape), rng.normal(size=shape)
    f, v = torch.from_numpy(f).cuda(), torch.from_numpy(v).cuda()
    v[:, [0, -1]] = 0.0
    v[:, :, [0, -1]] = 0.0
    length = (1.0, 1.1 * n[1] / n[0])
    kw = {} if layer is None else dict(c_lo=1.0, c_hi=1.4, interface=0.37 * length[layer],
                                       layer_axis=layer)
    outs = {}
    for tb in (1, 4, 8, 16):
        s = M.Solver(n, length, om, f, n_p=1 if nf < 4 else 2, time_block=tb,
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
    assert np.isfinite(outs[1][0]).all()
