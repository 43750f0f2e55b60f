"""The warm-start network where its workspace does not fit: the batch goes through in parts
(mfwh_debug_fail_allocations stands in for the end of memory)."""

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


@pytest.mark.parametrize("B,channels,fails", [(7, 24, 1), (8, 1, 2), (5, 32, 3), (1, 8, 0)])
def test_batches_in_parts(B, channels, fails):
    H, W = 33, 40
    g = torch.Generator(device="cuda").manual_seed(2)
    x = torch.randn(B, 2, H, W, device="cuda", generator=g)
    t = torch.randn(B, 1, H, W, device="cuda", generator=g)
    mask = torch.zeros(H, W, device="cuda")
    mask[1:-1, 1:-1] = 1.0
    got = []
    for short in (False, True):
        net = M.CNN(layers=4, channels=channels, seed=4)
        if short:
            # attempts for B, B / 2, .. images fail in turn
            _lib.check(_lib.load().mfwh_debug_fail_allocations(0, fails))
        y = torch.full((B, 1, H, W), float("nan"), device="cuda")
        net.forward(x, y)
        loss = net.train_step(x, t, mask, 1e-3)
        params, grads = net.get_params(grads=True)
        z = torch.full_like(y, float("nan"))
        net.forward(x, z)
        got.append((y.cpu().numpy(), loss, grads))
        _lib.check(_lib.load().mfwh_debug_fail_allocations(0, 0))
    (y0, l0, g0), (y1, l1, g1) = got
    assert np.array_equal(y0, y1)
    # sums of the same FP32 terms, of the parts one after the other
    terms = B * H * W
    assert abs(l0 - l1) <= 2.0 ** -24 * terms ** 0.5 * 8 * abs(l0)
    assert np.max(np.abs(g0 - g1)) <= 2.0 ** -24 * terms ** 0.5 * 8 * np.max(np.abs(g0))


def test_one_image_that_does_not_fit():
    net = M.CNN(layers=3, channels=8, seed=4)
    x = torch.zeros(2, 2, 16, 16, device="cuda")
    y = torch.zeros(2, 1, 16, 16, device="cuda")
    _lib.check(_lib.load().mfwh_debug_fail_allocations(0, 1000))
    with pytest.raises(_lib.MfwhError) as e:
        net.forward(x, y)
    _lib.check(_lib.load().mfwh_debug_fail_allocations(0, 0))
    assert e.value.status == _lib.ERR_NOMEM
    net.forward(x, y)   # the network stays usable
    torch.cuda.synchronize()
