"""The warm-start network's channel-innermost kernels at the sizes where they can go wrong: channel
counts around the padding groups (8, 16, 32), one channel, images narrower than a warp and wider
than one gradient strip, row counts around the strip height, batches of fewer pixels than one
tile.  Reference and tolerances as in test_gpu_cnn.py (BF16 activations)."""

import numpy as np
import pytest

import paper_2507_23613_gb300 as M
from oracle import cnn
from test_gpu_cnn import bf16, dev32, lib, unflatten  # noqa: F401

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("layers,channels,cin,B,H,W", [
    (2, 1, 1, 1, 3, 5), (3, 9, 2, 2, 16, 64), (3, 16, 8, 1, 17, 65), (3, 17, 9, 1, 15, 130),
    (4, 24, 3, 3, 33, 31), (3, 32, 32, 1, 5, 200), (2, 8, 17, 2, 1, 1)])
def test_network_matches_the_reference_at_awkward_shapes(layers, channels, cin, B, H, W):
    chans = [cin] + [channels] * (layers - 1) + [1]
    net = M.CNN(layers=layers, channels=channels, in_channels=cin, seed=3)
    rng = np.random.default_rng(7)
    flat = np.concatenate([np.concatenate([rng.normal(size=co * ci * 9) * np.sqrt(2 / (9 * ci)),
                                           rng.normal(size=co) * 0.05])
                           for ci, co in zip(chans[:-1], chans[1:])]).astype(np.float32)
    net.set_params(flat)
    x = rng.normal(size=(B, cin, H, W)).astype(np.float32)
    t = rng.normal(size=(B, 1, H, W)).astype(np.float32)
    mask = np.ones((H, W), dtype=np.float32)
    params = [(bf16(w), b) for w, b in unflatten(flat, chans)]
    want, _ = cnn.forward(params, bf16(x))
    y = torch.empty((B, 1, H, W), dtype=torch.float32, device="cuda")
    net.forward(dev32(x), y)
    torch.cuda.synchronize()
    assert np.max(np.abs(y.cpu().numpy() - want)) <= 2e-2 * np.max(np.abs(want))
    loss = net.train_step(dev32(x), dev32(t), dev32(mask), 1e-3)
    want_loss, want_grads = cnn.loss_and_grads(params, bf16(x), t.astype(np.float64), mask)
    assert abs(loss - want_loss) <= 2e-2 * want_loss
    _, g = net.get_params(grads=True)
    for (gw, gb), (ow, ob) in zip(unflatten(g, chans), want_grads):
        assert np.linalg.norm(gw - ow) <= 5e-2 * max(np.linalg.norm(ow), 1e-12)
        assert np.linalg.norm(gb - ob) <= 5e-2 * max(np.linalg.norm(ob), 1e-12)
