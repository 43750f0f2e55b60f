"""mfwh_solve_fpi of problems in fixed point: b = Pi(0) once and v <- S v + b, against as many
applications of Pi, launched one by one and replayed from graphs."""

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


@pytest.mark.parametrize("update", [_lib.UPDATE_IMPLICIT, _lib.UPDATE_EXPLICIT])
@pytest.mark.parametrize("iters", [1, 2, 3, 8])
def test_iterations_equal_maps(update, iters):
    n, om = (70, 45), np.array([6.1, 9.3, 13.0])
    rng = np.random.default_rng(8)
    shape = (3, n[1] + 1, n[0] + 1)
    f, v = rng.normal(size=shape), rng.normal(size=shape)
    v[:, [0, -1]] = 0.0
    v[:, :, [0, -1]] = 0.0

    def solver():
        return M.Solver(n, (1.0, n[1] / n[0]), om, torch.from_numpy(f).cuda(),
                        filter_mode=_lib.FILTER_TRADITIONAL, filter_update=update)
    s = solver()
    want = torch.from_numpy(v).cuda()
    scale = want.abs().amax().item()
    for _ in range(iters):
        s.apply_Pi(want, want, forced=True)
        scale = max(scale, want.abs().amax().item())
    got = torch.from_numpy(v).cuda()
    s.solve_fpi(got, iters)
    # a map is within n_t^2 / 2 roundings of a step (2^-52 of the levels) of the exact one, the
    # levels at most 8 sum |v| + n_t^2 dt^2 sum |f| (test_gpu_fixed64.py), and the maps that follow
    # amplify it by less than |B^{-1}| sum |w| (1 at the fixed point's frequencies)
    n_t, dt = s.setup["n_t"], s.setup["dt"]
    level = 8.0 * 3 * scale + n_t ** 2 * dt ** 2 * np.abs(f).sum(0).max()
    p, keep = M.make_problem(n, (1.0, n[1] / n[0]), om, None, filter_mode=_lib.FILTER_TRADITIONAL)
    amp = (np.abs(s.setup["B_inv"]) @ np.abs(M.plan_weights(p, n_t, 3)).sum(0)).max()
    bound = 2 * (iters + 1) * amp ** iters * n_t ** 2 * 2.0 ** -52 * level
    assert (got - want).abs().amax().item() <= bound
    g = solver()
    g.set_graphs(True)
    for _ in range(2):   # captured, then replayed
        x = torch.from_numpy(v).cuda()
        g.solve_fpi(x, iters)
        assert torch.equal(x, got)
        steps = g.last_timing()[1]
        assert steps == -(-n_t // 8) * (iters + 1 if iters >= 3 else iters)
    # (the graph of the maps that add is dropped with the others, and made again)
    g.set_graphs(False)
    g.set_graphs(True)
    h = rng.normal(size=shape)
    for t in (s, g):
        t.set_forcing(torch.from_numpy(h).cuda())
    a, b = torch.from_numpy(v).cuda(), torch.from_numpy(v).cuda()
    s.solve_fpi(a, iters)
    g.solve_fpi(b, iters)
    assert torch.equal(a, b)
