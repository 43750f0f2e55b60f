"""The fixed-point kernels in the index-checked build (libmfwh_bc.so): levels, sums, forcing, outputs and
shared memory, at the tile edges of both orders and in the FP64 steps of values without a quantum;
and the pipelined FP64 kernel, which the problems of test_gpu_bounds_check.py no longer reach.  No
fault is recorded and the results are those of the normal build, bit for bit."""

import os
import subprocess
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CASES = r'''
import numpy as np
import torch
import paper_2507_23613_gb300 as M
from paper_2507_23613_gb300 import _lib


def run_cases():
    torch.cuda.set_device(0)
    out, faults = {}, {}
    cases = [
        ("edges", (48, 33), (1.0, 0.7), 3, 1.0, {}),
        ("ragged", (200, 170), (1.0, 1.02), 9, 1.0, dict(c_lo=1.0, c_hi=1.4, interface=0.4,
                                                       layer_axis=0)),
        ("order4", (97, 63), (1.0, 0.66), 2, 1.0, dict(order=4)),
        ("no_quantum", (60, 40), (1.0, 0.7), 2, 1e-300, {}),
        ("no_quantum4", (60, 40), (1.0, 0.7), 2, 1e-300, dict(order=4)),
        ("explicit_filter", (70, 45), (1.0, 0.64), 4, 1.0, dict(filter_update=_lib.UPDATE_EXPLICIT)),
        ("pipelined", (200, 45), (1.0, 4.0), 3, 1.0, dict(time_block=3, tile_shape=5)),
    ]
    for name, n, length, nf, scale, kw in cases:
        om = np.linspace(6.0, 6.0 + 2.5 * (nf - 1), nf) + 0.37
        rng = np.random.default_rng(5)
        f = rng.normal(size=(nf, n[1] + 1, n[0] + 1)) * scale
        v = rng.normal(size=f.shape) * scale
        s = M.Solver(n, length, om, torch.from_numpy(f).cuda(), n_p=2 if nf > 4 else 1,
                     filter_mode=_lib.FILTER_TRADITIONAL, **kw)
        res = []
        for forced in (True, False):
            o = torch.empty(v.shape, dtype=torch.float64, device="cuda")
            s.apply_Pi(torch.from_numpy(v).cuda(), o, forced=forced)
            res.append(o.cpu().numpy())
        x = torch.from_numpy(v).cuda()
        s.solve_fpi(x, 4)
        res.append(x.cpu().numpy())
        out[name] = np.stack(res)
        faults[name] = s.debug_bounds()
        s.close()
    return out, faults
'''

CHILD = CASES + r'''
import sys
out, faults = run_cases()
np.savez(sys.argv[1], **out, **{"faults_" + k: np.array(v) for k, v in faults.items()})
'''


@pytest.mark.gpu
def test_checked_build_records_no_fault_in_fixed_point(tmp_path):
    from paper_2507_23613_gb300 import build
    lib_bc = build.build(bounds_check=True)
    env = dict(os.environ, MFWH_LIBRARY=lib_bc, PYTHONPATH=ROOT)
    dump = str(tmp_path / "checked.npz")
    r = subprocess.run([sys.executable, "-c", CHILD, dump], env=env, cwd=ROOT,
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr
    got = np.load(dump)
    scope = {}
    exec(CASES, scope)
    want, _ = scope["run_cases"]()
    for name, ref in want.items():
        assert int(got["faults_" + name][0]) == 0, (name, got["faults_" + name])
        assert np.array_equal(got[name], ref), (name, np.max(np.abs(got[name] - ref)))


def test_every_array_of_the_fixed_point_kernel_is_checked():
    """Each global array and each buffer in shared memory of k_fx2d has its extent tested (the FP64
    kernels that it stands for had)."""
    src = open(os.path.join(ROOT, "paper_2507_23613_gb300", "csrc", "wave_fx_kernels.cuh")).read()
    for extent in ("g.wpoints)", "8 * g.wpoints)", "tiles * NF * kFxTile)", "g.points)",
                   "2 * kFxStep * ORDER * kFxEX)", "STEPS * kFxTile)", "kTileValues)"):
        assert any("MFWH_IDX(" in line and extent in line
                   for line in src.replace(",\n", ", ").splitlines()), extent
