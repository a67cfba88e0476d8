"""Scalar D2Q4 steps in shared-memory windows (FP32, omega = 1) against one storing step a launch:
bit-identical distributions on grids that one window holds, grids around its edges and grids of many
windows, under every side set, for calls of one to several hundred steps."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

_SCRIPT = r"""
import sys
sys.path.insert(0, sys.argv[1])
import numpy as np
import torch
from paper_1504_07034_gb300.solver import Solver

T, P = ("transmissive", None), ("periodic", None)
D = lambda a, b: ("dirichlet", (a, b, 0.0, 0.0))
SETS = [[D(1.0, 0.0), D(-1.0, 0.2), D(1.0, -2.0), T], [T, T, T, T], [P, P, P, P], [P, P, D(0.5, -0.4), T],
        [T, D(0.3, 0.1), D(-0.4, 0.5), D(0.2, 0.3)], [T, T, P, P], [D(0.2, 0.1), T, P, P]]
SHAPES = [(1, 1), (2, 3), (5, 64), (64, 64), (63, 61), (65, 66), (128, 96), (127, 131), (300, 40), (41, 517), (515, 260)]
rng = np.random.default_rng(11)
out = []
for bc in SETS:
    for nx, ny in SHAPES:
        W = rng.uniform(-1.2, 1.2, (1, ny, nx))
        s = Solver("d2q4s", nx, ny, lam=2.6, dx=1.0 / nx, bc=bc, precision="f32")
        s.set_state(torch.from_numpy(W).cuda())
        for n in (1, 2, 3, 17, 30, 530 if nx * ny <= 5000 else 33):
            s.step(n)
            out.append(s.get_distributions().cpu().numpy().ravel())
        s.close()
np.save(sys.argv[2], np.concatenate(out))
"""


def test_windows_equal_single_steps(tmp_path):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    script = tmp_path / "scalar.py"
    script.write_text(_SCRIPT)
    res = {}
    for name, env in (("windows", {}), ("single", {"LBRS_F32S_FUSE": "0"})):
        out = tmp_path / f"{name}.npy"
        subprocess.run([sys.executable, str(script), root, str(out)], check=True, env=dict(os.environ, **env), timeout=600)
        res[name] = np.load(out)
    assert np.all(np.isfinite(res["single"]))
    assert np.array_equal(res["windows"], res["single"]), np.max(np.abs(res["windows"] - res["single"]))
