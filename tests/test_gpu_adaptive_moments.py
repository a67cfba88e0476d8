"""Adaptive lambda on the moments (FP32, omega = 1), two steps a launch, against one storing step a launch:
bit-identical distributions and records under every side set without Dirichlet states (and one with, which
keeps the storing steps), on ragged and tiny grids, for calls of odd and even numbers of steps, across the
run's end and after it."""
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

T, P, R = ("transmissive", None), ("periodic", None), ("wall", None)
SETS = [[T, T, T, T], [P, P, P, P], [T, T, R, R], [P, P, R, T], [T, T, P, P], [("dirichlet", (1.0, 0.4, 0.0, 1.0)), T, R, T], [P, P, R, R]]
SHAPES = [(1, 2), (3, 2), (16, 32), (33, 17), (131, 45), (260, 70)]
rng = np.random.default_rng(5)
out = []
for bc in SETS:
    for nx, ny in SHAPES:
        W = np.stack([1 + rng.random((ny, nx)), rng.uniform(-.3, .3, (ny, nx)), rng.uniform(-.3, .3, (ny, nx)),
                      1 + rng.random((ny, nx))])
        dx = 1.0 / nx
        for t_final in (0.0, 13.2 * dx / 3.4, 29.7 * dx / 3.4):
            s = Solver("d2q4", nx, ny, lam=3.4, dx=dx, bc=bc, precision="f32")
            s.set_state(torch.from_numpy(W).cuda())
            for n in (8, 9, 1, 16, 7, 12):
                s.step_adaptive(n, 1.1, t_final)
                st = s.adaptive_state()
                out.append(np.array([st["t"], st["lambda"], st["steps"], st["done"]], float))
                out.append(s.get_distributions().double().cpu().numpy().ravel())
            s.close()
np.save(sys.argv[2], np.concatenate(out))
"""


def test_chains_equal_storing_steps(tmp_path):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    script = tmp_path / "adaptive.py"
    script.write_text(_SCRIPT)
    res = {}
    for name, env in (("chains", {}), ("storing", {"LBRS_F32_ADAPT_MOMENTS": "0"})):
        out = tmp_path / f"{name}.npy"
        subprocess.run([sys.executable, str(script), root, str(out)], check=True, env=dict(os.environ, **env), timeout=600)
        res[name] = np.load(out)
    assert np.all(np.isfinite(res["storing"]))
    assert np.array_equal(res["chains"], res["storing"]), np.max(np.abs(res["chains"] - res["storing"]))
