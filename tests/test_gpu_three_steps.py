"""The three-steps-per-launch tile kernel in the calls that it serves: three to seven steps at omega = 1 (below
the number from which steps go to the moments), three of a call at omega != 1, recording steps.  Distributions
and recorded moments against one step a launch, bit for bit, on grids around the 32 x 12 tiles and 40 x 20 boxes,
under every side set it takes."""
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

D0, D1 = ("dirichlet", (0.9, 0.6, -0.2, 0.8)), ("dirichlet", (1.1, -0.3, 0.4, 1.2))
T, P, WL = ("transmissive", None), ("periodic", None), ("wall", None)
SETS = [[P, P, P, P], [T, T, T, T], [D0, T, WL, D1], [P, P, WL, WL], [T, D1, D0, WL], [D1, D0, P, P]]
SHAPES = [(4, 2), (8, 12), (12, 13), (28, 5), (32, 12), (36, 24), (40, 20), (64, 25), (68, 48), (128, 37), (256, 48), (700, 640)]
rng = np.random.default_rng(3)
out, launches = [], []
for bc in SETS:
    for nx, ny in SHAPES:
        W = np.stack([rng.uniform(0.3, 1.5, (ny, nx)), rng.uniform(-0.8, 0.8, (ny, nx)),
                      rng.uniform(-0.8, 0.8, (ny, nx)), rng.uniform(0.2, 1.5, (ny, nx))])
        for omega in (1.0, 1.4):
            s = Solver("d2q4", nx, ny, lam=7.0, dx=0.01, bc=bc, omega=omega, precision="f32")
            s.set_state(torch.from_numpy(W).cuda())
            for n in (3, 4, 5, 6, 7):
                l0 = s.launch_count
                s.step(n)
                launches.append(s.launch_count - l0)
                out.append(s.get_distributions().cpu().numpy().ravel())
            for n in (3, 5, 6):
                out.append(s.step_record(n).cpu().numpy().ravel())
                out.append(s.get_distributions().cpu().numpy().ravel())
            s.close()
np.savez(sys.argv[2], f=np.concatenate(out), launches=np.array(launches))
"""


def test_three_steps_equal_single_steps(tmp_path):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    script = tmp_path / "three.py"
    script.write_text(_SCRIPT)
    res = {}
    for name, env in (("three", {}), ("single", {"LBRS_F32_FUSE": "0"})):
        out = tmp_path / f"{name}.npz"
        subprocess.run([sys.executable, str(script), root, str(out)], check=True, env=dict(os.environ, **env), timeout=600)
        res[name] = np.load(out)
    assert np.all(np.isfinite(res["single"]["f"]))
    assert np.array_equal(res["three"]["f"], res["single"]["f"])
    # a call of three is one launch, of five two
    three = res["three"]["launches"].reshape(-1, 5)
    assert np.all(three[:, 0] == 1) and np.all(three[:, 2] == 2)
