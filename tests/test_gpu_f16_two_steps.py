"""The FP16 non-equilibrium form's two-step kernel against one step a launch: the same bytes (moments,
half-precision parts, scales), on the side sets and grids of the moments-only form's test."""
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
D0, D1 = (0.9, 0.6, -0.2, 0.8), (1.1, -0.3, 0.4, 1.2)
T, P, WL = ("transmissive", None), ("periodic", None), ("wall", None)
SETS = [[P, P, P, P], [T, T, T, T], [("dirichlet", D0), T, WL, ("dirichlet", D1)], [P, P, WL, WL],
        [T, ("dirichlet", D1), ("dirichlet", D0), WL]]
rng = np.random.default_rng(3)
out = []
for bc in SETS:
    for nx, ny in ((1, 2), (5, 3), (33, 17), (32, 16), (64, 40), (97, 50), (300, 31)):
        W = np.stack([rng.uniform(0.8, 1.2, (ny, nx)), rng.uniform(-0.4, 0.4, (ny, nx)),
                      rng.uniform(-0.4, 0.4, (ny, nx)), rng.uniform(0.8, 1.2, (ny, nx))])
        for omega in (1.0, 1.4):
            s = Solver("d2q4", nx, ny, lam=6.0, dx=0.01, bc=bc, omega=omega, precision="f16neq")
            s.set_state(torch.from_numpy(W).cuda())
            for n in (1, 2, 5, 70):
                s.step(n)
                out.append(s.raw_state().cpu().numpy())
            s.close()
np.save(sys.argv[2], np.concatenate(out))
"""


def test_two_step_kernel_equals_single_steps(tmp_path):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    script = tmp_path / "f16.py"
    script.write_text(_SCRIPT)
    res = {}
    for name, env in (("two", {}), ("one", {"LBRS_F16_FUSE": "0"})):
        out = tmp_path / f"{name}.npy"
        subprocess.run([sys.executable, str(script), root, str(out)], check=True, env=dict(os.environ, **env), timeout=600)
        res[name] = np.load(out)
    assert np.array_equal(res["two"], res["one"])
