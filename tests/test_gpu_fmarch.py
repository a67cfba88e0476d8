"""FP32 D2Q4 steps at omega != 1 by the marching kernel (two steps a launch) against the tile kernels
that took these grids: bit-identical distributions under every kind of side, recorded moments (through the gradient of a
periodic run) the same.  Grids sit at the edges of the kernel's 30-column strips and of its rows per warp;
the largest takes several rows a warp."""
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
from paper_1504_07034_gb300 import autograd
from paper_1504_07034_gb300.solver import Solver

D0, D1 = ("dirichlet", (0.9, 0.6, -0.2, 0.8)), ("dirichlet", (1.1, -0.3, 0.4, 1.2))
T, P, WL = ("transmissive", None), ("periodic", None), ("wall", None)
SETS = [[P, P, P, P], [T, T, T, T], [D0, T, WL, D1], [P, P, WL, WL], [T, D1, D0, WL], [D1, D0, P, P], [T, T, P, P],
        [D0, D1, T, D0]]
SHAPES = [(1, 2), (2, 3), (29, 2), (30, 5), (31, 4), (61, 33), (130, 47), (700, 645), (3, 65540)]
rng = np.random.default_rng(9)
out = []
for bc in SETS:
    for nx, ny in SHAPES:
        W = np.stack([1 + rng.random((ny, nx)), rng.uniform(-.3, .3, (ny, nx)), rng.uniform(-.3, .3, (ny, nx)),
                      1 + rng.random((ny, nx))])
        s = Solver("d2q4", nx, ny, lam=4.0, omega=1.5 if nx % 2 else 0.7, dx=1.0 / nx, bc=bc, precision="f32")
        s.set_state(torch.from_numpy(W).cuda())
        for n in (2, 3, 7, 40):
            s.step(n)
            out.append(s.get_distributions().cpu().numpy().ravel())
        s.close()
for nx, ny in [(3, 2), (31, 33), (60, 47)]:
    s = Solver("d2q4", nx, ny, lam=4.0, omega=1.3, dx=1.0 / nx, bc=[P] * 4, precision="f32")
    U0 = torch.from_numpy(np.stack([1 + rng.random((ny, nx)), rng.uniform(-.3, .3, (ny, nx)),
                                    rng.uniform(-.3, .3, (ny, nx)), 3 + rng.random((ny, nx))])).float().cuda()
    U0.requires_grad_(True)
    U = autograd.run(U0, s, 13)
    (U[0] ** 2).sum().backward()
    out += [U.detach().cpu().numpy().ravel(), U0.grad.cpu().numpy().ravel()]
    s.close()
np.save(sys.argv[2], np.concatenate(out))
"""


def test_march_equals_tiles(tmp_path):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    script = tmp_path / "fmarch.py"
    script.write_text(_SCRIPT)
    res = {}
    for name, env in (("march", {}), ("off", {"LBRS_F32_FMARCH": "0"})):
        out = tmp_path / f"{name}.npy"
        subprocess.run([sys.executable, str(script), root, str(out)], check=True, env=dict(os.environ, **env), timeout=600)
        res[name] = np.load(out)
    assert np.all(np.isfinite(res["off"]))
    assert np.array_equal(res["march"], res["off"]), np.max(np.abs(res["march"] - res["off"]))
