"""The marching kernel (FP32 D2Q4 at omega = 1 on the moments, two steps a launch) against one storing
step a launch: bit-identical distributions, moments and recorded moments.

Grids sit at the edges of the kernel's 60-column strips and 64-column windows, of its rows per warp and
of the rows beside a y side; sides of every kind it takes.  Small grids step
on the moments-only form's tiles by default, so the march is also run on all of them
(LBRS_F32_MARCH=2).  The paths run in processes of their own (the switches are read once per process)."""
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
        [T, ("dirichlet", D1), ("dirichlet", D0), WL], [("dirichlet", D1), ("dirichlet", D0), P, P],
        [("dirichlet", D0), ("dirichlet", D1), T, ("dirichlet", D0)]]
SHAPES = [(1, 1), (2, 3), (59, 2), (60, 5), (61, 4), (62, 7), (63, 9), (64, 33), (65, 40), (119, 6), (120, 64),
          (121, 17), (257, 70), (1021, 13), (1200, 131), (3, 65540)]
rng = np.random.default_rng(7)
out = []
for bc in SETS:
    for nx, ny in SHAPES:
        if "wall" in (bc[2][0], bc[3][0]) and ny < 2:
            continue
        W = np.stack([rng.uniform(0.3, 1.5, (ny, nx)), rng.uniform(-0.8, 0.8, (ny, nx)),
                      rng.uniform(-0.8, 0.8, (ny, nx)), rng.uniform(0.2, 1.5, (ny, nx))])
        for precision in ("f32", "f32u"):
            s = Solver("d2q4", nx, ny, lam=7.0, dx=0.01, bc=bc, omega=1.0, precision=precision)
            s.set_state(torch.from_numpy(W).cuda())
            for n in (1, 2, 8, 9, 70):           # single launches, and a captured graph with a remainder
                s.step(n)
                out.append(s.raw_state().cpu().numpy().view(np.float32).ravel())
            if precision == "f32":
                out.append(s.step_record(9).cpu().numpy().ravel())
                out.append(s.raw_state().cpu().numpy().view(np.float32).ravel())
            s.close()
np.save(sys.argv[2], np.concatenate(out))
"""


def test_march_equals_single_steps(tmp_path):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    script = tmp_path / "march.py"
    script.write_text(_SCRIPT)
    res = {}
    for name, env in (("march", {"LBRS_F32_MARCH": "2"}), ("default", {}), ("single", {"LBRS_F32_MARCH": "0", "LBRS_F32_FUSE": "0", "LBRS_F32U_FUSE": "0"})):
        out = tmp_path / f"{name}.npy"
        subprocess.run([sys.executable, str(script), root, str(out)], check=True, env=dict(os.environ, **env), timeout=600)
        res[name] = np.load(out)
    assert np.all(np.isfinite(res["single"]))
    for name in ("march", "default"):
        assert np.array_equal(res[name], res["single"]), (name, np.max(np.abs(res[name] - res["single"])))


_WALLS_SCRIPT = r"""
import os
import sys
sys.path[:0] = [sys.argv[1], os.path.join(sys.argv[1], "tests")]
import numpy as np
import torch
import workloads as W
from test_gpu_obstacles import random_obstacle_case
from paper_1504_07034_gb300.solver import Solver
cases = [W.forward_facing_step(), W.shock_diffraction(n=100)]
for k, (nx, ny) in enumerate(((64, 40), (132, 18), (36, 29), (97, 48), (37, 29))):
    for bcname in ("periodic", "walls_periodic_x", "transmissive", "mixed"):
        cases.append(random_obstacle_case(nx, ny, bcname, 1.0, seed=7 * k + len(bcname), steps=0))
out = []
for wl in cases:
    s = Solver.from_workload(wl, precision="f32")
    s.set_state(torch.from_numpy(wl.prim).cuda())
    for n in (8, 9, 70, 131):                 # even and odd calls, with and without captured graphs
        s.step(n)
        out.append(s.get_distributions().cpu().numpy().ravel())
    s.set_obstacles(None)                     # without walls, and with them again
    s.step(66)
    out.append(s.get_distributions().cpu().numpy().ravel())
    s.set_obstacles(torch.from_numpy(wl.solid))
    s.step(67)
    out.append(s.get_distributions().cpu().numpy().ravel())
    s.close()
np.save(sys.argv[2], np.concatenate(out))
"""


def test_internal_walls_on_the_moments_equal_single_steps(tmp_path):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    script = tmp_path / "walls.py"
    script.write_text(_WALLS_SCRIPT)
    res = {}
    for name, env in (("moments", {}), ("single", {"LBRS_F32_FUSE": "0"})):
        out = tmp_path / f"{name}.npy"
        subprocess.run([sys.executable, str(script), root, str(out)], check=True, env=dict(os.environ, **env), timeout=600)
        res[name] = np.load(out)
    assert np.array_equal(res["moments"], res["single"], equal_nan=True)
