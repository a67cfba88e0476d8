"""The D1Q3 rest population U/3 by a product and a correction against the division, bit for bit: zeros of
both signs, infinities, subnormal and tiny values, the largest ones, and mantissas at random (FP64: the
oracle; FP32: the one-step kernel and the shared-memory batch kernel, which divide)."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def _same(got, want, what):
    bits = {8: np.int64, 4: np.int32}[want.dtype.itemsize]
    got, want = got.ravel(), want.ravel()
    nan = np.isnan(want)
    assert np.array_equal(np.isnan(got), nan), (what, np.flatnonzero(np.isnan(got) != nan)[:5])
    assert np.array_equal(got[~nan].view(bits), want[~nan].view(bits)), what


def cells(small, large):
    """U (3, n): each field in turn takes the special values, the others ordinary ones."""
    rng = np.random.default_rng(4)
    tiny = small * np.array([1, 2, 3, 4, 5, 7, 2 ** 20, 2.0 ** 23 + 1, 2.0 ** 24 - 1, 3 * 2.0 ** 22])
    spec = np.concatenate([[0.0, -0.0, np.inf, -np.inf, np.nan, large, -large, 1.0, 3.0], tiny, -tiny,
                           rng.uniform(0.5, 2.0, 200), rng.uniform(0.5, 2.0, 200) * tiny[-1]])
    U = np.empty((3, 3 * len(spec)))
    U[0], U[1], U[2] = 1.0, 0.25, 2.5
    for k in range(3):
        U[k, k * len(spec):(k + 1) * len(spec)] = spec
    return U


@pytest.mark.filterwarnings("ignore")
@pytest.mark.parametrize("omega", [0.8, 1.4])
def test_fp64_equals_oracle(omega):
    from paper_1504_07034_gb300.solver import Solver
    U = cells(5e-324, 1.7e308)
    n = U.shape[1]
    bc = [("periodic", None)] * 2
    o = oracle.Oracle(oracle.D1Q3, n, 1, lam=9.0, dx=0.01, omega=omega, bc=bc)
    s = Solver("d1q3", n, 1, lam=9.0, dx=0.01, omega=omega, bc=bc, precision="f64")
    s.set_state(torch.from_numpy(U).cuda(), primitive=False)
    f = o.init(U)
    _same(s.get_distributions().cpu().numpy(), f, "equilibria")
    for n in (1, 2):
        s.step(n)
        f, _ = o.run(f, n)
        _same(s.get_distributions().cpu().numpy(), f, n)
    s.close()


_SCRIPT = r"""
import os, sys
sys.path[:0] = [sys.argv[1], os.path.join(sys.argv[1], "tests")]
import numpy as np, torch
from test_gpu_d1q3_thirds import cells
from paper_1504_07034_gb300.solver import Solver
out = []
U = cells(2.0 ** -149, 3e38)
for omega in (0.8, 1.4):
    for k in (1, 2, 3):
        s = Solver("d1q3", U.shape[1], 1, lam=9.0, dx=0.01, omega=omega, bc=[("periodic", None)] * 2, precision="f32")
        s.set_state(torch.from_numpy(U).cuda(), primitive=False)
        s.step(k)
        out.append(s.get_distributions().cpu().numpy().ravel())
        s.close()
np.save(sys.argv[2], np.concatenate(out))
"""


def test_fp32_equals_single_steps(tmp_path):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    script = tmp_path / "thirds.py"
    script.write_text(_SCRIPT)
    res = {}
    for name, env in (("registers", {}), ("single", {"LBRS_1D_BLOCKED": "0"})):
        out = tmp_path / f"{name}.npy"
        subprocess.run([sys.executable, str(script), root, str(out)], check=True, env=dict(os.environ, **env), timeout=300)
        res[name] = np.load(out)
    _same(res["registers"], res["single"], "steps")


@pytest.mark.parametrize("omega", [1.0, 0.8])
def test_fp32_batch_equals_the_shared_memory_kernel(omega):
    from paper_1504_07034_gb300.solver import BatchSolver
    U = cells(2.0 ** -149, 3e38)
    n = U.shape[1]
    res = []
    for tuning in ((256, 4, 32), (256, 4, 96)):       # the second beyond the register kernel's steps per launch
        for steps in (1, 2, 3):
            b = BatchSolver([n, 7], [9.0, 8.0], omega=omega, precision="f32", lattice="d1q3")
            b.tuning = tuning
            b.set_state(torch.from_numpy(np.concatenate([U, U[:, :7]], axis=1)).cuda(), primitive=False)
            b.run([steps, steps])
            res.append(b.get_distributions().cpu().numpy())
            b.close()
    for k in range(3):
        _same(res[k], res[3 + k], k + 1)
