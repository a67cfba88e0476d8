"""FP32 tubes by themselves: tiles of 64 to 120 cells in registers, batched windows for long tubes and the
shared-memory kernel for few steps or few cells at omega != 1.

States against one step a launch (LBRS_1D_BLOCKED=0) bit for bit, at lengths beside one, two and three tiles,
beside the lines between the kernels and at ragged last tiles; and no line may be crossed to a slower kernel."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

_STATES = r"""
import sys
sys.path.insert(0, sys.argv[1])
import numpy as np, torch
from paper_1504_07034_gb300.solver import Solver
rng = np.random.default_rng(9)
out = []
LENGTHS = (3, 4, 31, 32, 33, 63, 64, 65, 66, 95, 96, 97, 127, 128, 129, 130, 193, 255, 256, 257, 961, 999, 1000, 49999,
           77825, 150000, 150113)
for lattice in ("d1q2", "d1q3"):
    for ends in ("transmissive", "periodic"):
        for omega in (1.0, 0.8, 1.5):
            for nx in LENGTHS + ((400001,) if omega == 1.0 else (170000, 170077)):
                if nx > 1000 and omega == 1.5:
                    continue
                rho = 1.0 + 0.3 * rng.random(nx)
                u, p = 0.2 * rng.standard_normal(nx), 1.0 + 0.3 * rng.random(nx)
                s = Solver(lattice, nx, 1, lam=4.5, dx=1.0 / nx, bc=[(ends, None)] * 2, omega=omega, precision="f32")
                s.set_state(torch.from_numpy(np.stack([rho, u, p])).cuda())
                for n in (1, 4, 5, 8, 9, 16, 17, 31, 32, 33):
                    s.step(n)
                    f = s.get_distributions().cpu().numpy().ravel()
                    out.append(f if nx <= 1000 else np.concatenate([f[:4000], f[len(f) // 2 - 2000:len(f) // 2 + 2000], f[-4000:], [f.astype(np.float64).sum()]]))
                s.close()
np.save(sys.argv[2], np.concatenate(out))
"""

_TIMES = r"""
import json, sys
sys.path.insert(0, sys.argv[1])
import torch
from paper_1504_07034_gb300.solver import Solver


def best(lattice, omega, nx, n):
    s = Solver(lattice, nx, 1, lam=4.0, dx=1.0 / nx, bc=[("transmissive", None)] * 2, omega=omega, precision="f32")
    x = torch.arange(nx, device="cuda").double() / nx
    s.set_state(torch.stack([1.0 + 0.1 * torch.cos(9 * x), 0.0 * x, 1.0 + 0.1 * torch.sin(5 * x)]))
    for _ in range(3):
        s.step(n)
    ts = []
    for _ in range(25):
        torch.cuda._sleep(400000)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        s.step(n)
        b.record()
        torch.cuda.synchronize()
        ts.append(1e3 * a.elapsed_time(b))
    s.close()
    return min(ts)


print(json.dumps([best(*c) for c in json.loads(sys.argv[2])]))
"""


def _root():
    return os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_states_equal_single_steps(tmp_path):
    script = tmp_path / "states.py"
    script.write_text(_STATES)
    res = {}
    for name, env in (("blocked", {}), ("single", {"LBRS_1D_BLOCKED": "0"})):
        out = tmp_path / f"{name}.npy"
        subprocess.run([sys.executable, str(script), _root(), str(out)], check=True, env=dict(os.environ, **env), timeout=900)
        res[name] = np.load(out)
    assert np.all(np.isfinite(res["single"]))
    assert np.array_equal(res["blocked"], res["single"]), np.max(np.abs(res["blocked"] - res["single"]))


def test_lines_between_the_kernels(tmp_path):
    """100 steps just above a line may take 15 % and 2 us longer than just below it; one step of a long tube at
    omega != 1 at most 0.35 of 32 steps (a launch of the register kernel takes half of them)."""
    import json
    script = tmp_path / "times.py"
    script.write_text(_TIMES)
    pairs = [(lat, w, nx, n) for lat in ("d1q2", "d1q3") for w, lines in ((1.0, (50000, 78000, 400000)), (1.3, (256, 1000, 50000, 170000)))
             for nx in lines for n in (100,)]
    cases = [c for lat, w, nx, n in pairs for c in ((lat, w, nx - 300 if nx > 1000 else nx - 3, n), (lat, w, nx + 300 if nx > 1000 else nx + 3, n))]
    long = [("d1q3", 1.3, 4000000), ("d1q2", 1.3, 4000000), ("d1q3", 1.3, 1000000)]
    cases += [(lat, w, nx, n) for lat, w, nx in long for n in (1, 32)]
    t = np.inf
    for _ in range(3):                           # a busy moment of the machine is not the kernel's
        r = subprocess.run([sys.executable, str(script), _root(), json.dumps(cases)], check=True, capture_output=True, text=True, timeout=600)
        t = np.minimum(t, json.loads(r.stdout.strip().splitlines()[-1]))
        bad = [(c, t[2 * k], t[2 * k + 1]) for k, c in enumerate(pairs) if t[2 * k + 1] > 1.15 * t[2 * k] + 2.0]
        k = 2 * len(pairs)
        bad += [(c, t[k + 2 * i], t[k + 2 * i + 1]) for i, c in enumerate(long) if t[k + 2 * i] > 0.35 * t[k + 2 * i + 1]]
        if not bad:
            break
    assert not bad, bad
