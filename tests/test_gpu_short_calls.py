"""Calls of few steps: a kernel of many steps a launch must not take a call that the kernel it replaced does
faster.  Each case is timed with the default choice and with the switch that turns the many-step kernel off
(the least of repeated calls on warm caches, launches queued behind a waiting kernel so that the host's time
is not in it): the default may not take more than 12 % and 1.5 us longer.  The states must agree bit for bit."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

_SCRIPT = r"""
import json, sys
sys.path.insert(0, sys.argv[1])
import numpy as np, torch
from paper_1504_07034_gb300.solver import Solver

T, P = ("transmissive", None), ("periodic", None)
D = lambda a, b: ("dirichlet", (a, b, 0.0, 0.0))


def best(fn):
    for _ in range(3):
        fn()
    ts = []
    for _ in range(25):
        torch.cuda._sleep(400000)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        fn()
        b.record()
        torch.cuda.synchronize()
        ts.append(1e3 * a.elapsed_time(b))
    return min(ts)


def solver(c):
    nx, ny = c["nx"], c["ny"]
    x, y = torch.arange(nx, device="cuda") / nx, torch.arange(ny, device="cuda") / ny
    if c["kind"] == "scalar":
        s = Solver("d2q4s", nx, ny, lam=2.6, dx=1.0 / nx, bc=[D(1.0, 0.0), D(-1.0, 0.2), D(1.0, -2.0), T], precision="f32")
        return s, (torch.cos(7 * x)[None, :] * torch.sin(5 * y)[:, None] + 0.1)[None].double()
    s = Solver("d2q4", nx, ny, lam=5.0, dx=1.0 / ny, bc=[P] * 4 if c.get("periodic") else [T] * 4,
               omega=c.get("omega", 1.0), precision="f32")
    if c["kind"] == "walls":
        solid = torch.zeros(ny, nx, dtype=torch.uint8)
        solid[:ny // 5, nx // 5:] = 1
        s.set_obstacles(solid)
    w = 0.1 * torch.cos(6.2831853 * x)[None, :] * torch.sin(6.2831853 * y)[:, None]
    return s, torch.stack([1.0 + w, 0.3 + w, 0.2 - w, 1.0 - w]).double()


times, states = [], []
for c in json.loads(sys.argv[2]):
    s, W = solver(c)
    n = c["n"]
    hist = s._fields_tensor(n) if c.get("record") else None
    run = (lambda: s.step_record(n, hist)) if c.get("record") else (lambda: s.step(n))
    s.set_state(W)
    run()
    states.append(s.raw_state().cpu().numpy())
    if c.get("record"):
        states.append(hist.cpu().numpy().view(np.uint8).ravel())
    times.append(best(run))
    s.close()
np.savez(sys.argv[3], times=np.array(times), **{f"s{k}": v for k, v in enumerate(states)})
"""


def _compare(tmp_path, cases, off):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    script = tmp_path / "short.py"
    script.write_text(_SCRIPT)
    best = {}
    for attempt in range(3):                     # a busy moment of the machine is not the kernel's
        res = {}
        for name, env in (("default", {}), ("off", off)):
            out = tmp_path / f"{name}{attempt}.npz"
            subprocess.run([sys.executable, str(script), root, json.dumps(cases), str(out)], check=True,
                           env=dict(os.environ, **env), timeout=600)
            res[name] = np.load(out)
            best[name] = np.minimum(best.get(name, np.inf), res[name]["times"])
        for k in res["off"].files:
            if k != "times":
                assert np.array_equal(res["default"][k], res["off"][k]), k
        slow = [(c, round(a, 1), round(b, 1)) for c, a, b in zip(cases, best["default"], best["off"]) if a > 1.12 * b + 1.5]
        if not slow:
            break
    assert not slow, slow


def test_scalar_windows(tmp_path):
    """One window, windows of either size, and calls that leave a short rest after full windows."""
    sizes = [(64, 64, (2, 3, 4)), (80, 80, (2, 3, 4, 5)), (125, 62, (2, 3, 4)), (256, 250, (2, 3)), (768, 768, (2, 3)),
             (1024, 1000, (2, 3, 4, 5, 6, 7, 10)), (2048, 2048, (2, 4, 6, 10, 11)), (3000, 3000, (2, 3, 4, 6, 10, 12, 13, 18)),
             (4096, 4090, (2, 4, 6, 10, 11, 12, 18))]
    _compare(tmp_path, [{"kind": "scalar", "nx": nx, "ny": ny, "n": n} for nx, ny, ns in sizes for n in ns],
             {"LBRS_F32S_WINDOW": "0"})


def test_internal_walls_on_the_moments(tmp_path):
    """Even calls take a storing step before the pairs."""
    sizes = [(960, 320, (6, 7, 8)), (1800, 600, (6, 8)), (2400, 800, (6, 8, 10)), (2048, 1024, (6, 7, 8, 10, 12)),
             (4096, 1024, (6, 8, 10, 12, 14))]
    _compare(tmp_path, [{"kind": "walls", "nx": nx, "ny": ny, "n": n} for nx, ny, ns in sizes for n in ns],
             {"LBRS_F32_MARCH": "0"})


def test_full_collision_march(tmp_path):
    """omega != 1: the marching kernel, three steps a launch on tiles and pairs beside them, recording and not,
    on either side of the rules' lines."""
    plain = [(128, 128, (2, 4, 8)), (800, 800, (2, 4, 6, 8)), (1024, 1024, (2, 4, 5, 6, 12, 24)), (2048, 500, (6, 12))]
    record = [(128, 128, (2, 4, 6)), (800, 800, (2, 6, 12)), (896, 896, (2, 6, 12)), (1024, 1024, (2, 4, 5, 6, 8, 12)),
              (4096, 250, (6, 9))]
    cases = [{"kind": "euler", "periodic": True, "omega": 1.5, "nx": nx, "ny": ny, "n": n, "record": r}
             for r, sizes in ((False, plain), (True, record)) for nx, ny, ns in sizes for n in ns]
    cases += [{"kind": "euler", "omega": 1.5, "nx": 1024, "ny": 1024, "n": n} for n in (2, 6, 12)]
    _compare(tmp_path, cases, {"LBRS_F32_FMARCH": "0"})


def test_repeated_batch_runs():
    """Runs of one launch leave the state in the other buffer each time: repeating one must not take longer than
    repeating a run of two launches (both replay what the first runs planned).  Any sequence of runs, plans and
    tunings equals one run of all steps bit for bit."""
    import time

    import torch
    from paper_1504_07034_gb300.solver import BatchSolver

    def batch(lengths, lattice, omega):
        b = BatchSolver(lengths, [4.0] * len(lengths), precision="f32", lattice=lattice, omega=omega)
        x = torch.arange(int(sum(lengths)), device="cuda").double()
        b.set_state(torch.stack([1.0 + 0.1 * torch.cos(x / 7), 0.1 * torch.sin(x / 5), 1.0 - 0.1 * torch.sin(x / 11)]))
        return b

    b = batch([200] * 8, "d1q2", 1.0)

    def seconds(n, reps=40):
        steps = np.full(8, n)
        for _ in range(4):
            b.run(steps)
        torch.cuda.synchronize()
        best = np.inf
        for _ in range(5):
            t = time.perf_counter()
            for _ in range(reps):
                b.run(steps)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t)
        return best / reps

    one, two = seconds(17), seconds(40)
    for _ in range(2):                           # a busy moment of the machine is not the runtime's
        one, two = min(one, seconds(17)), min(two, seconds(40))
    b.close()
    assert one < 1.1 * two, (one, two)

    lengths = [1, 5, 33, 64, 65, 200, 449, 1000]
    for lattice, omega in (("d1q2", 1.0), ("d1q2", 1.3), ("d1q3", 1.0), ("d1q3", 0.9)):
        a, c = batch(lengths, lattice, omega), batch(lengths, lattice, omega)
        total = np.zeros(len(lengths), dtype=np.int64)
        uneven = np.array([17, 3, 40, 0, 1, 33, 64, 5])
        for k, steps in enumerate((1, 1, 2, 17, 17, 40, 40, uneven, uneven, 17, 31, 32, 33, uneven, 5)):
            steps = np.broadcast_to(steps, total.shape).astype(np.int64)
            a.run(steps)
            total += steps
            if k == 8:
                a.autotune(steps)
                a.tuning = (256, 4, 32)
        c.tuning = (256, 2, 128)              # the shared-memory kernel
        c.run(total)
        assert torch.equal(a.get_distributions(), c.get_distributions()), (lattice, omega)
        a.close()
        c.close()


@pytest.mark.parametrize("lattice, cells, in_registers", [("d1q2", 127, False), ("d1q2", 128, True), ("d1q2", 16, False),
                                                         ("d1q3", 16, True)])
def test_batches_of_tiny_tubes(lattice, cells, in_registers):
    """D1Q2 tubes of few cells step in shared memory (16 steps a launch), others in registers (32), with the same
    bits as by the other kernel (halo 65 is beyond the register kernel's)."""
    import torch
    from paper_1504_07034_gb300.solver import BatchSolver
    count, steps = 50, np.full(50, 40)
    x = torch.arange(count * cells, device="cuda").double()
    W = torch.stack([1.0 + 0.1 * torch.cos(x / 7), 0.1 * torch.sin(x / 5), 1.0 - 0.1 * torch.sin(x / 11)])
    res = []
    for tuning in (None, (256, 2, 65)):
        b = BatchSolver([cells] * count, [4.0] * count, precision="f32", lattice=lattice)
        if tuning:
            b.tuning = tuning
        b.set_state(W)
        n0 = b.launch_count
        b.run(steps)
        launches = b.launch_count - n0
        res.append(b.get_distributions())
        if tuning is None:
            assert launches == (2 if in_registers else 3)
        b.close()
    assert torch.equal(res[0], res[1])


def test_flat_scalar_grids(tmp_path):
    """Grids of few rows fill the windows' rows badly."""
    sizes = [(20000, 8, (10, 40)), (20000, 12, (10,)), (65536, 4, (10, 40)), (65536, 8, (10, 40)), (65536, 16, (10, 40)),
             (65536, 20, (10,)), (200000, 2, (10,)), (200000, 6, (10, 40)), (200000, 16, (10,))]
    _compare(tmp_path, [{"kind": "scalar", "nx": nx, "ny": ny, "n": n} for nx, ny, ns in sizes for n in ns],
             {"LBRS_F32S_WINDOW": "0"})


def test_moments_on_small_grids(tmp_path):
    """Entering and leaving the moments costs two launches, which small odd grids do not win back outside a graph."""
    cases = [{"kind": "euler", "periodic": p, "nx": nx, "ny": ny, "n": n, "record": r}
             for nx, ny in ((65, 65), (130, 130), (257, 64), (201, 201), (128, 128)) for n in (8, 10, 16, 40)
             for p, r in ((True, False), (False, False), (True, True))]
    _compare(tmp_path, cases, {"LBRS_F32_MARCH": "0"})
