"""The bounds-checked build on the kernels that step the moments, march, pair and tile tubes: every side kind by
the marching kernel (odd and even grids), internal walls, adaptive chains, recording into a buffer on any float,
the omega != 1 march, FP16 pairs, scalar grids of several windows, lone tubes in narrow and batched windows and in
shared memory, batches, and the checkpointed adjoint.  No checked index may leave its buffer, and the results
must equal the release library's to 1e-5 of the field's scale (the checks change the code around the
arithmetic, and with it where the compiler may fuse a multiply and an add)."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

_SCRIPT = r"""
import ctypes
import sys
import numpy as np
import torch
sys.path[:0] = [sys.argv[1], sys.argv[1] + "/tests"]
from paper_1504_07034_gb300 import abi
from paper_1504_07034_gb300.solver import BatchSolver, Solver
from test_gpu_obstacles import random_obstacle_case

lib = abi.load()
out, names, records = [], [], []


def done(name, *tensors):
    torch.cuda.synchronize()
    w = ctypes.c_uint64(0)
    lib.lbrs_debug_check(ctypes.byref(w))
    if w.value:
        records.append((name, int(w.value) >> 40, int(w.value) & ((1 << 40) - 1)))
    for t in tensors:
        out.append(t.detach().double().cpu().numpy().ravel())
        names.append(name)


T, P, WL = ("transmissive", None), ("periodic", None), ("wall", None)
D = [("dirichlet", (1.0, 0.4, 0.1, 1.0)), ("dirichlet", (0.9, -0.2, 0.0, 0.9))]
rng = np.random.default_rng(1)


def fields(nx, ny):
    return torch.from_numpy(np.stack([rng.uniform(0.8, 1.2, (ny, nx)), rng.uniform(-0.3, 0.3, (ny, nx)),
                                      rng.uniform(-0.3, 0.3, (ny, nx)), rng.uniform(0.8, 1.2, (ny, nx))])).cuda()


SETS = {"periodic": [P] * 4, "clamped": [T] * 4, "mixed": [D[0], T, WL, D[1]], "walls": [P, P, WL, WL], "held": [D[0], D[1], T, T]}
SHAPES = ((1, 2), (2, 3), (59, 5), (60, 9), (64, 17), (65, 40), (121, 33), (122, 70))
for bname, bc in SETS.items():
    for nx, ny in SHAPES:
        for precision, omega in (("f32", 1.0), ("f32u", 1.0), ("f32", 1.4), ("f16neq", 1.4)):
            s = Solver("d2q4", nx, ny, lam=7.0, dx=0.01, bc=bc, omega=omega, precision=precision)
            s.set_state(fields(nx, ny))
            for n in (1, 2, 9, 70):
                s.step(n)
            name = f"{precision}-{omega}-{bname}-{nx}x{ny}"
            res = [s.moments()]
            if precision == "f32":
                buf = torch.zeros(9 * 4 * ny * nx + 1, device="cuda")
                res.append(s.step_record(9, U_hist=buf[1:].view(9, 4, ny, nx)))
                res.append(s.get_distributions())
            done(name, *res)
            s.close()
        if D[0] not in bc and D[1] not in bc:
            s = Solver("d2q4", nx, ny, lam=7.0, dx=0.01, bc=bc, precision="f32")
            s.set_state(fields(nx, ny))
            s.step_adaptive(9, 1.1)
            s.step_adaptive(12, 1.1)
            done(f"adaptive-{bname}-{nx}x{ny}", s.moments())
            s.close()
for k, (nx, ny) in enumerate(((36, 29), (132, 18), (64, 40))):
    for bname in ("periodic", "mixed", "walls_periodic_x"):
        wl = random_obstacle_case(nx, ny, bname, 1.0, seed=7 * k + len(bname), steps=0)
        s = Solver.from_workload(wl, precision="f32")
        s.set_state(torch.from_numpy(wl.prim).cuda())
        for n in (8, 9, 70):
            s.step(n)
        fluid = torch.from_numpy(np.asarray(wl.solid) == 0).cuda()
        done(f"solid-{bname}-{nx}x{ny}", s.moments() * fluid)
        s.close()
S = lambda a, b: ("dirichlet", (a, b, 0.0, 0.0))
for bname, bc in {"profiles": [S(1.0, 0.0), S(-1.0, 0.2), S(1.0, -2.0), T], "periodic": [P] * 4, "clamped": [T] * 4}.items():
    for nx, ny in ((3, 5), (64, 64), (90, 71), (97, 130), (515, 300), (1100, 1000)):
        s = Solver("d2q4s", nx, ny, lam=2.6, dx=1.0 / nx, bc=bc, precision="f32")
        s.set_state(torch.from_numpy(rng.uniform(-0.5, 0.5, (1, ny, nx))).cuda())
        for n in (3, 7, 10, 18):
            s.step(n)
        done(f"scalar-{bname}-{nx}x{ny}", s.get_distributions())
        s.close()
for lattice in ("d1q2", "d1q3"):
    for ends in ("transmissive", "periodic"):
        for precision, omega in (("f32", 1.0), ("f32", 1.3), ("f64", 1.0), ("f64", 1.3)):
            for nx in (1, 5, 33, 65, 257, 1001, 170001, 400003):
                W = np.stack([rng.uniform(0.8, 1.2, nx), rng.uniform(-0.3, 0.3, nx), rng.uniform(0.8, 1.2, nx)])
                s = Solver(lattice, nx, 1, lam=4.5, dx=1.0 / nx, bc=[(ends, None)] * 2, omega=omega, precision=precision)
                s.set_state(torch.from_numpy(W).cuda())
                for n in (1, 7, 20, 40):
                    s.step(n)
                done(f"tube-{lattice}-{ends}-{precision}-{omega}-{nx}", s.moments())
                s.close()
    lengths = [1, 2, 17, 63, 64, 65, 200, 447, 449, 3001]
    for boundary in ("transmissive", "periodic"):
        for omega in (1.0, 1.3):
            for tuning in ((256, 4, 32), (256, 4, 64), (256, 2, 128)):
                b = BatchSolver(lengths, [4.5] * len(lengths), omega=omega, precision="f32", lattice=lattice, boundary=boundary)
                b.tuning = tuning
                n = sum(lengths)
                b.set_state(torch.from_numpy(np.stack([rng.uniform(0.8, 1.2, n), rng.uniform(-0.3, 0.3, n), rng.uniform(0.8, 1.2, n)])).cuda())
                b.run(np.array([5, 0, 70, 33, 1, 64, 65, 32, 31, 100]))
                b.run(np.full(len(lengths), 3))
                done(f"batch-{lattice}-{boundary}-{omega}-{tuning}", b.moments())
                b.close()
for nx, ny in ((60, 36), (61, 31)):
    s = Solver("d2q4", nx, ny, lam=7.0, dx=0.01, bc=[P] * 4, precision="f32")
    s.set_state(fields(nx, ny))
    s.forward_checkpointed(23, 5)
    _, g = s.vjp_loss(torch.ones(ny, nx, dtype=torch.float64, device="cuda"))
    done(f"adjoint-{nx}x{ny}", s.backward_checkpointed(g), s.get_distributions())
    s.close()
np.savez(sys.argv[2], names=np.array(names), debug=lib.lbrs_debug_build(),
         records=np.array([f"{n}: site {s}, index {i}" for n, s, i in records]),
         **{f"a{k}": v for k, v in enumerate(out)})
"""


def test_bounds_checked_build(tmp_path):
    from paper_1504_07034_gb300.build import build
    build()
    debug = build(debug=True)
    script = tmp_path / "cases.py"
    script.write_text(_SCRIPT)
    res = {}
    for name, env in (("debug", {"LBRS_LIBRARY": str(debug)}), ("release", {})):
        out = tmp_path / f"{name}.npz"
        subprocess.run([sys.executable, str(script), ROOT, str(out)], check=True,
                       env=dict(os.environ, LBRS_F32_MARCH="2", **env), timeout=900)
        res[name] = np.load(out)
    dbg, rel = res["debug"], res["release"]
    assert int(dbg["debug"]) == 1 and int(rel["debug"]) == 0
    assert len(dbg["records"]) == 0, list(dbg["records"])[:20]
    assert list(dbg["names"]) == list(rel["names"])
    for k, name in enumerate(rel["names"]):
        a, b = dbg[f"a{k}"], rel[f"a{k}"]
        assert np.all(np.isfinite(b)), name
        assert np.max(np.abs(a - b)) <= 1e-5 * np.max(np.abs(b)), name
