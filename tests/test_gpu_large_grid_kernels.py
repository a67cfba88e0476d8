"""The marching, pairing, window and tube kernels past the 32-bit element range: grids whose planes together hold
more than 2^31 values (and, where the state is one value or four a cell, whose single offsets do).

The states are patchworks of constant states chosen by integer cell coordinates, so that both sides build them
exactly.  Sampled cells, among them the corners and the last rows, are compared with the oracle run on a crop
around each, as far as its steps reach.  FP64 to 1e-12 of the largest value, FP32 to 2e-6 times sqrt(steps / 5),
FP16 parts to 2e-4."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

T, P, WL = ("transmissive", None), ("periodic", None), ("wall", None)
D = ("dirichlet", (1.1, 0.4, 0.0, 1.2))
STATES = np.array([[1.0, 0.3, -0.2, 1.0], [0.5, -0.4, 0.1, 0.6], [0.8, 0.0, 0.5, 1.4]])
SCALAR = np.array([0.7, -0.4, 0.2])
LAM = 4.0


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1504_07034_gb300.build import build
    build()
    oracle.build()


def which(i, j):
    return (i // 37 + j // 53) % 3


def device_fields(table, nx, ny, wall):
    """(K, ny, nx) of table[which], FP32 (the values of the states are rounded once, on both sides)."""
    out = torch.empty((table.shape[1], ny, nx), dtype=torch.float32, device="cuda")
    st = torch.from_numpy(table).float().cuda()
    i = torch.arange(nx, device="cuda")[None, :]
    for j0 in range(0, ny, 2048):
        j = torch.arange(j0, min(j0 + 2048, ny), device="cuda")[:, None]
        idx = (torch.div(i, 37, rounding_mode="floor") + torch.div(j, 53, rounding_mode="floor")) % 3
        out[:, j0:j0 + idx.shape[0]] = st[idx].permute(2, 0, 1)
    if wall:
        out[2, 0] = 0.0
    return out


def crop(c, i, j, steps, table, bc, lattice, omega):
    """Moments of cell (i, j) after `steps` steps from the oracle."""
    nx, ny = c
    m = steps + 1
    i0, i1, j0, j1 = max(0, i - m), min(nx, i + m + 1), max(0, j - m), min(ny, j + m + 1)
    sides = [bc[0] if i0 == 0 else T, bc[1] if i1 == nx else T, bc[2] if j0 == 0 else T, bc[3] if j1 == ny else T]
    jj, ii = np.meshgrid(np.arange(j0, j1), np.arange(i0, i1), indexing="ij")
    W = table.astype(np.float32).astype(np.float64)[which(ii, jj)].transpose(2, 0, 1).copy()
    if bc[2] == WL:
        W[2][jj == 0] = 0.0
    o = oracle.Oracle(lattice, i1 - i0, j1 - j0, lam=LAM, omega=omega, bc=sides, dx=0.01)
    f, _ = o.run(o.init(o.prim_to_cons(W) if lattice == oracle.D2Q4 else W), steps)
    return o.moments(f)[:, j - j0, i - i0]


def samples(nx, ny):
    return [(0, 0), (nx - 1, 0), (0, ny - 1), (nx - 1, ny - 1), (nx - 2, ny - 3), (3, ny - 1), (nx - 1, 4), (nx // 2, ny // 2),
            (nx * 3 // 4, ny - 256), (37 * 300, 53 * 120), (37 * 300 - 1, 53 * 120 - 1), (5, 2), (nx - 1, ny - 2)]


MIXED = [D, T, WL, T]


@pytest.mark.parametrize("precision, omega, nx, ny, bc, steps", [
    ("f32", 1.0, 16384, 8256, MIXED, 9),               # moments march, pairs of columns
    ("f32", 1.0, 16383, 8256, MIXED, 8),               # moments march, odd nx
    ("f32", 1.3, 16383, 8256, MIXED, 4),               # marching collisions on a grid without tensor copies
    ("f32u", 1.0, 23296, 23168, [T, T, T, T], 5),      # offsets beyond 2^31 within the four planes
    ("f16neq", 1.3, 16384, 11008, MIXED, 4),           # pairs of steps, 12 planes of half precision
])
def test_d2q4(precision, omega, nx, ny, bc, steps):
    from paper_1504_07034_gb300.solver import Solver
    values = {"f32": 16, "f32u": 4, "f16neq": 12}[precision] * nx * ny
    assert values > 2 ** 31
    s = Solver("d2q4", nx, ny, lam=LAM, dx=0.01, bc=bc, omega=omega, precision=precision)
    s.set_state(device_fields(STATES, nx, ny, bc[2] == WL))
    s.step(steps)
    s.sync()
    U = s.moments(torch.float32)
    pts = samples(nx, ny)
    got = torch.stack([U[:, j, i] for i, j in pts]).double().cpu().numpy()
    s.close()
    del U
    torch.cuda.empty_cache()
    want = np.array([crop((nx, ny), i, j, steps, STATES, bc, oracle.D2Q4, omega) for i, j in pts])
    tol = 2e-4 if precision == "f16neq" else 2e-6 * np.sqrt(max(steps, 5) / 5)
    err = np.abs(got - want).max(axis=1) / np.abs(want).max()
    assert np.all(err <= tol), dict(zip(pts, err))


def test_d2q4_internal_walls():
    from paper_1504_07034_gb300.solver import Solver
    nx, ny, steps = 16384, 8256, 15
    s = Solver("d2q4", nx, ny, lam=LAM, dx=0.01, bc=MIXED, omega=1.0, precision="f32")
    solid = torch.zeros(ny, nx, dtype=torch.uint8)
    solid[400:600, 300:900] = 1
    solid[ny - 300:ny - 200, nx - 500:nx - 100] = 1
    s.set_obstacles(solid)
    s.set_state(device_fields(STATES, nx, ny, True))
    s.step(steps)
    s.sync()
    U = s.moments(torch.float32)
    # away from the solid cells as without them
    pts = [p for p in samples(nx, ny) if not solid[max(p[1] - 17, 0):p[1] + 18, max(p[0] - 17, 0):p[0] + 18].any()]
    # beside them: a crop with the mask
    near = [(299, 500), (900, 400), (600, 600), (nx - 501, ny - 250), (nx - 99, ny - 201), (nx - 300, ny - 199)]
    got = torch.stack([U[:, j, i] for i, j in pts + near]).double().cpu().numpy()
    s.close()
    del U
    torch.cuda.empty_cache()
    want = [crop((nx, ny), i, j, steps, STATES, MIXED, oracle.D2Q4, 1.0) for i, j in pts]
    m = steps + 1
    for i, j in near:
        jj, ii = np.meshgrid(np.arange(j - m, j + m + 1), np.arange(i - m, i + m + 1), indexing="ij")
        W = STATES.astype(np.float32).astype(np.float64)[which(ii, jj)].transpose(2, 0, 1).copy()
        o = oracle.Oracle(oracle.D2Q4, 2 * m + 1, 2 * m + 1, lam=LAM, bc=[T] * 4, dx=0.01,
                          solid=solid[j - m:j + m + 1, i - m:i + m + 1].numpy())
        f, _ = o.run(o.init(o.prim_to_cons(W)), steps)
        want.append(o.moments(f)[:, m, m])
    want = np.array(want)
    err = np.abs(got - want).max(axis=1) / np.abs(want).max()
    assert len(pts) > 9 and np.all(err <= 2e-6 * np.sqrt(3)), dict(zip(pts + near, err))


def test_scalar_windows():
    from paper_1504_07034_gb300.solver import Solver
    nx, ny, steps = 23296, 23168, 9
    assert 4 * nx * ny > 2 ** 31
    bc = [("dirichlet", (1.0, 0.0, 0.0, 0.0)), T, T, T]
    s = Solver("d2q4s", nx, ny, lam=LAM, dx=0.01, bc=bc, precision="f32")
    s.set_state(device_fields(SCALAR[:, None], nx, ny, False))
    s.step(steps)
    s.sync()
    U = s.moments(torch.float32)
    pts = samples(nx, ny)
    got = torch.stack([U[:, j, i] for i, j in pts]).double().cpu().numpy()
    s.close()
    del U
    torch.cuda.empty_cache()
    want = np.array([crop((nx, ny), i, j, steps, SCALAR[:, None], bc, oracle.D2Q4S, 1.0) for i, j in pts])
    err = np.abs(got - want).max(axis=1) / np.abs(want).max()
    assert np.all(err <= 2e-6 * np.sqrt(steps / 5)), dict(zip(pts, err))


@pytest.mark.parametrize("lattice, precision, omega, nx, steps", [
    ("d1q2", "f32", 1.0, 360000013, 20), ("d1q3", "f32", 1.3, 240000007, 20), ("d1q3", "f32", 1.0, 240000007, 5),
    ("d1q2", "f32", 1.3, 360000013, 3), ("d1q3", "f64", 1.0, 240000007, 20)])
def test_lone_tubes(lattice, precision, omega, nx, steps):
    from paper_1504_07034_gb300.solver import Solver
    assert (6 if lattice == "d1q2" else 9) * nx > 2 ** 31
    dt = torch.float32 if precision == "f32" else torch.float64
    table = STATES[:, [0, 1, 3]].astype(np.float32).astype(np.float64)
    x = torch.arange(nx, device="cuda")
    W = torch.from_numpy(table).to(dt).cuda()[torch.div(x, 101, rounding_mode="floor") % 3].T.contiguous()
    s = Solver(lattice, nx, 1, lam=LAM, dx=0.01, bc=[T, T], omega=omega, precision=precision)
    s.set_state(W)
    del W, x
    s.step(steps)
    s.sync()
    U = s.moments(dt)
    pts = [0, 1, 100, 101, 5000, nx // 3, nx // 2, nx - 1000, nx - 102, nx - 101, nx - 2, nx - 1]
    pts += [nx // 101 // 3 * 202 + k for k in (0, 3, 9)]
    got = torch.stack([U[:, i] for i in pts]).double().cpu().numpy()
    s.close()
    del U
    torch.cuda.empty_cache()
    want = []
    for i in pts:
        i0, i1 = max(0, i - steps - 1), min(nx, i + steps + 2)
        o = oracle.Oracle(oracle.D1Q2 if lattice == "d1q2" else oracle.D1Q3, i1 - i0, 1, lam=LAM, omega=omega, bc=[T, T], dx=0.01)
        f, _ = o.run(o.init(o.prim_to_cons(table[np.arange(i0, i1) // 101 % 3].T.copy())), steps)
        want.append(o.moments(f)[:, i - i0])
    want = np.array(want)
    err = np.abs(got - want).max(axis=1) / np.abs(want).max()
    assert np.all(err <= (1e-12 if precision == "f64" else 2e-6 * np.sqrt(max(steps, 5) / 5))), dict(zip(pts, err))
