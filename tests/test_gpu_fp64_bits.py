"""The FP64 path's velocities and equilibria with a shared, corrected reciprocal against the oracle, bit
for bit: random states, zero momenta, and magnitudes from one end of the exponent range to the other
(where the kernels take the plain division)."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def _fields(rng, shape, scale):
    rho = rng.uniform(0.05, 2.0, shape) * scale
    m = [rho * rng.uniform(-1.5, 1.5, shape) for _ in range(2)]
    for f in m:
        f[rng.uniform(size=shape) < 0.1] = 0.0
    p = rng.uniform(0.01, 2.0, shape) * scale
    return rho, m, p


@pytest.mark.parametrize("scale", [1.0, 1e-150, 1e150, 1e-250, 1e-300])
@pytest.mark.parametrize("omega", [1.0, 1.4])
def test_d2q4_steps_equal_oracle_bits(scale, omega):
    from paper_1504_07034_gb300.solver import Solver
    nx, ny = 96, 61
    rho, (mx, my), p = _fields(np.random.default_rng(5), (ny, nx), scale)
    U = np.stack([rho, mx, my, p / 0.4 + 0.5 * (mx * (mx / rho) + my * (my / rho))])
    o = oracle.Oracle(oracle.D2Q4, nx, ny, lam=9.0, dx=0.01, omega=omega, bc=[("periodic", None)] * 4)
    f, _ = o.run(o.init(U), 3)
    s = Solver("d2q4", nx, ny, lam=9.0, dx=0.01, omega=omega, bc=[("periodic", None)] * 4, precision="f64")
    s.set_state(torch.from_numpy(U).cuda(), primitive=False)
    s.step(3)
    got = s.get_distributions().cpu().numpy()
    s.close()
    assert np.array_equal(got, np.asarray(f).reshape(got.shape))


@pytest.mark.parametrize("lattice", ["d1q2", "d1q3"])
@pytest.mark.parametrize("nx, ends", [(1, "transmissive"), (31, "periodic"), (32, "transmissive"), (33, "dirichlet"),
                                      (97, "periodic"), (1000, "transmissive"), (12345, "dirichlet")])
def test_tube_steps_equal_oracle_bits(lattice, nx, ends):
    """The register kernel's tiles: one cell, around a warp, around a tile, many tiles; 1 to 101 steps."""
    from paper_1504_07034_gb300.solver import Solver
    rho, (m, _), p = _fields(np.random.default_rng(nx), (nx,), 1.0)
    U = np.stack([rho, m, p / 0.4 + 0.5 * (m * (m / rho))])
    states = [(0.9, 0.3, 0.8), (1.2, -0.4, 1.1)]
    bc = [(ends, w if ends == "dirichlet" else None) for w in states]
    lam = 8.0
    for omega in (1.0, 1.1):
        o = oracle.Oracle(oracle.D1Q2 if lattice == "d1q2" else oracle.D1Q3, nx, 1, lam=lam, dx=0.01, omega=omega, bc=bc)
        s = Solver(lattice, nx, 1, lam=lam, dx=0.01, omega=omega, bc=bc, precision="f64")
        f = o.init(U)
        s.set_state(torch.from_numpy(U).cuda(), primitive=False)
        for n in (1, 47, 101):
            f, _ = o.run(f, n)
            s.step(n)
            got = s.get_distributions().cpu().numpy()
            assert np.array_equal(got, np.asarray(f).reshape(got.shape)), (omega, n)
        s.close()
