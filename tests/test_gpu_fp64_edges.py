"""FP64 velocities by a corrected reciprocal where that has to leave the way to the division: densities with a
mantissa of all ones, densities and momenta so far apart that the quotient overflows or is subnormal, signed
zeros, infinities; and a large sample of mantissas.  Distributions against the oracle's divisions, bit for
bit (NaN in the same places), and the adaptive run's bound."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

ONES = 1.0 - 2.0 ** -53                            # the mantissa of all ones


def _same(got, want, what):
    got, want = np.asarray(got).ravel(), np.asarray(want).ravel()
    nan = np.isnan(want)
    assert np.array_equal(np.isnan(got), nan), what
    bad = np.flatnonzero(got[~nan].view(np.int64) != want[~nan].view(np.int64))
    assert len(bad) == 0, (what, len(bad), got[~nan][bad[:3]], want[~nan][bad[:3]])


def _edge_cells():
    """(rho, m) pairs."""
    cells = []
    for k in (-3, 0, 1, 40, -60):
        for rho in (ONES, 2 * ONES, ONES / 4, 1.0, 1.0 + 2.0 ** -52):
            cells += [(rho, s * 2.0 ** k) for s in (1, -1)] + [(rho, 1.7 * 2.0 ** k), (rho, ONES * 2.0 ** k)]
    for a, b in ((700, -700), (-700, 700), (500, -540), (-540, 500), (-530, 500), (760, 240), (-760, -240),
                 (1000, 10), (-1060, 3), (30, 600), (251, 3), (-251, 3), (250, 767), (-250, -767)):
        for x, y in ((1.0, 1.0), (1.3, 1.9), (1.9, 1.1), (1.25, -1.75)):
            cells.append((x * 2.0 ** b, y * 2.0 ** a))
    cells += [(1.0, 0.0), (1.0, -0.0), (0.7, -0.0), (-1.0, 0.0), (-1.0, -0.0), (0.0, 1.0), (0.0, 0.0), (-1.5, 0.3),
              (np.inf, 1.0), (1.0, np.inf), (1.0, -np.inf), (5e-324, 5e-324), (np.nan, 1.0), (1.0, np.nan)]
    return np.array(cells).T


def _sample_cells(n):
    """Mantissas at random, and some units from a power of two."""
    rng = np.random.default_rng(11)
    rho, m = rng.uniform(0.5, 2.0, n), rng.uniform(-2.0, 2.0, n)
    near = rng.integers(1, 64, n) * 2.0 ** -53
    rho[::3] = (1.0 - near)[::3]
    rho[1::9] = (1.0 + 2 * near)[1::9]
    m[::2] = np.where(rng.uniform(size=n) < 0.5, 1.0 - near, 1.0 + 4 * near)[::2]
    return rho, m


def _cells(which):
    return _edge_cells() if which == "edges" else _sample_cells(300000)


@pytest.mark.parametrize("which", ["edges", "sample"])
@pytest.mark.parametrize("lattice", ["d2q4", "d1q2"])
@pytest.mark.filterwarnings("ignore")
def test_distributions_equal_the_divisions(lattice, which):
    from paper_1504_07034_gb300.solver import Solver
    rho, m = _cells(which)
    two = lattice == "d2q4"
    n = len(rho)
    E = np.where(np.abs(m) < 1e100, 3.0, np.abs(m)) * np.ones(n)
    # alternating momenta in 2-D, so that each cell has two different quotients
    U = np.stack([rho, m, 0.37 * m[::-1], E] if two else [rho, m, E])
    U = U.reshape((4, 1, n) if two else (3, n))
    nx, ny = n, 1
    bc = [("periodic", None)] * (4 if two else 2)
    # (at omega = 1 the oracle's 0 f is NaN where f is infinite; the kernels return the equilibria there)
    for omega in (1.4,) if which == "edges" else (1.0, 1.4):
        o = oracle.Oracle(oracle.D2Q4 if two else oracle.D1Q2, nx, ny, lam=9.0, dx=0.01, omega=omega, bc=bc)
        s = Solver(lattice, nx, ny, lam=9.0, dx=0.01, omega=omega, bc=bc, precision="f64")
        s.set_state(torch.from_numpy(U).cuda(), primitive=False)
        f = o.init(U)
        _same(s.get_distributions().cpu().numpy(), f, "equilibria")
        s.step(1)
        f, _ = o.run(f, 1)
        _same(s.get_distributions().cpu().numpy(), f, "step")
        s.close()


@pytest.mark.parametrize("rho, m, p", [(ONES, 0.5, 1.0), (2 * ONES, 1.0, 1.0), (ONES, 0.25, ONES), (1.0, 0.3, 1.0),
                                       (2.0 ** -300, 2.0 ** -301, 2.0 ** -300)])
def test_adaptive_bound_equals_the_divisions(rho, m, p):
    from paper_1504_07034_gb300.solver import Solver
    U = np.empty((4, 4, 8))
    U[:] = np.array([rho, m, -0.5 * m, p / 0.4 + 0.5 * (m * (m / rho) * 1.25)])[:, None, None]
    bc = [("periodic", None)] * 4
    o = oracle.Oracle(oracle.D2Q4, 8, 4, lam=9.0, dx=0.01, bc=bc)
    f, lam, t, _ = o.run_adaptive(o.init(U), 3, 0.01, 1.1, 0.0)
    s = Solver("d2q4", 8, 4, lam=9.0, dx=0.01, bc=bc, precision="f64")
    s.set_state(torch.from_numpy(U).cuda(), primitive=False)
    s.step_adaptive(3, 1.1)
    st = s.adaptive_state()
    assert st["t"] == t
    _same(s.get_distributions().cpu().numpy(), f, "adaptive")
    s.close()
