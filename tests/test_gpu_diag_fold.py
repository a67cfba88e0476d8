"""Diagnostics' partial records folded by one block: totals, extremes and counts for one cell, one cell a
record, uneven records, and more records than one shared-memory load takes (the form without a workspace)
against sums and extremes of the moments.  Totals: N FP64 additions of terms of about one size, error below
N eps of the sum of magnitudes, with the totals' own sums in other orders on both sides: 2 N eps.  Counts
and the density's minimum are exact."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _state(nx, ny):
    g = torch.Generator().manual_seed(nx + ny)
    W = torch.rand(4, ny, nx, generator=g, dtype=torch.float64)
    W[0] += 0.5
    W[1:3] -= 0.5
    W[3] += 1.0
    W[3].view(-1)[:: max(3, nx * ny // 17)] = -1.0
    return W.cuda()


@pytest.mark.parametrize("nx,ny,precision", [(1, 1, "f64"), (608, 1, "f32"), (607, 257, "f64"), (2100, 2051, "f32")])
def test_folded_records(nx, ny, precision):
    from paper_1504_07034_gb300 import abi
    from paper_1504_07034_gb300.solver import Solver
    s = Solver("d2q4", nx, ny, lam=6.0, dx=0.5, bc=[("transmissive", None)] * 4, precision=precision)
    s.set_state(_state(nx, ny))
    U = s.moments(torch.float64).cpu()
    d = abi.lbrs_diag()
    fs = s.get_distributions()
    abi.load().lbrs_diagnostics_noalloc(ctypes.byref(s.cfg), ctypes.c_void_p(fs.data_ptr()), ctypes.byref(d))
    ref = s.diagnostics()
    s.close()
    N = nx * ny
    bad = len(range(0, N, max(3, N // 17)))
    # FP32 states: the read-out sums the four populations in FP64, the diagnostics in FP32 (three roundings)
    one = 2 * N * np.finfo(np.float64).eps + (0.0 if precision == "f64" else 3 * np.finfo(np.float32).eps)
    for k in range(4):
        tol = 0.25 * float(U[k].abs().sum()) * one
        total = 0.25 * float(U[k].sum())
        assert abs(ref["totals"][k] - total) <= tol and abs(d.totals[k] - total) <= tol, k
    assert ref["n_nonphysical"] == bad and d.n_nonphysical == bad
    assert ref["n_subchar"] == d.n_subchar
    assert ref["min_rho"] == d.min_rho and abs(ref["min_rho"] - float(U[0].min())) <= 4 * np.finfo(np.float32).eps
    assert ref["min_p"] == d.min_p and ref["max_lambda_local"] == d.max_lambda_local
