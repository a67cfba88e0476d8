"""The checkpointed driver at omega = 1 (checkpoints of moments) on contexts whose state is not plain."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

NX, NY = 64, 40


def _solver(precision="f32", omega=1.0):
    from paper_1504_07034_gb300.solver import Solver
    s = Solver("d2q4", NX, NY, lam=7.0, dx=0.01, bc=[("periodic", None)] * 4, omega=omega, precision=precision)
    rng = np.random.default_rng(2)
    W = np.stack([rng.uniform(0.5, 1.5, (NY, NX)), rng.uniform(-0.5, 0.5, (NY, NX)),
                  rng.uniform(-0.5, 0.5, (NY, NX)), rng.uniform(0.5, 1.5, (NY, NX))])
    s.set_state(torch.from_numpy(W).cuda())
    return s


@pytest.mark.parametrize("precision, omega", [("f32", 1.0), ("f32", 1.4), ("f64", 1.0)])
def test_adaptive_distributions_are_refused(precision, omega):
    """As lbrs_step refuses them: their lambda is not the context's."""
    from paper_1504_07034_gb300 import abi
    s = _solver(precision, omega)
    s.step_adaptive(5, 1.2)
    with pytest.raises(abi.LbrsError) as e:
        s.forward_checkpointed(9, 3)
    assert e.value.status == abi.LBRS_ESTATE
    s.close()
