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


def test_mask_set_between_forward_and_backward():
    """The backward pass is the forward run's: a mask set after it changes neither the gradient nor the
    state that the backward pass puts back, in the mask's cells as in the others."""
    res = []
    for masked in (False, True):
        s = _solver()
        s.forward_checkpointed(11, 4)
        end = s.raw_state().cpu().numpy()
        _, g = s.vjp_loss(torch.ones(NY, NX, dtype=torch.float64, device="cuda"))
        s.step(5)
        if masked:
            solid = torch.zeros(NY, NX, dtype=torch.uint8)
            solid[10:20, 12:30] = 1
            s.set_obstacles(solid)
        grad = s.backward_checkpointed(g).cpu().numpy()
        assert np.array_equal(s.raw_state().cpu().numpy(), end)
        res.append(grad)
        s.close()
    assert np.array_equal(res[0], res[1])
