"""Recording steps into a buffer that starts on any float: lbrs_step_record asks for no alignment, and the
marching kernel, which moves pairs of columns as 8-byte words where it can, must do without them where the
buffer does not start on one.  Moments and the state after must equal those of an aligned buffer bit for
bit, in calls on the moments (8 steps and more) and in short ones."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

T, P, WL = ("transmissive", None), ("periodic", None), ("wall", None)
D0, D1 = ("dirichlet", (0.9, 0.6, -0.2, 0.8)), ("dirichlet", (1.1, -0.3, 0.4, 1.2))


@pytest.mark.parametrize("bc", [[P] * 4, [T] * 4, [D0, T, WL, D1]], ids=["periodic", "clamped", "mixed"])
@pytest.mark.parametrize("nx, ny", [(2, 3), (60, 9), (64, 33), (122, 40), (121, 17)])
def test_misaligned_record_buffer(nx, ny, bc):
    from paper_1504_07034_gb300.solver import Solver
    rng = np.random.default_rng(nx)
    W = np.stack([rng.uniform(0.3, 1.5, (ny, nx)), rng.uniform(-0.8, 0.8, (ny, nx)),
                  rng.uniform(-0.8, 0.8, (ny, nx)), rng.uniform(0.2, 1.5, (ny, nx))])
    for n in (3, 8, 9):
        got = []
        for shift in (0, 1, 2, 3):
            s = Solver("d2q4", nx, ny, lam=7.0, dx=0.01, bc=bc, omega=1.0, precision="f32")
            s.set_state(torch.from_numpy(W).cuda())
            buf = torch.full((n * 4 * ny * nx + 8,), -7.0, dtype=torch.float32, device="cuda")
            assert buf.data_ptr() % 256 == 0
            hist = buf[shift:shift + n * 4 * ny * nx].view(n, 4, ny, nx)
            s.step_record(n, U_hist=hist)
            got.append((hist.cpu().numpy().copy(), s.get_distributions().cpu().numpy()))
            rest = torch.cat([buf[:shift], buf[shift + n * 4 * ny * nx:]])
            assert bool((rest == -7.0).all())
            s.close()
        for h, f in got[1:]:
            assert np.array_equal(h, got[0][0]) and np.array_equal(f, got[0][1])
