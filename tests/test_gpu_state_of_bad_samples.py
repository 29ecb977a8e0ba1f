"""The final state of a sample outside the domain or of a run that stops is NaN in every row, in both
precisions, on one SM and on clusters."""
import ctypes

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1910_12007_gb300 as g  # noqa: E402
from paper_1910_12007_gb300._lib import check, lib  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("precision,batch", [(g.FP32C, 10), (g.FP32C, 100), (g.FP64, 10), (g.FP64, 100)])
def test_state_of_samples_without_a_run(precision, batch):
    n = 100
    h = g.swimmer_init(g.SwimmerConfig(n_max=n, b_max=batch, dt=1e-8, steps=4, obs_every=2, precision=precision))
    b = torch.arange(batch, dtype=torch.float64, device=DEV)
    theta = torch.stack([0.5 + 0.02 * b, 0.1 * torch.sin(b), 0.09 + 0.01 * torch.cos(b)], 1).contiguous()
    theta[1, 0] = -1.0          # no such resistance
    theta[2, 1] = float("nan")  # no stiffness
    theta[3, 1] = 11.0          # stops at once
    state = torch.full((batch, n, 4), 7.0, dtype=torch.float64, device=DEV)
    traj = torch.full((batch, 2, 2), 7.0, dtype=torch.float64, device=DEV)
    status = torch.full((batch,), 9, dtype=torch.int32, device=DEV)
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())
    check(lib().forward_batch_state(h.ptr, batch, ptr(theta), None, ptr(traj), None, ptr(status), ptr(state), None))
    torch.cuda.synchronize()
    assert (status[[1, 2, 3]] != 0).all() and (status[4:] == 0).all()
    assert state[1:4].isnan().all() and traj[1:3].isnan().all()
    assert state[0].isfinite().all() and state[4:].isfinite().all()
    h.close()
