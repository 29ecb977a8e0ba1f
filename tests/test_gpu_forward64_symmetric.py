"""The FP64 kernel's symmetric pair sum (batches with a CTA per run) against the oracle at the edges
of its blocks of 32 points, and mixed with runs that take the ordered sum in one launch."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import swimmer as sw

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1910_12007_gb300 as g  # noqa: E402

DEV = torch.device("cuda:0")
TOL = 1e-13  # absolute, positions about 1: the rounding of 40 steps and of the pair sums


@pytest.mark.parametrize("n,batch", [(32, 100), (31, 80), (64, 200), (63, 100), (128, 330), (126, 90), (150, 160), (256, 80)])
def test_symmetric_sum_matches_oracle(n, batch):
    p = sw.SwimmerParams(n=n, dt=1e-6 if n < 70 else 5e-8, steps=40, obs_every=10)
    rows = [(0.3 + 0.03 * b, -0.2 + 0.01 * (b % 7), 0.08 + 0.001 * (b % 11)) for b in range(batch)]
    some = [0, batch // 2, batch - 1]
    obs, _, _, st = sw.run_c_batch([p.with_theta(rows[b]) for b in some])
    h = g.swimmer_init(g.SwimmerConfig(n_max=n, b_max=batch, dt=p.dt, steps=p.steps, obs_every=p.obs_every,
                                       precision=g.FP64))
    theta = torch.tensor(rows, dtype=torch.float64, device=DEV)
    traj, _, status = g.forward_batch(h, theta)
    assert (status == 0).all()
    assert np.abs(traj.cpu().numpy()[some] - obs).max() < TOL
    again, _, _ = g.forward_batch(h, theta)
    assert torch.equal(traj, again)  # the order of every sum is fixed
    h.close()


def test_symmetric_and_ordered_sums_in_one_launch():
    # n_max = 128: 128 and 62 points take the symmetric sum, 33 and 70 (padded by half) the ordered one
    ns = [128, 33, 70, 62] * 25
    h = g.swimmer_init(g.SwimmerConfig(n_max=128, b_max=100, ds_fixed=1.0 / 127, dt=5e-8, steps=40, obs_every=20,
                                       precision=g.FP64))
    rows = [(1.0 + 0.05 * b, -0.1, 0.1) for b in range(100)]
    traj, _, status = g.forward_batch(h, torch.tensor(rows, dtype=torch.float64, device=DEV),
                                      torch.tensor(ns, dtype=torch.int32, device=DEV))
    assert (status == 0).all()
    for b in (0, 1, 2, 3, 97):
        p = sw.SwimmerParams(n=ns[b], length=(ns[b] - 1) / 127, dt=5e-8, steps=40, obs_every=20).with_theta(rows[b])
        assert np.abs(traj[b].cpu().numpy() - sw.run_c_batch([p])[0][0]).max() < TOL
    h.close()
