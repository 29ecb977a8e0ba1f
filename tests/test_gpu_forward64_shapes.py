"""The FP64 forward kernel's launch shapes against the FP64 oracle and one another: lone runs on a
cluster of CTAs (a CTA owning few points, one or none), the points of a warp's worth and one
more or less, more threads than points, and runs of unequal length in one launch."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import sperm as sp
from oracle import swimmer as sw

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1910_12007_gb300 as g  # noqa: E402

DEV = torch.device("cuda:0")


def _theta(rows):
    return torch.tensor(rows, dtype=torch.float64, device=DEV)


# positions are about 1 and displacements about 1e-5 after 64 steps (the sines are made 32 steps at
# a time); FP64 rounding of a position is 1e-16 per step, of a velocity some 1e-14 of it
TOL = 1e-13


@pytest.mark.parametrize("n,batch", [(3, 1), (8, 2), (31, 1), (32, 3), (33, 1), (64, 5), (65, 1), (100, 40), (129, 9),
                                     (33, 77), (130, 160)])
def test_forward64_matches_oracle(n, batch):
    p = sw.SwimmerParams(n=n, dt=1e-6 if n < 70 else 1e-7, steps=64, obs_every=16)
    rows = [(0.3 + 0.13 * b, -0.2 + 0.01 * (b % 7), 0.08 + 0.001 * (b % 11)) for b in range(batch)]
    some = sorted({0, batch // 2, batch - 1})
    obs, _, xc, st = sw.run_c_batch([p.with_theta(rows[b]) for b in some])
    h = g.swimmer_init(g.SwimmerConfig(n_max=n, b_max=batch, dt=p.dt, steps=p.steps, obs_every=p.obs_every,
                                       precision=g.FP64))
    traj, _, status = g.forward_batch(h, _theta(rows))
    assert (status == 0).all() and np.all(np.asarray(st) == 0)
    assert np.abs(traj.cpu().numpy()[some] - obs).max() < TOL
    h.close()


def test_forward64_short_samples_in_a_cluster():
    # n_max = 128 takes a cluster of 16 for few runs; a sample of 5 points leaves CTAs without any
    ns = [128, 5, 17, 3]
    h = g.swimmer_init(g.SwimmerConfig(n_max=128, b_max=4, ds_fixed=1.0 / 127, dt=1e-7, steps=40, obs_every=20,
                                       precision=g.FP64))
    rows = [(1.0 + b, -0.1, 0.1) for b in range(4)]
    traj, _, status = g.forward_batch(h, _theta(rows), torch.tensor(ns, dtype=torch.int32, device=DEV))
    assert (status == 0).all()
    for b, n in enumerate(ns):
        p = sw.SwimmerParams(n=n, length=(n - 1) / 127, dt=1e-7, steps=40, obs_every=20).with_theta(rows[b])
        obs = sw.run_c_batch([p])[0][0]
        assert np.abs(traj[b].cpu().numpy() - obs).max() < TOL
    h.close()


@pytest.mark.parametrize("batch", [1, 12, 90])
def test_forward64_sperm_in_a_cluster(batch):
    # the head ring's ends lie on different CTAs; a run that diverges stops on all of them
    kw = dict(n_max=74, b_max=batch, length=1.0, delta_over_ds=0.045 * 49, dt=1e-4 / 8, k_t=1e4, omega=4 * math.pi,
              steps=60, obs_every=20, precision=g.FP64, n_head=24, obs_kind=g.OBS_HEAD_VELOCITY)
    rows = [(1.0 + 0.05 * b, 0.9, 0.1) for b in range(batch)]
    h = g.swimmer_init(g.SwimmerConfig(**kw))
    traj, _, status, state = g.forward_batch_state(h, _theta(rows))
    assert (status == 0).all()
    fp = sw.SwimmerParams(n=50, length=1.0, delta_over_ds=0.045 * 49, dt=1e-4 / 8, k_t=1e4, omega=4 * math.pi, steps=60,
                          obs_every=20)
    obs, X, _ = sp.run_numpy(sp.SpermParams(flag=fp).with_theta(rows[-1]))
    # velocities are displacements over 2.5e-4: a position's 1e-16 shows as 1e-12 of them
    assert np.abs(traj[-1].cpu().numpy() - obs).max() < 1e-10 * np.abs(obs).max()
    assert np.abs(state[-1, :, :2].cpu().numpy() - X).max() < 1e-12
    bad = g.swimmer_init(g.SwimmerConfig(**dict(kw, dt=1e-4, steps=400)))
    traj, speed, status = g.forward_batch(bad, _theta(rows))
    assert (status == 1).all() and torch.isnan(speed).all() and torch.isnan(traj[:, -1]).all()
    h.close()
    bad.close()
