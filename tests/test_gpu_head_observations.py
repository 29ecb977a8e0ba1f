"""FP32 log-likelihoods of head models where the thread that keeps the sum also updates the proximal
flagellum point (its number is a multiple of the threads of a run): the sum holds the observed head velocities
or pair distances and nothing of that point."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1910_12007_gb300 as g  # noqa: E402

DEV = torch.device("cuda:0")


# flagellum points, swimmers, runs, launch shape (0: the default); point nf - 1 is thread 0's at 128, 256 and 512
# threads, and another's (n = 130, 120)
@pytest.mark.parametrize("nf,swimmers,batch,shape", [(129, 1, 100, 128), (129, 1, 700, 0), (257, 1, 100, 256),
                                                     (257, 1, 90, 128), (129, 2, 80, 128), (513, 1, 100, 512),
                                                     (513, 1, 1, 0), (257, 1, 3, 0), (130, 1, 100, 128),
                                                     (120, 2, 80, 128)])
def test_loglik_is_that_of_the_observations(nf, swimmers, batch, shape):
    nh, steps, every = 16, 12, 3
    # (time steps far below the stability limit at the finest spacing, and stiffnesses that keep the run smooth)
    cfg = g.SwimmerConfig(n_max=swimmers * (nf + nh), b_max=batch, length=1.0, delta_over_ds=4.0, dt=1e-10, k_t=1e3,
                          steps=steps, obs_every=every, precision=g.FP32C, n_head=nh, n_swimmers=swimmers,
                          swimmer_distance=0.5, sigma_ratio=2.0 if swimmers == 2 else 0.0,
                          obs_kind=g.OBS_PAIR_DISTANCES if swimmers == 2 else g.OBS_HEAD_VELOCITY)
    h = g.swimmer_init(cfg)
    if shape:
        g.swimmer_tuning(h, g.FP32C, [shape] * 17)
    b = torch.arange(batch, dtype=torch.float64, device=DEV)
    theta = torch.stack([0.5 + 0.02 * (b % 50), -0.5 + 0.1 * torch.sin(b), 0.09 + 0.01 * torch.cos(b)], 1).contiguous()
    model, _, status = g.forward_batch(h, theta)
    assert (status == 0).all()
    model = model.cpu().numpy()
    assert np.isfinite(model).all()
    rng = np.random.default_rng(nf)
    sigma, ratio = 0.1, cfg.sigma_ratio or 1.0
    obs = model[0] + sigma * rng.normal(size=model[0].shape)
    ll, _ = g.loglik_batch(h, theta, torch.tensor(obs, device=DEV), sigma)
    n_obs = steps // every
    res = (obs - model) / np.array([1.0, ratio])
    J = np.sum(res ** 2, axis=(1, 2))
    ref = -n_obs * (math.log(2 * math.pi * sigma ** 2) + math.log(ratio)) - 0.5 * J / sigma ** 2
    # FP64 sums of eight squares on both sides
    assert np.max(np.abs(ll.cpu().numpy() - ref) / (np.abs(ref) + J / sigma ** 2 + 1.0)) < 1e-13
    h.close()
