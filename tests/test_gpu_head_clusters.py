"""FP32 head models on clusters of SMs, from four blocks of 32 points on (with fewer a run stays on one SM):
the same bits as with one run per SM, also in the final state of rows that have no run."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1910_12007_gb300 as g  # noqa: E402

DEV = torch.device("cuda:0")
nan = lambda t: torch.nan_to_num(t, nan=7.0)


# at, above and below an edge of a block, the smallest size on clusters, the proximal point in another block than the head
@pytest.mark.parametrize("nf,nh,swimmers", [(73, 24, 1), (80, 24, 1), (104, 24, 1), (125, 36, 1), (200, 24, 1), (40, 24, 2)])
@pytest.mark.parametrize("batch", [1, 25, 60])
@pytest.mark.parametrize("observed", [g.OBS_HEAD_VELOCITY, g.OBS_HEAD_POINT])
def test_head_models_on_clusters(nf, nh, swimmers, batch, observed):
    points = (nf + nh) * swimmers
    assert (points + 31) // 32 >= 4
    if swimmers == 2 and observed == g.OBS_HEAD_VELOCITY:
        observed = g.OBS_PAIR_DISTANCES
    h = g.swimmer_init(g.SwimmerConfig(n_max=points, b_max=120, dt=1e-9, steps=25, obs_every=8, precision=g.FP32C,
                                       k_t=1e4, delta_over_ds=0.045 * 49, omega=12.0, n_head=nh, obs_kind=observed,
                                       n_swimmers=swimmers, swimmer_distance=0.5))
    b = torch.arange(120, dtype=torch.float64, device=DEV)
    theta = torch.stack([0.5 + 0.02 * b, 0.1 * torch.sin(b), 0.09 + 0.01 * torch.cos(b)], 1).contiguous()
    theta[3, 1] = 13.0
    theta[5, 0] = -1.0
    ref = g.forward_batch_state(h, theta)
    got = g.forward_batch_state(h, theta[:batch].contiguous())
    assert (ref[2] == 0).sum() >= 118 and ref[3][5].isnan().all()
    for a, r in zip(got, ref):
        assert torch.equal(nan(a), nan(r[:batch]))
    obs = nan(ref[0][0]).contiguous()
    la, _ = g.loglik_batch(h, theta[:batch].contiguous(), obs, 0.1)
    lr, _ = g.loglik_batch(h, theta, obs, 0.1)
    assert torch.equal(la, lr[:batch])
    h.close()
