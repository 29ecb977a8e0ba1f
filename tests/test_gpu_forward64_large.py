"""FP64 runs above 512 points, which a launch with one run per CTA gives 1024 threads: the symmetric sum where eight
of its warps' arrays fit (513, 768 points), every ordered pair where they do not (900, 1024), against the same runs
on clusters."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1910_12007_gb300 as g  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("n,more", [(513, {}), (768, {}), (900, {}), (1024, {}), (600, dict(n_head=24)),
                                    (1000, dict(n_head=24))])
def test_large_runs_agree_with_clusters(n, more):
    B = 80
    if more:
        more = dict(more, omega=12.0, k_t=1e4, delta_over_ds=0.045 * 49, obs_kind=g.OBS_HEAD_POINT)
    h = g.swimmer_init(g.SwimmerConfig(n_max=n, b_max=B, dt=1e-13, steps=3, obs_every=1, precision=g.FP64, **more))
    b = torch.arange(B, dtype=torch.float64, device=DEV)
    theta = torch.stack([0.5 + 0.02 * b, 0.1 * torch.sin(b), 0.09 + 0.01 * torch.cos(b)], 1).contiguous()
    one = g.forward_batch_state(h, theta)
    few = g.forward_batch_state(h, theta[:3].contiguous())
    assert (one[2] == 0).all() and (few[2] == 0).all()
    assert not torch.equal(one[3][0], one[3][1])
    # positions of size 1 after three steps whose sums are split otherwise; forces of them by the same operations,
    # within what a last place of a position changes (2 K / ds and, for the bending, 4 K / ds^4 times 1e-16)
    assert (one[3][:3, :, :2] - few[3][:, :, :2]).abs().max() <= 1e-15
    scale = one[3][:3, :, 2:].abs().max()
    assert (one[3][:3, :, 2:] - few[3][:, :, 2:]).abs().max() <= 1e-6 * scale
    assert (one[0][:3] - few[0]).abs().max() <= 1e-15
    h.close()
