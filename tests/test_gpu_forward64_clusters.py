"""FP64 runs on clusters of SMs, launched many times over: the CTAs of a cluster write into each other's
shared memory from the first step of a launch on, so that a launch in which one of them started late would
give other numbers than the next."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1910_12007_gb300 as g  # noqa: E402

DEV = torch.device("cuda:0")


# clusters of 16 and 8 SMs (64, 130 points), of 4 and 2 (16 and 8 points), and more runs, whose clusters are smaller
@pytest.mark.parametrize("n,batch", [(64, 1), (64, 9), (130, 5), (130, 30), (16, 1), (8, 2), (64, 70)])
def test_repeated_cluster_launches_agree(n, batch):
    h = g.swimmer_init(g.SwimmerConfig(n_max=n, b_max=100, dt=1e-8, steps=3, obs_every=1, precision=g.FP64))
    b = torch.arange(100, dtype=torch.float64, device=DEV)
    theta = torch.stack([0.5 + 0.02 * b, 0.1 * torch.sin(b), 0.09 + 0.01 * torch.cos(b)], 1).contiguous()
    few = theta[:batch].contiguous()
    first = g.forward_batch(h, few)
    assert (first[2] == 0).all()
    # one run per CTA: the sums are split otherwise, so rounding of three steps
    whole = g.forward_batch(h, theta)
    assert (first[0] - whole[0][:batch]).abs().max() <= 1e-14
    for _ in range(100):
        got = g.forward_batch(h, few)
        assert all(torch.equal(a, r) for a, r in zip(got, first))
    h.close()
