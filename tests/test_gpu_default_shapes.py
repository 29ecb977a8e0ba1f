"""The launch shapes of a handle that was never tuned, where no tuning table can name them: from six runs per SM
on, flagella of 4 to 7 blocks of 32 points take two-target units at 128 registers a thread."""
import pytest

torch = pytest.importorskip("torch")

import synthetic
from test_gpu_velocity_all_points import N128, _check, _states

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1910_12007_gb300 as g  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("n", [97, 128, 161, 224])
@pytest.mark.parametrize("batch", [800, 1024, 2100])
def test_default_shape_has_the_two_target_lists_bits(n, batch):
    h = g.swimmer_init(g.SwimmerConfig(n_max=n, b_max=batch, dt=1e-8, steps=30, obs_every=10, precision=g.FP32C))
    theta = torch.tensor(synthetic.prior_samples(5, (0.0, -1.0, 0.05), (10.0, 0.2, 0.2), batch), device=DEV)
    got = g.forward_batch_state(h, theta)
    g.swimmer_tuning(h, g.FP32C, [128 | g.SHAPE_WIDE] * 17)
    ref = g.forward_batch_state(h, theta)
    assert (ref[2] == 0).all()
    for a, r in zip(got, ref):
        assert torch.equal(a, r)
    h.close()


# the bounds of test_gpu_velocity_all_points
def test_all_point_velocities_of_the_default_shape():
    th = synthetic.prior_samples(31, (0.0, -1.0, 0.05), (10.0, 0.2, 0.2), 1024)
    th[0] = (1.0, 0.0, 0.1)
    steps = 20000
    s0, s1 = _states(N128, th, steps, 0, 1024)
    for b in (0, 1, 511, 1023):
        err_v, err_f, _, _ = _check(N128, th[b], s0[b], s1[b], steps)
        assert err_v < 1e-4, (b, err_v)
        assert err_f < 1e-3, (b, err_f)
