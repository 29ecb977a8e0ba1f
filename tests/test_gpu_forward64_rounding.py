"""Rounding of an FP64 run against the same run in extended precision: the positions a run ends with are those
of exact arithmetic to about their own last place, whatever the number of steps (the update carries its
rounding along, and positions are kept in the caller's units).  For alpha = 0 the kernel functions have a
closed form, so that the reference needs no table; ds and delta are exact."""
import functools

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import swimmer as sw

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1910_12007_gb300 as g  # noqa: E402

DEV = torch.device("cuda:0")
STEPS = 400
THETAS = ((0.0, 0.0, 0.09), (0.0, 0.0, 0.12))


def _stokeslet(delta):
    d = np.longdouble(delta)
    pi4 = 16 * np.arctan(np.longdouble(1))  # 4 pi

    def table(r):
        R = np.sqrt(r * r + d * d)
        return ((np.log(R + d) - d * (R + 2 * d) / (R * (R + d))) / pi4, (R + 2 * d) / (pi4 * R * (R + d) ** 2))

    return table


@functools.lru_cache(maxsize=None)
def _reference(n, theta):
    p = sw.SwimmerParams(n=n, length=(n - 1) / 64.0, dt=2.0 ** -17, k_t=1e3, steps=STEPS, obs_every=STEPS).with_theta(theta)
    X = sw.initial_shape(p).astype(np.longdouble)
    assert X.dtype == np.longdouble and p.ds == 1 / 64 and p.delta == 1.5 / 64
    for k in range(STEPS):
        X = X + np.longdouble(p.dt) * sw.velocity(X, sw.forces(X, p, k * p.dt), _stokeslet(p.delta))
    return X


# the symmetric sum (64 points), the ordered one (65), each with one run per CTA and on clusters
@pytest.mark.parametrize("n", [64, 65])
@pytest.mark.parametrize("batch", [2, 90])
def test_positions_are_those_of_exact_arithmetic(n, batch):
    h = g.swimmer_init(g.SwimmerConfig(n_max=n, b_max=batch, length=(n - 1) / 64.0, dt=2.0 ** -17, k_t=1e3, steps=STEPS,
                                       obs_every=STEPS, precision=g.FP64))
    theta = torch.tensor(THETAS, dtype=torch.float64, device=DEV).repeat(batch // 2, 1)
    _, _, status, state = g.forward_batch_state(h, theta)
    assert (status == 0).all()
    state = state.cpu().numpy()
    moved = 0.0
    for b, t in enumerate(THETAS):
        X = _reference(n, t)
        moved = max(moved, float(np.max(np.abs(X - sw.initial_shape(sw.SwimmerParams(n=n, length=(n - 1) / 64.0))))))
        x = np.asarray(state[b, :, 0] - X[:, 0], dtype=np.float64)
        # what is stored lies below 1/2 and what is returned below 1: rounding of 2^-55 and 2^-54 at
        # most, 3.6e-17 of both together in the mean square of a uniform spread, and as much again
        assert np.sqrt(np.mean(x ** 2)) < 7.2e-17
        assert np.max(np.abs(state[b, :, 1] - X[:, 1])) < 1e-16
    assert moved > 1e-4  # the run is one
    h.close()
