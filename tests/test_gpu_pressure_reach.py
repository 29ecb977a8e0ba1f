"""Pressure at targets farther from the points than r_max, the reach of the velocity's table: the pressure
does not depend on that table and holds at any distance."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import swimmer as sw

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1910_12007_gb300 as g  # noqa: E402
from paper_1910_12007_gb300._lib import check, lib  # noqa: E402

DEV = torch.device("cuda:0")


# the tables end at the octave of 1 + (r_max / delta)^2; the farthest targets lie beyond 24 octaves
@pytest.mark.parametrize("r_max", [0.04, 0.3, 1.0])
@pytest.mark.parametrize("velocity", [False, True])
def test_pressure_beyond_the_velocity_table(r_max, velocity):
    rng = np.random.default_rng(7)
    n, delta = 33, 0.05
    S = np.concatenate([rng.uniform(0, 0.2, (n, 2)), rng.normal(size=(n, 2))], 1)
    r = np.concatenate([[0.0], np.geomspace(1e-3, 3e3, 120)])
    a = rng.uniform(0, 2 * np.pi, r.size)
    grid = np.array([0.1, 0.1]) + r[:, None] * np.stack([np.cos(a), np.sin(a)], 1)
    h = g.swimmer_init(g.SwimmerConfig(n_max=8, b_max=1, dt=1e-6, steps=1, obs_every=1, precision=g.FP64))
    Sd, gd = (torch.tensor(v, device=DEV) for v in (S, grid))
    vel = torch.zeros((r.size, 2), dtype=torch.float64, device=DEV)
    pres = torch.full((r.size,), 7.0, dtype=torch.float64, device=DEV)
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())
    check(lib().swimmer_flow_field(h.ptr, 2.0, delta, r_max, n, ptr(Sd), r.size, ptr(gd),
                                   ptr(vel) if velocity else None, ptr(pres), None))
    torch.cuda.synchronize()
    d = grid[:, None, :] - S[None, :, :2]
    kernel = sw.pressure_kernel(np.hypot(d[..., 0], d[..., 1]), delta)
    products = S[:, 2:] * d
    ref = (products.sum(2) * kernel).sum(1)
    # rounding of the distances, of a kernel value and of 33 sums, against the sizes of the products
    assert np.all(np.abs(pres.cpu().numpy() - ref) <= 64 * 2.3e-16 * (np.abs(products).sum(2) * kernel).sum(1))
    h.close()


def test_pressure_of_targets_that_are_no_numbers():
    h = g.swimmer_init(g.SwimmerConfig(n_max=8, b_max=1, dt=1e-6, steps=1, obs_every=1, precision=g.FP64))
    S = torch.tensor([[0.0, 0.0, 1.0, 0.5]], dtype=torch.float64, device=DEV)
    grid = torch.tensor([[float("nan"), 0.0], [float("inf"), 0.0], [0.1, 0.0]], dtype=torch.float64, device=DEV)
    _, pres = g.swimmer_flow_field(h, 2.0, 0.05, 1.0, S, grid)
    assert pres[:2].isnan().all() and pres[2].isfinite()
    h.close()
