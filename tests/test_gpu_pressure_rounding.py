"""Rounding of the pressure kernel's table: a source's pressure is the closed form's (in extended precision) to
a few roundings, as an evaluation of the closed form in FP64 would be."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1910_12007_gb300 as g  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("angle", [0.0, 0.7])
def test_pressure_of_one_source(angle):
    delta = 1.0 / 64
    S = np.array([[0.3, 0.2, 1.0, -0.4]])
    r = np.geomspace(1e-5, 3.0, 20000)
    grid = S[:, :2] + r[:, None] * np.array([[np.cos(angle), np.sin(angle)]])
    h = g.swimmer_init(g.SwimmerConfig(n_max=8, b_max=1, dt=1e-6, steps=1, obs_every=1, precision=g.FP64))
    _, pres = g.swimmer_flow_field(h, 2.0, delta, 4.0, torch.tensor(S, device=DEV), torch.tensor(grid, device=DEV))
    LD = np.longdouble
    d = grid.astype(LD) - S[0, :2]
    D = LD(delta)
    R = np.sqrt(d[:, 0] ** 2 + d[:, 1] ** 2 + D * D)
    kernel = (R * R + R * D + D * D) / (8 * np.arctan(LD(1)) * R ** 3 * (R + D))
    products = d * S[0, 2:]
    err = (pres.cpu().numpy() - products.sum(1) * kernel) / (np.abs(products).sum(1) * kernel)
    # five roundings, two of them of u, on which the kernel depends up to its 3/2nd power: 1.25e-16 in the mean
    # square of uniform spreads, and as much again
    assert float(np.sqrt(np.mean(err ** 2))) < 2.5e-16
    h.close()
