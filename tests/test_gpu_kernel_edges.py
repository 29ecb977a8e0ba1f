"""Kernels at the edges of their tiles: the surrogate network around its tiles of 16 and 32 rows and its
slices of the batch, the flow field around its tiles of sources and targets and with one output only, the
table build around its slices of 4096 samples, FP32 runs on clusters, and tables at large
alpha."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import brinkmanlet as br
from oracle import mlp as om
from oracle import swimmer as sw

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1910_12007_gb300 as g  # noqa: E402
from paper_1910_12007_gb300._lib import check, lib  # noqa: E402

DEV = torch.device("cuda:0")


def _network(n):
    rng = np.random.default_rng(n)
    params = [(W.astype(np.float32), rng.normal(0, 0.1, b.shape).astype(np.float32)) for W, b in om.init_params(rng)]
    flat = np.concatenate([np.concatenate([W.ravel(), b]) for W, b in params])
    rounded = [(om.bf16_round(W), b.astype(np.float64)) for W, b in params]
    return (flat, rounded, rng.uniform(-1, 1, (n, 5)).astype(np.float32),
            rng.normal(size=(n, 80)).astype(np.float32))


# the oracle's bounds of test_gpu_mlp: FP32 sums, and a BF16 neighbour where an activation lies on the line
@pytest.mark.parametrize("n", [15, 16, 17, 33, 385, 2432, 2433, 4865])
def test_mlp_at_tile_edges(n):
    flat, rounded, x, t = _network(n)
    fl, xd, td = (torch.tensor(v, device=DEV) for v in (flat, x, t))
    y = g.mlp_forward(fl, xd).cpu().numpy()
    ref = om.forward(rounded, x.astype(np.float64), bf16_operands=True)
    assert np.max(np.abs(y - ref)) < 2e-3 * np.max(np.abs(ref))
    grad, loss = g.mlp_backward(fl, xd, td)
    mean = float(np.mean((ref - t) ** 2))
    assert abs(loss.item() - mean) < 1e-4 * mean
    grad, o = grad.cpu().numpy().astype(np.float64), 0
    for W, b in om.backward(rounded, x.astype(np.float64), t.astype(np.float64), bf16_operands=True):
        for part in (W.ravel(), b):
            assert np.max(np.abs(grad[o:o + part.size] - part)) < 2e-3 * np.max(np.abs(part))
            o += part.size


@pytest.mark.parametrize("sources,targets,out", [(1, 1, 3), (2, 255, 3), (511, 257, 3), (512, 64, 1), (513, 64, 2),
                                                 (1025, 1000, 3)])
def test_flow_at_tile_edges(sources, targets, out):
    rng = np.random.default_rng(sources)
    alpha, delta = 2.0, 0.05
    S = np.concatenate([rng.uniform(0, 1, (sources, 2)), rng.normal(size=(sources, 2))], 1)
    grid = rng.uniform(-0.5, 1.5, (targets, 2))
    grid[0] = S[0, :2]
    h = g.swimmer_init(g.SwimmerConfig(n_max=8, b_max=1, dt=1e-6, steps=1, obs_every=1, precision=g.FP64))
    args = [torch.tensor(v, device=DEV) for v in (S, grid)]
    vel = torch.full((targets, 2), 7.0, dtype=torch.float64, device=DEV)
    pres = torch.full((targets,), 7.0, dtype=torch.float64, device=DEV)
    ptr = lambda t, on=True: ctypes.c_void_p(t.data_ptr() if on else None)
    check(lib().swimmer_flow_field(h.ptr, alpha, delta, 3.0, sources, ptr(args[0]), targets, ptr(args[1]),
                                   ptr(vel, out & 1), ptr(pres, out & 2), None))
    torch.cuda.synchronize()
    v, p = sw.flow_field(S[:, :2], S[:, 2:], grid, sw.KernelTable(alpha, delta, 3.0), delta, 1.0)
    for got, ref, on in ((vel, v, out & 1), (pres, p, out & 2)):
        if on:
            assert np.max(np.abs(got.cpu().numpy() - ref)) <= 1e-9 * np.max(np.abs(ref))
        else:
            assert (got == 7.0).all()
    h.close()


@pytest.mark.parametrize("precision", [g.FP64, g.FP32C])
def test_table_build_in_slices(precision):
    # every sample's table is its own: a batch over the edge of a slice equals its parts, bit for bit
    B = 4099
    h = g.swimmer_init(g.SwimmerConfig(n_max=8, b_max=B, dt=1e-5, steps=20, obs_every=10, precision=precision))
    b = torch.arange(B, dtype=torch.float64, device=DEV)
    theta = torch.stack([0.2 + 9.0 * b / B, -0.5 + 0.4 * torch.sin(b), 0.08 + 0.02 * torch.cos(b)], 1).contiguous()
    whole, _, status = g.forward_batch(h, theta)
    assert (status == 0).all()
    for lo, hi in ((0, 5), (4090, 4099)):
        part, _, _ = g.forward_batch(h, theta[lo:hi].contiguous())
        # (few FP64 runs go on clusters, whose sums are split further: rounding of 20 steps)
        assert (part - whole[lo:hi]).abs().max() <= (1e-13 if precision == g.FP64 else 0.0)
    h.close()


CLUSTER_CASES = [(65, {}), (97, {}), (128, {}), (161, {}), (224, {}), (256, {}), (500, {}),
                 (50, dict(n_head=24, omega=12.0)),
                 (50, dict(n_head=24, omega=12.0, n_swimmers=2, swimmer_distance=0.5))]


@pytest.mark.parametrize("n,more", CLUSTER_CASES)
@pytest.mark.parametrize("batch", [1, 25, 60])
def test_runs_on_clusters_equal_runs_on_one_sm(n, more, batch):
    # few runs are spread over clusters of SMs, more than half as many as SMs are not: the same sums in
    # the same order, so the same bits; a row outside the domain and one that diverges among them
    points = (n + more.get("n_head", 0)) * more.get("n_swimmers", 1)
    if more:
        more = dict(more, obs_kind=g.OBS_PAIR_DISTANCES if "n_swimmers" in more else g.OBS_HEAD_VELOCITY,
                    k_t=1e4, delta_over_ds=0.045 * 49)
    h = g.swimmer_init(g.SwimmerConfig(n_max=points, b_max=120, dt=1e-8, steps=25, obs_every=8, precision=g.FP32C,
                                       **more))
    b = torch.arange(120, dtype=torch.float64, device=DEV)
    theta = torch.stack([0.5 + 0.02 * b, 0.1 * torch.sin(b), 0.09 + 0.01 * torch.cos(b)], 1).contiguous()
    theta[3, 1] = 11.0
    theta[5, 0] = -1.0
    nan = lambda t: torch.nan_to_num(t, nan=7.0)
    ref = g.forward_batch_state(h, theta)
    got = g.forward_batch_state(h, theta[:batch].contiguous())
    assert (ref[2] == 0).sum() >= 118
    rows = [k for k in range(batch) if k != 5]  # (no final state is written for a row outside the domain)
    for a, r in zip(got, ref):
        assert torch.equal(nan(a[rows]), nan(r[rows]))
    assert torch.equal(got[2], ref[2][:batch])
    obs = nan(ref[0][0]).contiguous()
    la, _ = g.loglik_batch(h, theta[:batch].contiguous(), obs, 0.1)
    lr, _ = g.loglik_batch(h, theta, obs, 0.1)
    assert torch.equal(la, lr[:batch])
    h.close()


@pytest.mark.parametrize("batch", [9, 40, 70])
def test_uneven_runs_on_clusters_equal_runs_on_one_sm(batch):
    # runs with fewer units than the launch has lists, down to one block
    h = g.swimmer_init(g.SwimmerConfig(n_max=200, b_max=120, ds_fixed=1.0 / 199, dt=1e-8, steps=20, obs_every=5,
                                       precision=g.FP32C))
    b = torch.arange(120, dtype=torch.float64, device=DEV)
    theta = torch.stack([0.5 + 0.02 * b, 0.1 * torch.sin(b), 0.09 + 0.01 * torch.cos(b)], 1).contiguous()
    n_pts = torch.tensor([200, 8, 33, 64, 97, 130, 161, 199] * 15, dtype=torch.int32, device=DEV)
    ref = g.forward_batch(h, theta, n_pts)
    got = g.forward_batch(h, theta[:batch].contiguous(), n_pts[:batch].contiguous())
    assert (ref[2] == 0).all()
    for a, r in zip(got, ref):
        assert torch.equal(a, r[:batch])
    h.close()


@pytest.mark.parametrize("precision,batch", [(g.FP32C, 1), (g.FP32C, 40), (g.FP64, 1), (g.FP64, 30)])
def test_cluster_launches_under_capture(precision, batch):
    h = g.swimmer_init(g.SwimmerConfig(n_max=130, b_max=batch, dt=1e-8, steps=20, obs_every=5, precision=precision))
    b = torch.arange(batch, dtype=torch.float64, device=DEV)
    theta = torch.stack([0.5 + 0.02 * b, 0.1 * torch.sin(b), 0.09 + 0.01 * torch.cos(b)], 1).contiguous()
    eager = g.forward_batch(h, theta)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = g.forward_batch(h, theta)
    for _ in range(2):
        out[0].zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, e) for a, e in zip(out, eager))
    del graph
    h.close()


@pytest.mark.parametrize("alpha", [100.0, 300.0])
def test_tables_of_strongly_screened_flow(alpha):
    # alpha delta up to 6, alpha r up to 570: intervals split in parts, products of large and small Bessel functions
    delta, r_max = 0.02, 1.9
    h = g.swimmer_init(g.SwimmerConfig(n_max=8, b_max=1, dt=1e-6, steps=1, obs_every=1, precision=g.FP64))
    r = np.concatenate([[0.0], np.geomspace(1e-4, 0.99 * r_max, 40)])
    g1, g2 = (v.cpu().numpy() for v in g.swimmer_kernel_eval(h, alpha, delta, r_max, torch.tensor(r, device=DEV)))
    ref = np.array([br.kernel_g(x, alpha, delta) for x in r])
    assert np.max(np.abs(g1 - ref[:, 0])) < 1e-12 * np.max(np.abs(ref[:, 0]))  # g1 crosses zero
    assert np.max(np.abs(g2 / ref[:, 1] - 1.0)) < 1e-12
    h.close()
