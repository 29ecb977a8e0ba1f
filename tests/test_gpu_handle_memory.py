"""Device memory of a handle: a table per sample in its own precision, the build's scratch, little else."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1910_12007_gb300 as g  # noqa: E402


@pytest.mark.parametrize("precision,table", [(g.FP64, 24 * 32 * 7 * 16), (g.FP32C, 24 * 64 * 24)])
def test_memory_of_a_handle(precision, table):
    B, n = 16384, 64
    g.swimmer_init(g.SwimmerConfig(n_max=n, b_max=1, steps=1, obs_every=1, precision=precision)).close()
    before = torch.cuda.mem_get_info()[0]
    h = g.swimmer_init(g.SwimmerConfig(n_max=n, b_max=B, steps=1, obs_every=1, precision=precision))
    used = before - torch.cuda.mem_get_info()[0]
    h.close()
    # what the header states, and the allocator's granules of 2 MB
    scratch = 4096 * (8 * 1920 + 16) * 8
    assert B * table + scratch <= used <= B * (table + 1024 + 8 * n) + scratch + (1 << 28)
