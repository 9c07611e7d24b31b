"""The column sums of squares (column scales, column norms) with one CTA and with two per SM (more than 32
columns for each SM): every column's sum is its own, so the columns of a wide matrix have the bits
they have in a narrow one (no tolerance)."""
import pytest

torch = pytest.importorskip("torch")
from test_gpu_parity import K  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 15, 16, 255, 257, 1000])
@pytest.mark.parametrize("extra", [0, 1, 40])
def test_wide_columns_have_the_narrow_ones_bits(rows, extra):
    n = 32 * torch.cuda.get_device_properties(0).multi_processor_count   # the last width with one
    g = torch.Generator("cuda").manual_seed(rows)
    W = torch.randn((rows, n + extra), device="cuda", generator=g)
    h = torch.rand(n + extra, device="cuda", generator=g) + 0.5

    def scales(lo, hi):
        w = W[:, lo:hi].contiguous()
        s = torch.empty(hi - lo, device="cuda")
        K().kq_compute_scales(w, torch.diag(h[lo:hi]), None, s, None)
        norms = torch.empty(hi - lo, dtype=torch.float64, device="cuda")
        ws = torch.empty(K().kq_biip_stats_workspace(rows, hi - lo), dtype=torch.uint8, device="cuda")
        K().kq_biip_stats(w, None, None, torch.zeros(4, dtype=torch.float64, device="cuda"), ws)
        norms.copy_(ws[:8 * (hi - lo)].view(torch.float64))              # the squared column norms
        return s, norms

    whole, parts = scales(0, n + extra), [scales(0, 777), scales(777, n), scales(n, n + extra)] if extra else [scales(0, 777), scales(777, n)]
    for k in (0, 1):
        assert torch.equal(whole[k], torch.cat([p[k] for p in parts]))
