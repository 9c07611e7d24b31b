"""The row transforms for n = 28 * 2^k over how many rows a CTA takes (few rows are spread over the grid,
many are taken a tile or several rows at a time, with the factors held or not): a row's result does
not depend on the rows beside it, so a block of rows has the bits it has in the whole matrix."""
import pytest

torch = pytest.importorskip("torch")
from test_gpu_parity import K  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [448, 896, 1792, 3584, 7168, 14336, 28672])
@pytest.mark.parametrize("scaled", [True, False])
def test_rows_do_not_depend_on_their_number(n, scaled):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    g = torch.Generator("cuda").manual_seed(n)
    W = torch.randn((4 * sms + 9, n), device="cuda", generator=g)
    sign = (torch.randint(0, 2, (n,), device="cuda", generator=g) * 2 - 1).to(torch.int8)
    s = torch.exp(0.3 * torch.randn(n, device="cuda", generator=g)) if scaled else None
    for direction in (K().KQ_FWD, K().KQ_INV):
        whole = W.clone()
        K().kq_rotate_in(whole, None, s, sign, direction)
        for lo, hi in [(0, 1), (1, 8), (8, 8 + sms), (3, 4 + sms), (5, 5 + 2 * sms), (0, 2 * sms + 1), (7, 8 + 4 * sms)]:
            part = W[lo:hi].clone()
            K().kq_rotate_in(part, None, s, sign, direction)
            assert torch.equal(part, whole[lo:hi]), (direction, lo, hi)
