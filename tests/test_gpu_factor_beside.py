"""A factor launched a wave of tiles at a time (kq_accum_factor's beside, from 32768 tokens) against
the one launch: the same bits, overwriting and adding, with ragged tokens and features."""
import pytest

torch = pytest.importorskip("torch")
from test_gpu_parity import K  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,d", [(32767, 3584), (32768, 3584), (32801, 3100), (32768, 2600), (33000, 136), (40000, 4744)])
def test_beside_has_the_same_bits(T, d):
    g = torch.Generator("cuda").manual_seed(d)
    A = torch.randn((T, (d + 7) // 8 * 8), device="cuda", generator=g).to(torch.bfloat16)[:, :d]
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    H = [torch.full((d, d), 2.0, device="cuda") for _ in range(2)]
    tr = [torch.zeros(1, dtype=torch.float64, device="cuda") for _ in range(2)]
    for accumulate in (False, True):
        for b in (0, 1):
            K().kq_accum_factor(A, H[b], accumulate=accumulate, trace=tr[b], info=info, beside=bool(b))
        assert K().kq_check(info)[0] == K().KQ_OK
        assert torch.equal(H[0], H[1]) and torch.equal(tr[0], tr[1]), accumulate
