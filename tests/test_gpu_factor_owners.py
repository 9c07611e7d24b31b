"""A tile shared among a cluster of 4 CTAs gives the bits that one CTA gives it: the same columns
alone (few tiles: shared) and at the head of a wider matrix (one CTA a tile). Gaussian values with
channel scales: other orders of the chunks' sums give other bits (no tolerance)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from test_gpu_parity import K  # noqa: E402

pytestmark = pytest.mark.gpu


def _tokens(T, d, seed):
    rng = np.random.default_rng(seed)
    x = rng.standard_normal((T, d)) * np.exp(rng.standard_normal(d))
    return torch.from_numpy(x.astype(np.float32)).cuda().to(torch.bfloat16)


@pytest.mark.parametrize("T,d,wide", [(2048, 1024, 2304), (5000, 512, 2304), (7777, 1280, 2048), (2600, 128, 2304)])
def test_shared_factor_tile_has_the_bits_of_one_cta(T, d, wide):
    A = _tokens(T, wide, T + d)
    H, Hw = torch.ones((d, d), device="cuda"), torch.ones((wide, wide), device="cuda")
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    for _ in range(2):   # the second time onto sums
        K().kq_accum_factor(A[:, :d], H, accumulate=True, info=info)
        K().kq_accum_factor(A, Hw, accumulate=True, info=info)
    assert K().kq_check(info)[0] == K().KQ_OK
    assert torch.equal(H, Hw[:d, :d])


@pytest.mark.parametrize("T,d,wide", [(1100, 512, 2048), (3001, 1024, 2048), (700, 256, 1536)])
def test_shared_drift_tile_has_the_bits_of_one_cta(T, d, wide):
    X = _tokens(T, wide, T)
    Xt = (X.float() + 0.1 * _tokens(T, wide, T + 1).float()).to(torch.bfloat16)
    out = []
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    for n in (d, wide):
        x, xt = X[:, :n].contiguous(), Xt[:, :n].contiguous()
        D = torch.empty((n, n), device="cuda")
        ws = torch.empty(K().kq_accum_drift_workspace(T, n), dtype=torch.uint8, device="cuda")
        K().kq_accum_drift(xt, x, D, info=info, ws=ws)
        out.append(D[:d, :d])
    assert K().kq_check(info)[0] == K().KQ_OK
    assert torch.equal(out[0], out[1])
