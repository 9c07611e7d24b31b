"""The factor products on both sides of the rule that shares a tile among a cluster of 4 CTAs (up to
38 tiles and at least 4 chunks of 512 tokens), with ragged tokens and features, a row stride and
accumulation. Small integers: every product and every partial sum is exact in fp32, so the
result is exact whatever the split (no tolerance)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from test_gpu_parity import K  # noqa: E402

pytestmark = pytest.mark.gpu


def _ints(T, d, seed, top=8):
    rng = np.random.default_rng(seed)
    ld = (d + 7) // 8 * 8
    return rng.integers(-top, top + 1, size=(T, ld)).astype(np.float32)


@pytest.mark.parametrize("T,d", [(1, 8), (63, 129), (65, 511), (2100, 1024), (1537, 1400), (1030, 1432), (600, 2048),
                                 (577, 2056), (64, 2304), (1024, 256), (2048, 300), (5000, 129)])
def test_factor_split_exact(T, d):
    a = _ints(T, d, d)
    A = torch.from_numpy(a).cuda().to(torch.bfloat16)[:, :d]
    H = torch.full((d, d), 1.0, device="cuda")
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    K().kq_accum_factor(A, H, accumulate=True, info=info)
    assert K().kq_check(info)[0] == K().KQ_OK
    want = a[:, :d].astype(np.float64).T @ a[:, :d] + 1.0
    assert np.array_equal(H.cpu().numpy(), want.astype(np.float32))


@pytest.mark.parametrize("T,d", [(65, 136), (577, 512), (1100, 768), (130, 1032), (600, 1536), (700, 8)])
def test_drift_split_exact(T, d):
    x, dx = _ints(T, d, d), _ints(T, d, d + 1, top=3)
    X = torch.from_numpy(x).cuda().to(torch.bfloat16)
    Xt = torch.from_numpy(x + dx).cuda().to(torch.bfloat16)
    D = torch.empty((d, d), device="cuda")
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(K().kq_accum_drift_workspace(T, d), dtype=torch.uint8, device="cuda")
    K().kq_accum_drift(Xt, X, D, info=info, ws=ws)
    assert K().kq_check(info)[0] == K().KQ_OK
    assert np.array_equal(D.cpu().numpy(), (dx.astype(np.float64).T @ x).astype(np.float32))
