"""Codes of rows whose grid has no finite zero (values so small that (max - min) / (2^b - 1) underflows to 0,
or a weight of -infinity): never outside the bits. In the row's last column and in rows with a grid:
clamp(rint(w / scale) + zero), NaN going to 0; the rows beside them are not touched."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from test_gpu_parity import K  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["fp32", "3xtf32"])
@pytest.mark.parametrize("d_in", [4, 128])
@pytest.mark.parametrize("bits,group", [(2, 0), (4, 128), (4, 0)])
def test_underflowed_scale(bits, group, d_in, mode):
    tiny = np.float32(1.401298464324817e-45)
    top = np.float32(2 ** bits - 1)
    W = np.zeros((7, d_in), np.float32)
    W[0, -1], W[2, -1], W[3, 0], W[4, 0], W[6, 0] = tiny, -tiny, tiny, -tiny, -np.inf
    W[5] = np.resize(np.float32([0.5, -1.0, 0.25, 2.0]), d_in)
    xmin, xmax = W.min(1, keepdims=True).clip(max=0), W.max(1, keepdims=True).clip(min=0)
    xmin[1], xmax[1] = -1, 1
    with np.errstate(all="ignore"):
        scale = (xmax - xmin) / top
        zero = np.rint(-xmin / scale)
        q = np.rint(W / scale) + zero                                 # identity L: no updates
    want = np.where(np.isnan(q), 0, np.clip(q, 0, top)).astype(np.uint8)
    assert (scale[[0, 2, 3, 4]] == 0).all()
    d_out = len(W)
    dev = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    Lt = torch.eye(d_in, device="cuda")
    codes = torch.full((d_out, d_in), 77, dtype=torch.uint8, device="cuda")
    sc, ze = torch.empty((d_out, 1), device="cuda"), torch.empty((d_out, 1), dtype=torch.int32, device="cuda")
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    m = K().KQ_TRAIL_FP32 if mode == "fp32" else K().KQ_TRAIL_3XTF32
    ws = torch.empty(K().kq_obs_quantize_workspace(d_out, d_in, 128, m), dtype=torch.uint8, device="cuda")
    K().kq_obs_quantize(dev(W), Lt, bits, group, 128, codes, sc, ze, None, None, ws, mode=m, info=info)
    got = codes.cpu().numpy()
    assert got.max() <= top
    assert np.array_equal(got[[0, 2], -1], want[[0, 2], -1])
    assert np.array_equal(got[[1, 5]], want[[1, 5]])
