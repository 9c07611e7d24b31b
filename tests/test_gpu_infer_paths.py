"""kq_infer over the forms its kernels take: every transform kernel (registers, clusters of seven and
eight, one CTA), the streamed product with x' from the transform kernel, and the tensor-core
product that takes over when x' does not fit beside the weight ring (many tokens times a long
d_in, or scales that are not 16-byte aligned), at cluster sizes 1 to 8. Against a float64
reference built from the definition, with the tolerance of the other decode tests (1e-5)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from oracle import kronq_oracle as ref  # noqa: E402
from test_gpu_infer import _dev, _layer, K  # noqa: E402

pytestmark = pytest.mark.gpu


def _hadamard(v):
    """H_n v / sqrt(n) along the last axis, by butterflies and the 28-point matrix."""
    n = v.shape[-1]
    a = 28 if n % 28 == 0 else 1
    x = v.reshape(-1, a, n // a)
    h = 1
    while h < n // a:
        x = x.reshape(-1, a, n // a // (2 * h), 2, h)
        x = np.stack((x[..., 0, :] + x[..., 1, :], x[..., 0, :] - x[..., 1, :]), axis=-2)
        h *= 2
    x = x.reshape(-1, a, n // a)
    if a == 28:
        x = np.einsum("ij,bjp->bip", ref.paley28().astype(np.float64), x)
    return x.reshape(v.shape) / np.sqrt(n)


def _want(codes, scale, zero, group, s_x, s_g, su, sv, x):
    d_out, d_in = codes.shape
    g = group or d_in
    q = (codes.reshape(d_out, -1, g).astype(np.float64) - zero[:, :, None]) * scale[:, :, None].astype(np.float64)
    xr = _hadamard(x.astype(np.float64) / s_x * sv)
    return _hadamard(xr @ q.reshape(d_out, d_in).T) * su / s_g


@pytest.mark.parametrize("d_out,d_in,bits,group,B,offset", [
    (512, 14336, 2, 128, 8, 0), (128, 14336, 3, 0, 5, 0), (112, 14336, 8, 128, 4, 0), (256, 28672, 4, 128, 3, 0),
    (64, 32768, 2, 128, 2, 0), (14336, 896, 4, 128, 1, 0), (28, 1792, 4, 128, 1, 0), (28672, 128, 8, 0, 1, 0),
    (1024, 2048, 4, 128, 1, 0), (512, 8192, 2, 128, 1, 0), (16, 16384, 4, 0, 1, 0), (4, 256, 2, 0, 8, 0),
    (128, 128, 4, 128, 3, 1), (256, 256, 2, 128, 8, 1), (448, 512, 8, 0, 1, 1), (112, 896, 3, 128, 7, 1)])
def test_infer_forms(d_out, d_in, bits, group, B, offset):
    codes, scale, zero, s_x, s_g, su, sv = _layer(d_out, d_in, bits, group, d_in + bits)
    x = np.random.default_rng(B).standard_normal((B, d_in)).astype(np.float32)
    want = _want(codes, scale, zero, group, s_x, s_g, su, sv, x)
    packed = torch.empty(K().kq_packed_codes_bytes(d_out, d_in, bits) // 4, dtype=torch.int32, device="cuda")
    K().kq_pack_codes(_dev(codes), bits, packed)

    def place(a):   # `offset` elements past an aligned address
        t = torch.zeros(a.size + offset, dtype=_dev(a).dtype, device="cuda")
        t[offset:] = _dev(a).reshape(-1)
        return t[offset:].view(a.shape)

    y = torch.full((B, d_out), float("nan"), device="cuda")
    ws = torch.empty(K().kq_infer_workspace(B, d_in, d_out), dtype=torch.uint8, device="cuda")
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    K().kq_infer(packed, place(scale), place(zero), d_out, d_in, bits, group, _dev(s_x), _dev(s_g), _dev(su), _dev(sv),
                 _dev(x), y, ws, info=info)
    torch.cuda.synchronize()
    assert K().kq_check(info)[0] == K().KQ_OK
    got = y.cpu().numpy().astype(np.float64)
    for b in range(B):
        assert np.linalg.norm(got[b] - want[b]) <= 1e-5 * np.linalg.norm(want[b]), b
