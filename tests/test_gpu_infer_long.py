"""kq_infer at the longest input it takes (d_in = 32768) with every number of tokens: six to eight
tokens' x' do not fit one product kernel's shared memory beside the grids, so they go in two halves.
Against a float64 reference built from the definition, with the tolerance of the other decode
tests (1e-5)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from test_gpu_infer import _dev, _layer, K  # noqa: E402
from test_gpu_infer_paths import _want  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_out,bits,group", [(64, 2, 128), (2048, 8, 128), (256, 8, 0), (64, 4, 128)])
@pytest.mark.parametrize("B", [1, 5, 6, 7, 8])
def test_infer_longest_input(d_out, bits, group, B):
    d_in = 32768
    codes, scale, zero, s_x, s_g, su, sv = _layer(d_out, d_in, bits, group, bits)
    x = np.random.default_rng(B).standard_normal((B, d_in)).astype(np.float32)
    want = _want(codes, scale, zero, group, s_x, s_g, su, sv, x)
    packed = torch.empty(K().kq_packed_codes_bytes(d_out, d_in, bits) // 4, dtype=torch.int32, device="cuda")
    K().kq_pack_codes(_dev(codes), bits, packed)
    y = torch.full((B, d_out), float("nan"), device="cuda")
    ws = torch.empty(K().kq_infer_workspace(B, d_in, d_out), dtype=torch.uint8, device="cuda")
    K().kq_infer(packed, _dev(scale), _dev(zero), d_out, d_in, bits, group, _dev(s_x), _dev(s_g), _dev(su), _dev(sv),
                 _dev(x), y, ws)
    got = y.cpu().numpy().astype(np.float64)
    for b in range(B):
        assert np.linalg.norm(got[b] - want[b]) <= 1e-5 * np.linalg.norm(want[b]), b
