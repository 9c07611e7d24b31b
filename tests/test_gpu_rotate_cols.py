"""The column transform for n = 256 in one pass (up to 4096 columns) against the two passes that
more columns take: the same stages and factors in the same order, so the same bits in the shared
columns (no tolerance)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from test_gpu_parity import K, dev  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ncols", [1, 15, 16, 17, 1000, 4096])
def test_one_pass_has_the_bits_of_two(ncols):
    rng = np.random.default_rng(ncols)
    W = rng.standard_normal((256, 4100)).astype(np.float32)
    sign = dev(np.where(rng.random(256) < 0.5, -1, 1).astype(np.int8), torch.int8)
    s = dev(np.exp(0.3 * rng.standard_normal(256)).astype(np.float32))
    for scale in (None, s):
        for direction in (K().KQ_FWD, K().KQ_INV):
            two, one = dev(W), dev(W[:, :ncols])
            K().kq_rotate_out(two, None, scale, sign, direction)
            K().kq_rotate_out(one, None, scale, sign, direction)
            assert torch.equal(one, two[:, :ncols]), direction
