"""The row transform for n = 28 * 2^k, 448 to 7168, against the general row kernel, which an
unaligned matrix still takes: the same stages, sums and factors in the same order, so the same
bits (no tolerance). Row counts around the rows a CTA takes at a time (512 / 2^k) and beyond the
grid, both directions, with and without scales; one sampled column set against the definition."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from oracle import kronq_oracle as ref  # noqa: E402
from test_gpu_parity import K, dev, host, rel_fro  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scaled", [True, False])
@pytest.mark.parametrize("n,rows", [(448, 1), (448, 33), (896, 17), (1792, 8), (1792, 2500), (3584, 3), (7168, 1),
                                    (7168, 2), (7168, 613)])
def test_same_bits_as_the_general_kernel(n, rows, scaled):
    rng = np.random.default_rng(n + rows)
    W = rng.standard_normal((rows, n)).astype(np.float32)
    sign = dev(np.where(rng.random(n) < 0.5, -1, 1).astype(np.int8), torch.int8)
    s = dev(np.exp(0.3 * rng.standard_normal(n)).astype(np.float32)) if scaled else None
    for direction in (K().KQ_FWD, K().KQ_INV):
        a = dev(W)
        buf = torch.empty(rows * n + 1, device="cuda")
        b = buf[1:].view(rows, n)
        b.copy_(a)
        K().kq_rotate_in(a, None, s, sign, direction)
        K().kq_rotate_in(b, None, s, sign, direction)
        assert torch.equal(a, b), direction
        if direction == K().KQ_FWD:
            cols = np.unique(rng.integers(0, n, 8))
            V = ref.rht_rows(n, sign.cpu().numpy(), cols)
            x = W.astype(np.float64) * (1.0 if s is None else s.cpu().numpy().astype(np.float64))
            assert rel_fro(host(a)[:, cols], x @ V.T) <= 1e-5
