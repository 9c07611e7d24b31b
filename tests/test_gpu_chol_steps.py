"""Inverse Cholesky with the next diagonal tile updated by the panel kernel (up to 40 blocks of
128) and by a kernel of its own (more): a matrix of 40 blocks, and the same matrix after an
identity block (41 blocks, whose elimination leaves the 40 blocks' arithmetic as it is), give the
same bits (no tolerance). And the smallest sizes of either launch form against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import kqsynth  # noqa: E402
from oracle import kronq_oracle as ref  # noqa: E402
from test_gpu_parity import K, dev, host, rel_fro  # noqa: E402

pytestmark = pytest.mark.gpu


def _inv(H, damp):
    n = H.shape[0]
    Lt = torch.empty((n, n), device="cuda")
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(K().kq_chol_inv_workspace(n), dtype=torch.uint8, device="cuda")
    K().kq_chol_inv(H, damp, Lt, info, ws)
    assert K().kq_check(info)[0] == 0
    return Lt


def test_40_and_41_blocks_same_bits():
    n = 5120
    g = torch.Generator("cuda").manual_seed(5)
    X = torch.randn((2 * n, n), device="cuda", generator=g)
    H = (X.T @ X) / (2 * n)
    big = torch.eye(n + 128, device="cuda")
    big[128:, 128:] = H
    a, b = _inv(H.contiguous(), 0.0), _inv(big, 0.0)
    assert torch.equal(a, b[128:, 128:])
    assert torch.equal(b[:128, :128], torch.eye(128, device="cuda"))


@pytest.mark.parametrize("n", [257, 384, 1024, 1025, 1152])
def test_steps_against_the_oracle(n):
    """Three blocks (the first with a second stream), one super-panel of eight, nine."""
    H = kqsynth.random_spd(n, seed=n, cond_decay=1.0).astype(np.float32)
    Lref = ref.lower_factor(ref.damp(H.astype(np.float64), 0.01))
    assert rel_fro(host(_inv(dev(H), 0.01)), Lref) <= 1e-5   # the tolerance of the other sizes
