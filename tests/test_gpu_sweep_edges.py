"""The sweep's block kernel (32 rows per CTA, 16 columns per warp) at the edges of its tiles:
row counts around 32, last blocks that end inside a warp's columns or leave warps without any,
aligned and unaligned row strides, and the fused update in both arithmetics. fp32 mode: bit for
bit against the fp32-ordered definition (the contract of KQ_TRAIL_FP32, so no tolerance)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
from oracle import obs_sweep_fp32  # noqa: E402
from test_gpu_parity import _gpu_sweep, _synthetic_lt, K  # noqa: E402

pytestmark = pytest.mark.gpu


def _w(d_out, d_in):
    return (np.random.default_rng(d_out + d_in).standard_normal((d_out, d_in)) * 0.05).astype(np.float32)


@pytest.mark.parametrize("group", [0, 128])
@pytest.mark.parametrize("d_out,d_in", [(1, 1), (31, 15), (33, 17), (32, 127), (65, 129), (2, 144), (95, 257), (64, 272),
                                        (33, 1040)])
def test_block_edges_bit_exact(d_out, d_in, group):
    Wp, Lt = _w(d_out, d_in), _synthetic_lt(d_in, seed=d_in)
    g = _gpu_sweep(Wp, Lt, 3, group)
    c = obs_sweep_fp32(Wp, Lt, 3, group, 128, want_pre_q=True)
    for k in ("codes", "scale", "pre_q"):
        assert np.array_equal(g[k], c[k]), k
    assert np.array_equal(g["zero"], c["zero"].astype(np.int32))


@pytest.mark.parametrize("d_out,d_in", [(33, 144), (65, 272), (31, 1040), (4865, 144)])
def test_block_edges_tensor_core_update(d_out, d_in):
    """3xTF32 mode (fused update on the tensor cores up to 4864 rows): teacher forced, as for
    the other shapes."""
    from sweep_checks import check_teacher_forced
    Wp, Lt = _w(d_out, d_in), _synthetic_lt(d_in, seed=d_in)
    g = _gpu_sweep(Wp, Lt, 4, 128, mode=K().KQ_TRAIL_3XTF32)
    check_teacher_forced(Wp, Lt, g, 4, 128, 128)
