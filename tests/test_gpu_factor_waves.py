"""Which factors are launched a wave at a time beside other work (kq_accum_factor's beside): those whose
equal waves leave at least 16 SMs free, in up to six launches; every other one in one launch."""
import pytest

torch = pytest.importorskip("torch")
from test_gpu_parity import K  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [1024, 2048, 3584, 4096, 7168, 8192, 14336])
def test_waves_only_where_they_free_sms(d):
    T = 32768
    rows, cols = -(-d // 128), -(-d // 256)
    tiles = sum(max(0, rows - 2 * j) for j in range(cols))   # 128 x 256 tiles that touch the lower triangle
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    waves = -(-tiles // sms)
    frees = 4 * tiles > sms and waves <= 6 and sms - -(-tiles // waves) >= 16
    A = torch.ones((T, d), device="cuda", dtype=torch.bfloat16)
    H = torch.empty((d, d), device="cuda")
    n0 = K().launch_count()
    K().kq_accum_factor(A, H, beside=True)
    assert K().launch_count() - n0 == (waves if frees else 1)
    assert bool((H == T).all())
