"""Device memory of orbit problems: the stored operator entries (12 values per node) exist only in the
precision whose operator reads them."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [300, 1 << 12, 1 << 14])
def test_operator_entries_in_the_working_precision_only(N):
    """A single-precision problem and a double-precision one with a single-precision preconditioner hold
    the same FP64 and FP32 arrays, but for the second's two FP32 staging vectors and for the entries:
    12 values of 8 bytes against 12 of 4."""
    from paper_2509_01855_gb300 import _lib, api
    try:
        api.set_f64_precond(1)
        p64 = api.Problem(_lib.BK_ORBIT, N, torch.float64, 0.0, 20.0, (0.01, 1.5))
    finally:
        api.set_f64_precond(-1)
    p32 = api.Problem(_lib.BK_ORBIT, N, torch.float32, 0.0, 20.0, (0.01, 1.5))
    assert p64.device_bytes() - p32.device_bytes() == 2 * 4 * p64.kkt_len + 12 * (8 - 4) * p64.pitch
