"""The stored operator entries of orbit problems (12 values per node) exist only in the precision whose
operator reads them; the FP64 products of a single-precision problem form theirs."""
import pytest
import torch

from paper_2509_01855_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [300, 1 << 12, 1 << 14])
def test_operator_entries_in_the_working_precision_only(N):
    """A single-precision problem and a double-precision one with a single-precision preconditioner hold
    the same FP64 and FP32 arrays, but for the second's two FP32 staging vectors and for the entries:
    12 values of 8 bytes against 12 of 4."""
    from paper_2509_01855_gb300 import _lib, api
    for d in (torch.float64, torch.float32):   # the first plan of a size also counts the tile tuner's vectors
        api.Problem(_lib.BK_ORBIT, N, d, 0.0, 20.0, (0.01, 1.5)).close()
    try:
        api.set_f64_precond(1)
        p64 = api.Problem(_lib.BK_ORBIT, N, torch.float64, 0.0, 20.0, (0.01, 1.5))
    finally:
        api.set_f64_precond(-1)
    p32 = api.Problem(_lib.BK_ORBIT, N, torch.float32, 0.0, 20.0, (0.01, 1.5))
    assert p64.device_bytes() - p32.device_bytes() == 2 * 4 * p64.kkt_len + 12 * (8 - 4) * p64.pitch


@pytest.mark.parametrize("N", [256, 1000, 1 << 13])
def test_refinement_products_of_a_single_precision_problem(N):
    """With four FP32 solves and FP64 residuals of the Newton system per step, the steps are FP64 ones:
    the solution of the double-precision problem to 1e-9, in at most one step more."""
    from paper_2509_01855_gb300 import _lib, api
    sols = []
    for dtype, refine in ((torch.float64, 0), (torch.float32, 4)):
        prob = api.Problem(_lib.BK_ORBIT, N, dtype, 0.0, 20.0, (0.01, 1.5))
        t, _ = api.Plan(N, t0=0.0, tf=20.0).grid()
        z = prob.pack(*synth.orbit_guess(t.numpy(), 1.5, 20.0))
        info = api.newton_solve(prob, z, tol=1e-10, max_refine=refine)
        assert info["converged"]
        sols.append((prob.split(z), info))
    (want, i64), (got, i32) = sols
    assert i32["kkt_solves"] > i32["iterations"] and i32["iterations"] <= i64["iterations"] + 1
    for a, b in zip(got[:2], want[:2]):
        assert float((a - b).abs().max()) < 1e-9 * max(1.0, float(b.abs().max()))
