"""GMRES cut off after k columns against the minimal residual over the same Krylov space.

The Gram-Schmidt passes take 1 to 3 columns in forms of their own, more of them in a general one, and
dots in groups of 4 (FP64) or 8 (FP32) columns; a solution that is not 16-byte aligned takes the
element loop. After k steps the relative residual must be the least-squares minimum over
A span{b, Ab, ...}, formed here from an orthonormal basis in FP64, within the accuracy of k backward
stable steps: 1e-9 in FP64, 1e-4 in FP32, far above k eps and far below one step's reduction.
"""
import pytest
import torch

from tests.helpers import from_packed

pytestmark = pytest.mark.gpu


def _least_residual(apply, b, k):
    """min ||b - A V y|| / ||b|| over an orthonormal basis V of the k-dimensional Krylov space."""
    V = [b / b.norm()]
    AV = []
    for _ in range(k):
        w = apply(V[-1])
        AV.append(w.clone())
        for _ in range(2):
            for v in V:
                w = w - (v @ w) * v
        V.append(w / w.norm())
    M = torch.stack(AV, 1).cpu()
    y = torch.linalg.lstsq(M, b.cpu().unsqueeze(1)).solution
    return float((b.cpu().unsqueeze(1) - M @ y).norm() / b.cpu().norm())


@pytest.mark.parametrize("dtype,tol", [(torch.float64, 1e-9), (torch.float32, 1e-4)])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 8, 9])
@pytest.mark.parametrize("off", [0, 1])
def test_residual_after_k_columns_is_minimal(dtype, tol, k, off):
    from oracle import problems as op
    from oracle.matfree import MatFreeKKT
    from paper_2509_01855_gb300 import _lib, api, synth
    N = 257 if dtype == torch.float64 else 256
    M = MatFreeKKT(op.Problem(op.ORBIT, 0.0, 20.0, (0.01, 1.5)), N)
    X, U = synth.orbit_guess(M.t, 1.5, 20.0)
    g = synth.rng("krylov-columns", N, k)
    p64 = api.Problem(_lib.BK_ORBIT, N, torch.float64, 0.0, 20.0, (0.01, 1.5))
    z = from_packed(p64,
                    M.pack(X, U, 0.01 * g.standard_normal((4, M.L)), 0.01 * g.standard_normal(3)))
    prob = api.Problem(_lib.BK_ORBIT, N, dtype, 0.0, 20.0, (0.01, 1.5))
    prob.linearize(z)
    p64.linearize(z)
    opc = _lib.BK_OP_STATE
    b64 = from_packed(p64, g.standard_normal(4 * M.L), op_kkt=False)
    n = b64.numel()
    rhs = torch.zeros(n + 4, dtype=dtype, device="cuda")[off:off + n]
    sol = torch.zeros(n + 4, dtype=dtype, device="cuda")[off:off + n]
    rhs.copy_(b64)
    info = api.krylov_solve(prob, opc, rhs, sol, rtol=1e-14, restart=30, max_iter=k, use_precond=False,
                            raise_on_fail=False)
    want = _least_residual(lambda v: api.kkt_apply(p64, opc, v.contiguous(), torch.zeros_like(v)), rhs.double(), k)
    r = rhs.double() - api.kkt_apply(p64, opc, sol.double(), torch.zeros(n, dtype=torch.float64, device="cuda"))
    assert info["iterations"] == k
    assert abs(info["rel_resid"] - want) < tol
    assert abs(float(r.norm() / rhs.double().norm()) - want) < tol
