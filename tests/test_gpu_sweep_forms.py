"""Sweep passes at the edges of their grids: single blocks, block and level boundaries,
the last warp's idle lanes, vectors that are only element-aligned, and the single-column and
side-by-side (terminal Schur) forms, against the matrix-free oracle.

Tolerances are those of the preconditioner tests: 1e-10 (FP64) and 1e-3 (FP32) for K-tilde^{-1};
an unaligned call must give the aligned call's values exactly (the same arithmetic).
"""
import numpy as np
import pytest
import torch

from oracle import problems as op
from oracle.matfree import MatFreeKKT
from paper_2509_01855_gb300 import synth
from tests.helpers import from_packed, to_packed

pytestmark = pytest.mark.gpu

TOL = {torch.float64: 1e-10, torch.float32: 1e-3}


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("N", [16, 255, 256, 500, 512, 1000, 2048])
def test_kkt_preconditioner_at_grid_edges(N, dtype):
    from paper_2509_01855_gb300 import _lib, api
    M = MatFreeKKT(op.Problem(op.ORBIT, 0.0, 20.0, (0.01, 1.5)), N)
    prob = api.Problem(_lib.BK_ORBIT, N, dtype, 0.0, 20.0, (0.01, 1.5))
    g = synth.rng("sweep-edges", N)
    X, U = synth.orbit_guess(M.t, 1.5, 20.0)
    vec = M.pack(X + 0.01 * g.standard_normal(X.shape), U, M.w * g.standard_normal((4, M.L)), g.standard_normal(3))
    prob.linearize(from_packed(prob, vec))
    M.linearize_precond(vec)
    r = g.standard_normal(M.n)
    x = from_packed(prob, r, dtype=dtype)
    out = api.precond_apply(prob, _lib.BK_OP_KKT, x, torch.full_like(x, 3.0))
    got, want = to_packed(prob, out.double()), M.precond_solve(r)
    assert np.linalg.norm(got - want) <= TOL[dtype] * np.linalg.norm(want)
    P, L = prob.pitch, prob.L
    assert torch.all(out[:10 * P].view(10, P)[:, L:] == 0)
    # the same vectors one element off a 16-byte boundary, and a second call on the same scratch
    xs = torch.empty(x.numel() + 1, dtype=dtype, device="cuda")[1:]
    xs.copy_(x)
    os_ = torch.full((x.numel() + 1,), 3.0, dtype=dtype, device="cuda")[1:]
    api.precond_apply(prob, _lib.BK_OP_KKT, xs, os_)
    assert torch.equal(os_, out)
