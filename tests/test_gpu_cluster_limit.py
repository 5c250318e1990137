"""Plans on a device that holds no large thread-block cluster (BK_MAX_CLUSTER stands for such a
device) take forms without one, and compute the same products."""
import numpy as np
import pytest
import torch

from oracle import birkhoff as ob
from paper_2509_01855_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = {torch.float64: 1e-12, torch.float32: 1e-5}


@pytest.mark.parametrize("limit", ["8", "0"])
@pytest.mark.parametrize("N,dtype", [(512, torch.float64), (1024, torch.float64), (4096, torch.float64), (4096, torch.float32)])
def test_products_without_large_clusters(N, dtype, limit, monkeypatch):
    from paper_2509_01855_gb300 import api
    assert api.Plan(N, n_comp=2, dtype=dtype).shape()["path"] == "four_step"
    monkeypatch.setenv("BK_MAX_CLUSTER", limit)
    plan = api.Plan(N, n_comp=2, max_batch=2, dtype=dtype, t0=0.5, tf=3.5)
    want = "single_cta" if dtype == torch.float32 else "split_four_step"
    assert plan.shape()["path"] == ("four_step" if (N, limit) == (512, "8") else want)   # FP64 512: clusters of 8
    V = synth.gaussian((2, 2, N + 1), "no-cluster", N)
    v = plan.empty(2)
    v[:, :, :N + 1] = torch.as_tensor(V, dtype=dtype)
    other = api.Plan(8192, n_comp=2, max_batch=2, dtype=dtype)
    u = other.empty(2).fill_(0.5)
    for f, trans, ref in ((api.birkhoff_apply, False, ob.fastbv), (api.birkhoff_apply_T, True, ob.fastbv_T)):
        out = f(plan, v, plan.empty(2))
        want = ref(V, 0.5, 3.5)
        assert np.linalg.norm(out[:, :, :N + 1].double().cpu().numpy() - want) <= TOL[dtype] * np.linalg.norm(want)
        got = plan.empty(2)
        api.birkhoff_apply_batch([other, plan], [u, v], [other.empty(2), got], trans=trans)
        assert torch.equal(got, out)
