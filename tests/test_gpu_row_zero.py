"""Row 0 of B v is exactly zero (and row N of B^b v), on every path and in both precisions."""
import pytest
import torch

from paper_2509_01855_gb300 import synth

pytestmark = pytest.mark.gpu

PATHS = {"single_cta": (16, 256), "four_step": (4096,), "split_four_step": (8192, 1 << 14, 1 << 18, 1 << 19, 1200, 6000),
         "dense": (100,), "bluestein": (1100, 3001)}


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("path,N", [(p, n) for p, ns in PATHS.items() for n in ns])
def test_first_row_is_exactly_zero(path, N, dtype):
    from paper_2509_01855_gb300 import api
    plan = api.Plan(N, n_comp=5, dtype=dtype, t0=0.5, tf=3.5)
    assert plan.shape()["path"] == path
    v = plan.empty(1)
    v[:, :, :N + 1] = torch.as_tensor(synth.gaussian((1, 5, N + 1), "row-zero", N), dtype=dtype)
    out = api.birkhoff_apply(plan, v, plan.empty(1).fill_(1.0))
    assert torch.all(out[:, :, 0] == 0)
    assert torch.all(out[:, :, N] != 0)
    v[0, 1, N // 2] = float("nan")   # a vector with a NaN has no product
    nan = api.birkhoff_apply(plan, v, plan.empty(1))
    assert torch.all(nan[0, 1, int(path == "dense"):N + 1].isnan()) and torch.equal(nan[0, 2], out[0, 2])
    v[0, 1, N // 2] = 0.0
    out = api.birkhoff_apply_b(plan, v, plan.empty(1).fill_(1.0))
    assert torch.all(out[:, :, N] == 0)


@pytest.mark.parametrize("N", [8192, 65536])
def test_first_row_without_allocation(N):
    from paper_2509_01855_gb300 import _lib
    pitch = N + 2
    v = torch.randn(3, pitch, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(N))
    out = torch.ones_like(v)
    _lib.check(_lib.lib().birkhoff_apply_noalloc(_lib.ptr(v), _lib.ptr(out), N, 3, pitch, 0.0, 2.0, _lib.stream_ptr(None)))
    assert torch.all(out[:, 0] == 0) and torch.all(out[:, N] != 0)
