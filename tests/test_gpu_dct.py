"""The real-even four-step passes at the edges of their shapes, against the FastBV oracle.

Sizes: the smallest factors (16 x 16), unequal factors, both sides of the borders between the
one-CTA, one-launch and launch-per-pass forms, tiles whose last pair is alone in its CTA, and the
8192-point rows of N = 2^24. Tolerances are the product's own: 1e-12 (FP64, double-float), 1e-5 (FP32).
"""
import numpy as np
import pytest
import torch

from oracle import birkhoff as ob
from paper_2509_01855_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = {torch.float64: 1e-12, torch.float32: 1e-5}
T0, TF = 0.5, 3.5


def _check(N, dtype, comps=3, batch=1, pitch=0, path=None):
    from paper_2509_01855_gb300 import api
    plan = api.Plan(N, n_comp=comps, max_batch=batch, dtype=dtype, t0=T0, tf=TF, pitch=pitch)
    if path:
        assert plan.shape()["path"] == path, plan.shape()
    V = synth.gaussian((batch, comps, N + 1), "dct", N, comps)
    v = plan.empty(batch).fill_(7.0)               # the padding of the inputs is not read
    v[:, :, :N + 1] = torch.as_tensor(V, dtype=dtype)
    for trans in (False, True):
        f = api.birkhoff_apply_T if trans else api.birkhoff_apply
        out = f(plan, v, plan.empty(batch).fill_(-3.0))
        ref = (ob.fastbv_T if trans else ob.fastbv)(V, T0, TF)
        got = out[:, :, :N + 1].double().cpu().numpy()
        assert np.linalg.norm(got - ref) <= TOL[dtype] * np.linalg.norm(ref), (N, trans)
        assert torch.all(out[:, :, N + 1:] == 0)
        same = f(plan, v.clone(), out)              # a second pass on the same scratch
        assert torch.equal(same, f(plan, w := v.clone(), w))   # in place


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("form,path", [("30", "four_step"), ("7", "split_four_step")])
@pytest.mark.parametrize("N", [128, 256, 512, 2048, 8192])
def test_forms_at_small_and_middle_sizes(N, form, path, dtype, monkeypatch):
    monkeypatch.setenv("BK_SMALL_MAX_LOG2", "6")
    monkeypatch.setenv("BK_SPLIT_MIN_LOG2", form)
    _check(N, dtype, path=path)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("N", [256, 512, 4096, 8192, 1 << 14, 1 << 16, 1 << 17, 1 << 18])
def test_default_forms_either_side_of_their_borders(N, dtype):
    _check(N, dtype, comps=1, batch=2, pitch=N + 36)


def test_longest_rows_in_double_float_and_binary64():
    """N = 2^24: rows of 8192 points in FP64, in both arithmetics."""
    from paper_2509_01855_gb300 import api
    try:
        for mode in (1, 0):
            api.set_f64_transform(mode)
            _check(1 << 24, torch.float64, comps=1, path="split_four_step")
    finally:
        api.set_f64_transform(-1)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("N", [1200, 1280, 2160, 6000, 16 * 625, 16 * 3 ** 6, 100000, 16 * 3 ** 4 * 5 ** 4])
def test_mixed_radix_sizes(N, dtype):
    """N = 16 m with m a product of 2, 3 and 5: every radix alone and mixed, odd and even stage counts."""
    _check(N, dtype, path="split_four_step")


@pytest.mark.parametrize("N", [1040, 1100, 3000, 4095, 16 * 7 * 11])
def test_sizes_without_a_mixed_radix_form_keep_the_convolution(N):
    _check(N, torch.float64, path="bluestein")


def test_mixed_radix_longest():
    _check(16 * 3 ** 4 * 5 ** 5, torch.float64, comps=1, path="split_four_step")   # N = 4050000
