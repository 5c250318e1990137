"""Clenshaw-Curtis weights of a plan, relative to each weight, and the plans that need them most.

The reference is the cosine sum with its cancellation taken out: with theta = pi k / N,
    N w_k / c = [1 - sum'' 2 cos(2 j theta) / (4 j^2 - 1)]      (c = 1 at the ends, 2 inside)
              = 1 / N + sum_{j <= (N-1)/2} 4 sin^2(j theta) / (4 j^2 - 1)                       (N odd)
              = (N + 1 - (-1)^k) / (N^2 - 1) + sum_{j < N/2} 4 sin^2(j theta) / (4 j^2 - 1)      (N even),
whose terms are all positive: its relative error is that of a term, 4 units in the last place. The
weights themselves are allowed 8 (a quotient, a sine, two products, a correction): 12 * 2.2e-16 < 4e-15.
"""
import math

import numpy as np
import pytest
import torch

from oracle import birkhoff as ob
from paper_2509_01855_gb300 import synth

pytestmark = pytest.mark.gpu


def _weight(N, k):
    k = min(k, N - k)
    jm = (N - 1) // 2
    j = np.arange(1, jm + 1, dtype=np.int64)
    r = (j * k) % N
    s = np.sin(np.pi * np.minimum(r, N - r) / N)
    t = 4.0 * s * s / (4.0 * j.astype(float) ** 2 - 1.0)
    first = 1.0 / N if N % 2 else (N + 1 - (-1) ** k) / ((N - 1.0) * (N + 1.0))
    return (1.0 if k == 0 else 2.0) / N * math.fsum([first, *t])


SIZES = [(n, torch.float64) for n in (4, 16, 64, 256, 1100, 1101, 3000, 4097, 6000, 65536, 100003, 1 << 18, 1 << 20)]
SIZES += [(n, torch.float32) for n in (8, 128, 2048, 1101, 6000, 1 << 16, 100003, 4800000)]


@pytest.mark.parametrize("N,dtype", SIZES)
def test_every_weight_to_its_own_accuracy(N, dtype):
    from paper_2509_01855_gb300 import api
    _, w = api.Plan(N, dtype=dtype).grid()
    w = w.numpy()
    assert np.all(w > 0) and abs(math.fsum(w) - 2.0) < 1e-14
    ks = {0, 1, 2, 3, 7, 30, 31, 32, 33, 100, 1022, 1023, 1024, 1025, N // 3, N // 2 - 1, N // 2, N // 2 + 1}
    ks |= {N - k for k in ks}
    for k in sorted(k for k in ks if 0 <= k <= N):
        want = _weight(N, k)
        assert abs(w[k] - want) <= 4e-15 * want, (k, w[k] / want - 1)


@pytest.mark.parametrize("N,path", [(4800000, "split_four_step"), (5000001, "bluestein"), ((1 << 23) - 1, "bluestein")])
def test_single_precision_lengths_above_2p22(N, path):
    """Lengths that only single-precision plans take: products against the FastBV chain, 1e-5."""
    from paper_2509_01855_gb300 import api
    plan = api.Plan(N, dtype=torch.float32, t0=0.0, tf=2.0)
    assert plan.shape()["path"] == path
    V = synth.gaussian((1, N + 1), "f32-long", N)
    v = plan.empty(1)
    v[0, :, :N + 1] = torch.as_tensor(V)
    for f, ref in ((api.birkhoff_apply, ob.fastbv), (api.birkhoff_apply_T, ob.fastbv_T)):
        out = f(plan, v, plan.empty(1))
        want = ref(V, 0.0, 2.0)
        assert np.linalg.norm(out[0, :, :N + 1].double().cpu().numpy() - want) <= 1e-5 * np.linalg.norm(want)
        assert torch.all(out[0, :, N + 1:] == 0)


def test_lengths_past_the_limits_stay_refused():
    from paper_2509_01855_gb300 import _lib, api
    for N, dtype in (((1 << 23) + 1, torch.float32), ((1 << 22) + 16, torch.float64)):
        with pytest.raises(_lib.BirkhoffError):
            api.Plan(N, dtype=dtype)
