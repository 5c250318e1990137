"""birkhoff_apply_batch with one plan in several entries, where its products need no scratch of
the plan (single-precision N = 4096) or run as launches of their own (binary64 from 2^17 on). Every entry must equal the plan's own product bitwise."""
import pytest
import torch

from paper_2509_01855_gb300 import synth

pytestmark = pytest.mark.gpu


def _run(dtype, Ns, order, trans):
    """Plans of sizes Ns; order: the plan of each entry."""
    from paper_2509_01855_gb300 import api
    plans = [api.Plan(N, n_comp=2, max_batch=2, dtype=dtype, t0=0.0, tf=2.0 + i) for i, N in enumerate(Ns)]
    vs, want = [], []
    for i, k in enumerate(order):
        p, b = plans[k], 1 + i % 2
        v = p.empty(b)
        v[:, :, :p.L] = torch.as_tensor(synth.gaussian((b, 2, p.L), "shared", p.N, i), dtype=dtype)
        vs.append(v)
        want.append((api.birkhoff_apply_T if trans else api.birkhoff_apply)(p, v, p.empty(b)))
    outs = [torch.full_like(w, 2.0) for w in want]
    api.birkhoff_apply_batch([plans[k] for k in order], vs, outs, trans=trans)
    for i, (o, w) in enumerate(zip(outs, want)):
        assert torch.equal(o, w), (i, plans[order[i]].N)


@pytest.mark.parametrize("trans", [False, True])
def test_single_precision_4096_in_several_entries(trans):
    _run(torch.float32, [4096, 256, 4096], [0, 1, 0, 2, 0, 1], trans)            # one-launch plans only
    _run(torch.float32, [4096, 8192, 2048, 1 << 14], [0, 1, 0, 2, 3, 0, 2], trans)   # with launch-per-pass ones
    _run(torch.float32, [4096, 8192], [0] * 20 + [1], trans)                        # more than one launch's entries


@pytest.mark.parametrize("trans", [False, True])
@pytest.mark.parametrize("batched", [False, True])
def test_single_precision_4096_on_several_streams(trans, batched):
    """Products of one plan, or batches that hold it, in flight on four streams at a time."""
    from paper_2509_01855_gb300 import api
    plan = api.Plan(4096, n_comp=4, dtype=torch.float32, t0=0.0, tf=2.0)
    f = api.birkhoff_apply_T if trans else api.birkhoff_apply
    vs, outs, want = [], [], []
    for i in range(4):
        vs.append([])
        for r in range(8):
            v = plan.empty(1)
            v[:, :, :plan.L] = torch.as_tensor(synth.gaussian((1, 4, plan.L), "streams", i, r), dtype=torch.float32)
            vs[i].append(v)
        want.append([f(plan, v, plan.empty(1)) for v in vs[i]])
        outs.append([plan.empty(1) for _ in vs[i]])
    # each stream's batches have a launch-per-pass plan of their own
    own = [api.Plan(8192, n_comp=4, dtype=torch.float32) for _ in range(4)]
    u = [(p.empty(1), p.empty(1)) for p in own]
    streams = [torch.cuda.Stream() for _ in range(4)]
    torch.cuda.synchronize()
    for r in range(8):
        for i, st in enumerate(streams):
            if batched:
                api.birkhoff_apply_batch([plan, own[i]], [vs[i][r], u[i][0]], [outs[i][r], u[i][1]], trans=trans, stream=st)
            else:
                f(plan, vs[i][r], outs[i][r], stream=st)
    torch.cuda.synchronize()
    for i in range(4):
        for o, w in zip(outs[i], want[i]):
            assert torch.equal(o, w)


@pytest.mark.parametrize("trans", [False, True])
def test_long_binary64_plans_in_several_entries(trans):
    _run(torch.float64, [1 << 17, 1 << 14, 4096], [0, 1, 0, 2, 0], trans)


def test_long_binary64_plans_without_double_float():
    from paper_2509_01855_gb300 import api
    try:
        api.set_f64_transform(0)
        _run(torch.float64, [1 << 18, 1 << 16], [0, 0, 1], False)
    finally:
        api.set_f64_transform(-1)


@pytest.mark.parametrize("N", [8192, 1 << 14, 1 << 18])
def test_short_four_step_plans_stay_refused(N):
    from paper_2509_01855_gb300 import _lib, api
    p = api.Plan(N, dtype=torch.float32)
    t = [p.empty(1) for _ in range(4)]
    with pytest.raises(_lib.BirkhoffError):
        api.birkhoff_apply_batch([p, p], t[:2], t[2:])
