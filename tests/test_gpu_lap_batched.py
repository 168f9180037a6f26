"""The batched Laplacian engine on lattices that the on-chip solver would take
by default (a tuning with its own graph length keeps the engine): what larger
lattices run.  Nested traces, 32 outputs per solve, slots that retire and are
refilled under a slot cap and a memory cap, a maxit that is reached, on the
even-odd and the full system, in every precision, against the oracle and the
engine's own results without caps."""
import numpy as np
import pytest

import oracle.estimator as OE
from oracle.colouring import greedy_colour

pytestmark = pytest.mark.gpu

PRECS = ["fp64", "mixed_fp32", "mixed_bf16"]


@pytest.fixture(scope="module")
def pt():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_01275_gb300 import build
    build.build()
    from paper_2106_01275_gb300 import ptrace
    return ptrace


def _t(a):
    import torch
    return torch.as_tensor(np.ascontiguousarray(a)).cuda()


def _op(pt, dims, m2, prec, ctx=None, **tuning):
    op = pt.laplacian(ctx or pt.Context(0), dims, m2)
    pt.set_tuning(op, prec, graph_iters=4, **tuning)
    return op


# relative 1e-8 of the estimate, as in the other trace tests (solves to 1e-10)
def _close(a, b):
    return np.allclose(a, b, rtol=1e-8, atol=1e-9 * np.abs(b).max())


@pytest.mark.parametrize("dims,tuning", [([8, 4, 6, 8], {}), ([8, 4, 6, 8], {"evenodd": 0}), ([8, 4, 6, 8], {"overlap": 1}),
                                         ([5, 3, 7, 6], {})])
@pytest.mark.parametrize("prec", PRECS)
def test_many_outputs_and_nested_levels(pt, dims, tuning, prec):
    import torch
    m2, mu = 0.2, 3
    c1, m1 = greedy_colour(dims, mu, [1], 1, 0)
    ctx = pt.Context(0)
    op = _op(pt, dims, m2, prec, ctx, **tuning)
    ps = list(range(-16, 16))
    want = OE.probed_estimates(OE.Laplacian(dims, m2), c1, m1, 3, 2, 0, mu, ps, 1e-13)
    est, _, _, st = pt.trace(op, _t(c1), m1, mu, ps, "z2", 3, 0, 2, True, prec, 1e-10, 5000)
    assert st["graph_launches"] > 0 and st["max_relres"] <= 1e-10 and _close(est, want)
    par, mp = pt.colour(ctx, dims, mu, [1], 1)
    fin, mf = pt.colour_nested(ctx, dims, mu, [1], 2, par, mp)
    cols = torch.stack([par, fin]).contiguous()
    nest, sn = pt.trace_nested(op, cols, [mp, mf], mu, [0, 1], "z2", 3, 0, 2, True, prec, 1e-10, 5000)
    assert sn["graph_launches"] > 0
    for lev, (c, m) in enumerate(((par, mp), (fin, mf))):
        w = OE.probed_estimates(OE.Laplacian(dims, m2), c.cpu().numpy(), m, 3, 2, 0, mu, [0, 1], 1e-13)
        assert _close(nest[lev], w), lev


@pytest.mark.parametrize("dims,tuning", [([16, 16, 8, 16], {}), ([16, 16, 8, 16], {"evenodd": 0}), ([15, 16, 9, 16], {})])
@pytest.mark.parametrize("prec", PRECS)
def test_caps_that_retire_and_refill_slots(pt, dims, tuning, prec):
    N, m = int(np.prod(dims)), 3
    col = _t((np.arange(N) * 7 % m).astype(np.int32))
    args = (col, m, 2, [0, 1], "z2", 5, 0, 20, True, prec, 1e-8, 5000)
    est, _, _, free = pt.trace(_op(pt, dims, 0.3, prec, **tuning), *args)
    assert free["n_slots"] == 60 and free["max_relres"] <= 1e-8
    for slots, budget in ((1, None), (7, None), (None, 1 << 24)):
        ctx = pt.Context(0)
        if slots:
            ctx.set_max_slots(slots)
        if budget:
            ctx.set_memory_budget(budget)
        got, _, _, st = pt.trace(_op(pt, dims, 0.3, prec, ctx, **tuning), *args)
        assert st["graph_launches"] > 0 and st["n_rhs"] == 60
        assert st["n_slots"] == slots if slots else 0 < st["n_slots"] < 60
        assert np.array_equal(got, est), (slots, budget)


@pytest.mark.parametrize("prec", PRECS)
def test_maxit_reached(pt, prec):
    dims = [8, 4, 6, 8]
    b = _t(np.random.default_rng(1).standard_normal((3, int(np.prod(dims)))))
    op = _op(pt, dims, 0.2, prec)
    with pytest.raises(pt.PtraceError) as ei:
        pt.solve(op, b, prec, 1e-12, 3)
    assert ei.value.code == pt.PT_ERR_NOCONV
    assert max(pt.solve(op, b, prec, 1e-8, 5000)[2]) <= 1e-8
