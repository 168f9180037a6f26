"""The cluster-resident Laplacian solver against the batched engine and the
oracle, over the forms that its dispatch accepts: one to sixteen CTAs per
cluster, slabs of unequal thickness, four-entry and one-entry units, even-odd
and full system, every precision, solves, plain, nested and 32-output traces,
and the caller's caps.  A tuning with its own graph length keeps the batched
engine, which is the general path that the results are compared with (both
solve to 1e-10, so estimates agree to the 1e-8 of the other trace tests)."""
import numpy as np
import pytest

import oracle.estimator as OE
from oracle.colouring import greedy_colour

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pt():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_01275_gb300 import build
    build.build()
    from paper_2106_01275_gb300 import ptrace
    return ptrace


@pytest.fixture(scope="module")
def ctx(pt):
    return pt.Context(0)


def _t(a):
    import torch
    return torch.as_tensor(np.ascontiguousarray(a)).cuda()


# one CTA: a single site, sides of 1 and 2, a row of units; several: more t planes than CTAs, a last
# slab of another thickness, one plane per CTA, planes that fill part of the threads
SHAPES = [[1, 1, 1, 1], [3, 1, 5, 2], [2, 2, 2, 2], [8, 2, 2, 4], [6, 4, 2, 10], [16, 16, 16, 2], [8, 24, 6, 14],
          [16, 16, 16, 16], [9, 13, 7, 11], [22, 23, 8, 9], [14, 18, 12, 18], [24, 22, 10, 22],
          [26, 26, 6, 8], [8, 16, 16, 36]]


def fits(dims, eo, prec):
    """The dispatch rule: the xy plane within a CTA's threads, and a slab of t
    planes per CTA within its threads' entries for at most sixteen CTAs."""
    v = 4 if eo and dims[0] % 8 == 0 else 1
    threads, entries = (256, 32) if v == 4 else (512, 16)
    entries //= 2 if prec == "fp64" else 1
    plane = dims[0] * dims[1] // (2 if eo else 1) // v
    if plane > threads:
        return False
    return any(c <= dims[3] and -(-(-(-dims[3] // c) * dims[2]) // (threads // plane)) * v <= entries for c in (1, 2, 4, 8, 16))


@pytest.mark.parametrize("dims", SHAPES)
@pytest.mark.parametrize("prec", ["fp64", "mixed_fp32", "mixed_bf16"])
def test_trace_and_solve_match_the_batched_engine(pt, ctx, dims, prec):
    import torch
    N, m2, mu = int(np.prod(dims)), 0.1, 2
    m = min(3, N)
    col = _t(((np.arange(N) * 7 + np.arange(N) // dims[0]) % m).astype(np.int32))
    op = pt.laplacian(ctx, dims, m2)
    B = torch.as_tensor(np.random.default_rng(5).standard_normal((5, N))).cuda()
    ps = [0, 1, 3, -2]
    for eo in ((1, 0) if pt.get_tuning(op, prec)["evenodd"] else (0,)):
        pt.set_tuning(op, prec, evenodd=eo)
        est, _, _, st = pt.trace(op, col, m, mu, ps, "z2", 9, 1, 2, True, prec, 1e-10, 20000)
        X, _, rel, _ = pt.solve(op, B, prec, 1e-10, 20000)
        pt.set_tuning(op, prec, evenodd=eo, graph_iters=4)
        want, _, _, sg = pt.trace(op, col, m, mu, ps, "z2", 9, 1, 2, True, prec, 1e-10, 20000)
        Y, _, _, _ = pt.solve(op, B, prec, 1e-10, 20000)
        pt.set_tuning(op, prec, reset=True)
        assert sg["graph_launches"] > 0 and st["n_rhs"] == 2 * m and st["max_relres"] <= 1e-10 and max(rel) <= 1e-10
        assert (st["graph_launches"] == 0) == fits(dims, eo, prec), eo
        assert np.allclose(est, want, rtol=1e-8, atol=1e-9 * np.abs(want).max()), eo
        assert torch.allclose(X, Y, rtol=1e-7, atol=1e-8 * Y.abs().max().item()), eo


def test_many_displacements_nested_levels_and_caps(pt, ctx):
    """32 outputs per solve, nested levels, a slot cap and a memory cap that
    leave one cluster, a maxit that is reached."""
    import torch
    dims, m2, mu = [8, 4, 6, 8], 0.2, 3
    N = int(np.prod(dims))
    c1, m1 = greedy_colour(dims, mu, [1], 1, 0)
    op = pt.laplacian(ctx, dims, m2)
    ps = list(range(-16, 16))
    want = OE.probed_estimates(OE.Laplacian(dims, m2), c1, m1, 3, 2, 0, mu, ps, 1e-13)
    est, _, _, st = pt.trace(op, _t(c1), m1, mu, ps, "z2", 3, 0, 2, True, "mixed_fp32", 1e-10, 5000)
    assert st["kernel_launches"] == 1 and np.allclose(est, want, rtol=1e-8, atol=1e-9 * np.abs(want).max())
    par, mp = pt.colour(ctx, dims, mu, [1], 1)
    fin, mf = pt.colour_nested(ctx, dims, mu, [1], 2, par, mp)
    cols = torch.stack([par, fin]).contiguous()
    nest, _ = pt.trace_nested(op, cols, [mp, mf], mu, [0, 1], "z2", 3, 0, 2, True, "mixed_fp32", 1e-10, 5000)
    for lev, (c, m) in enumerate(((par, mp), (fin, mf))):
        w = OE.probed_estimates(OE.Laplacian(dims, m2), c.cpu().numpy(), m, 3, 2, 0, mu, [0, 1], 1e-13)
        assert np.allclose(nest[lev], w, rtol=1e-8, atol=1e-9 * np.abs(w).max()), lev
    small = pt.Context(0)
    small.set_max_slots(1)
    small.set_memory_budget(1 << 24)
    ops = pt.laplacian(small, dims, m2)
    one, _, _, s1 = pt.trace(ops, _t(c1), m1, mu, ps, "z2", 3, 0, 2, True, "mixed_fp32", 1e-10, 5000)
    assert s1["n_slots"] == 1 and np.array_equal(one, est)
    with pytest.raises(pt.PtraceError) as ei:
        pt.solve(op, _t(np.random.default_rng(1).standard_normal((3, N))), "mixed_fp32", 1e-12, 3)
    assert ei.value.code == pt.PT_ERR_NOCONV


@pytest.mark.parametrize("dims,m2,mu,p", [([8, 8, 8, 16], 0.1587, 3, 5), ([12, 10, 10, 22], 0.1488, 0, 2)])
def test_kept_direction_ends_below_the_tolerance(pt, ctx, dims, m2, mu, p):
    """A last cycle that keeps its direction aims at tol / 8; it is kept only
    where the FP64 residual is within 1.5 times the recursion's, so with FP32
    drift of that size at most the final one is below 0.19 tol."""
    col, m = pt.colour(ctx, dims, mu, [p], 1, "natural")
    op = pt.laplacian(ctx, dims, m2)
    _, _, _, st = pt.trace(op, col, m, mu, [p], "z2", 5, 0, 2, True, "mixed_fp32", 1e-10, 5000)
    assert st["graph_launches"] == 0 and st["max_relres"] <= 0.19e-10
