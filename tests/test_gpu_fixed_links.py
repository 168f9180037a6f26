"""The fixed-point outer step of the Wilson solve on links that differ in size
from site to site, on links and sources that hold a NaN or an infinity, and on
links scaled by powers of two far from one."""
import numpy as np
import pytest

import oracle.operators as OO
from oracle.lattice import coords
from paper_2106_01275_gb300 import inputs

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


@pytest.mark.parametrize("prec", ["fp64", "mixed_fp32", "mixed_bf16"])
def test_links_that_shrink_across_the_lattice(pt, ctx, prec):
    """Links of the first half in t are 1e-8 of the others.  For a source on even sites the solution on an odd site
    is kappa times the hop of the even ones, one sum of 24 products per real part from its own neighbours.

    Bound: S = the largest of max |U| max |x| over the eight directions.  The oracle's sums have 48 products and
    additions of numbers below sqrt(2) S, rounded at 2^-53: below 8e-15 S.  Fixed point rounds eight times at a few units
    of 2^-56 S: below 2e-15 S.  2e-14 S in all.  (One exponent for all links would leave 2^-57 of the largest: 1e-9 S.)"""
    dims, kappa = [4, 6, 4, 12], 0.11
    N = int(np.prod(dims))
    xs = coords(dims)
    U = inputs.gauge_links(dims, 21)
    U = U * np.where(xs[:, 3] < dims[3] // 2, 1e-8, 1.0)[:, None, None, None]
    odd = xs.sum(1) % 2 == 1
    rng = np.random.default_rng(4)
    B = rng.standard_normal((2, N, 4, 3)) + 1j * rng.standard_normal((2, N, 4, 3))
    B[:, odd] = 0
    op = pt.wilson(ctx, dims, _t(U), kappa, True)
    X = pt.solve(op, _t(B), prec, 1e-12, 20000)[0].cpu().numpy()
    fwd, bwd = OO.neighbour_tables(dims)
    for x in X:
        want = x - OO.wilson_apply(x, U, kappa, dims, True)              # kappa H x
        u, a = np.abs(U).max((2, 3)), np.abs(x).max((1, 2))
        S = np.max([np.maximum(u[:, mu] * a[fwd[mu]], u[bwd[mu], mu] * a[bwd[mu]]) for mu in range(4)], axis=0)
        err = np.abs(x - want).max((1, 2))
        assert np.all(err[odd] <= 2e-14 * kappa * S[odd]), (err[odd] / S[odd]).max()


@pytest.mark.parametrize("dims", [[4, 4, 2, 6], [3, 5, 2, 4]])
@pytest.mark.parametrize("prec", ["fp64", "mixed_fp32"])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_not_a_number(pt, ctx, dims, prec, value):
    N = int(np.prod(dims))
    U = inputs.gauge_links(dims, 5)
    b = np.ones((1, N, 4, 3), np.complex128)
    bad = U.copy()
    bad[N // 2, 1, 2, 0] = value
    with pytest.raises(pt.PtraceError) as ei:
        pt.solve(pt.wilson(ctx, dims, _t(bad), 0.12, True), _t(b), prec, 1e-8, 500)
    assert ei.value.code == pt.PT_ERR_NUMERIC
    op = pt.wilson(ctx, dims, _t(U), 0.12, True)
    for site in (N // 2, N // 2 + 1):
        c = b.copy()
        c[0, site, 3, 1] = value
        with pytest.raises(pt.PtraceError) as ei:
            pt.solve(op, _t(c), prec, 1e-8, 500)
        assert ei.value.code == pt.PT_ERR_NUMERIC
    assert pt.solve(op, _t(b), prec, 1e-8, 500)[2][0] <= 1e-8           # and the context is usable


@pytest.mark.parametrize("dims", [[4, 4, 2, 6], [3, 5, 2, 4]])
def test_scaled_links_in_fp64(pt, ctx, dims):
    """A psi = psi - kappa H psi is the same operator for links times 2^e and kappa times 2^-e: the same bits."""
    N = int(np.prod(dims))
    U = inputs.gauge_links(dims, 5)
    rng = np.random.default_rng(3)
    b = _t(rng.standard_normal((1, N, 4, 3)) + 1j * rng.standard_normal((1, N, 4, 3)))
    want = pt.solve(pt.wilson(ctx, dims, _t(U), 0.12, True), b, "fp64", 1e-12, 2000)[0].cpu().numpy()
    for e in (-100, 100):
        got = pt.solve(pt.wilson(ctx, dims, _t(U * 2.0 ** e), 0.12 * 2.0 ** -e, True), b, "fp64", 1e-12, 2000)[0]
        assert np.array_equal(got.cpu().numpy(), want), e
