"""The windowed greedy walk against the sequential definition (the oracle's C
walk), bit for bit, at the edges of its dispatch: fewer nodes than a window,
one window and one node more, 8-bit and 16-bit colours in shared memory (a
stencil of at most 254 offsets or more), sides beyond the byte arithmetic and
volumes beyond shared memory (the extended array), stencils that cover the
whole lattice (every node its own colour, rows beyond 1024 colours), unions of
displacements, both orders, and nested walks."""
import numpy as np
import pytest

from oracle.colouring import greedy_colour, nested_colour

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


CASES = [([1, 1, 1, 1], 0, [0], 2), ([2, 2, 2, 2], 1, [1], 1), ([31, 1, 1, 1], 0, [3], 2), ([2, 2, 2, 4], 2, [0], 1),
         ([8, 8, 6, 10], 3, [2], 2), ([9, 7, 11, 15], 2, [2], 3), ([6, 6, 6, 6], 3, [1, 3], 4),
         ([130, 3, 2, 4], 0, [40], 3), ([7, 5, 300, 2], 2, [9], 2), ([127, 4, 3, 5], 0, [60], 2),
         ([16, 16, 16, 24], 2, [4], 2), ([24, 24, 16, 24], 3, [3], 2), ([20, 18, 16, 22], 1, [1], 4),
         ([6, 6, 6, 7], 3, [2], 12), ([12, 12, 12, 12], 3, [0], 6)]


@pytest.mark.parametrize("dims,mu,ps,k", CASES)
@pytest.mark.parametrize("order", ["natural", "redblack"])
def test_windowed_walk_is_the_sequential_walk(pt, ctx, dims, mu, ps, k, order):
    want, m = greedy_colour(dims, mu, ps, k, pt.ORDER[order])
    col, got = pt.colour(ctx, dims, mu, ps, k, order)
    assert got == m and np.array_equal(col.cpu().numpy(), want)


@pytest.mark.parametrize("dims,mu,p,k", [([8, 6, 5, 9], 3, 1, 2), ([16, 16, 12, 20], 2, 2, 3), ([5, 140, 2, 3], 1, 7, 2)])
def test_nested_walk(pt, ctx, dims, mu, p, k):
    import torch
    par, mp = greedy_colour(dims, mu, [p], 1, 0)
    want, m = nested_colour(dims, mu, [p], k, par, 0)
    col, got = pt.colour_nested(ctx, dims, mu, [p], k, torch.as_tensor(par).cuda(), mp)
    assert got == m and np.array_equal(col.cpu().numpy(), want)
