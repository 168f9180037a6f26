"""A solve, and the estimate of a noise set, has the same bits whatever else is
in its call: a run cut into chunks (resumed from a log, or split over ranks)
gives what one call gives.  On-chip lattices with one CTA and with several per
solve, even and odd sides, and the batched engines, in every precision."""
import numpy as np
import pytest

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


def _calls(pt, op, dims, prec, n_sets, n_rhs, noise):
    import torch
    N = int(np.prod(dims))
    col = torch.as_tensor((np.arange(N) * 7 % 3).astype(np.int32)).cuda()
    tr = lambda s0, n: pt.trace(op, col, 3, 2, [0, 1], noise, 4, s0, n, True, prec, 1e-9, 5000)[0]
    one = tr(0, n_sets)
    for s0 in (0, 1, n_sets - 2):
        assert np.array_equal(tr(s0, 1), one[s0:s0 + 1]), s0
    shape = (n_rhs, N) if op.dof == 1 else (n_rhs, N, 4, 3)
    rng = np.random.default_rng(2)
    B = rng.standard_normal(shape) + (0 if op.dof == 1 else 1j * rng.standard_normal(shape))
    B = torch.as_tensor(B).cuda()
    X = pt.solve(op, B, prec, 1e-9, 5000)[0]
    for a, b in ((0, 1), (5, 8), (n_rhs - 2, n_rhs)):
        assert torch.equal(pt.solve(op, B[a:b], prec, 1e-9, 5000)[0], X[a:b]), a


@pytest.mark.parametrize("dims", [[4, 4, 4, 4], [8, 8, 8, 16], [9, 7, 11, 15], [12, 10, 10, 22], [16, 16, 16, 16]])
@pytest.mark.parametrize("prec", ["fp64", "mixed_fp32", "mixed_bf16"])
@pytest.mark.parametrize("graph_iters", [8, 4])
def test_laplacian(pt, dims, prec, graph_iters):
    op = pt.laplacian(pt.Context(0), dims, 0.2)
    pt.set_tuning(op, prec, graph_iters=graph_iters)       # 4: the batched engine
    _calls(pt, op, dims, prec, 60, 170, "z2")


@pytest.mark.parametrize("dims", [[4, 4, 4, 8], [5, 3, 4, 6]])
@pytest.mark.parametrize("prec", ["fp64", "mixed_fp32", "mixed_bf16"])
def test_wilson(pt, dims, prec):
    import torch
    op = pt.wilson(pt.Context(0), dims, torch.as_tensor(inputs.gauge_links(dims, 3)).cuda(), 0.12, True)
    _calls(pt, op, dims, prec, 3, 12, "z4")
