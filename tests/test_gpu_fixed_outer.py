"""The FP64 outer residual of the Wilson solve (even-odd and full system), whose hops run in
block fixed point: solves to a tolerance near the FP64 floor, checked by the
oracle's FP64 operator, where a wrong digit would show: unitary and scaled
links, a point source (components over many orders of magnitude), a half
volume that is not a multiple of a work item, sides of 2, every storage
precision, and sources far from one.

Bound: the solver's own test promises 1e-14; the oracle's FP64 residual adds
its rounding, about 100 operations of 2^-53 per component, below 1e-14 of
|x| <= 2 |b| here: 3e-14 in all."""
import numpy as np
import pytest

import oracle.clover as OC
import oracle.operators as OO
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


@pytest.mark.parametrize("dims,scale,csw,eo", [([8, 8, 8, 16], 1.0, 0.0, 1), ([6, 2, 4, 10], 1.0, 0.0, 1),
                                               ([4, 6, 4, 8], 7.3, 0.0, 1), ([4, 4, 6, 8], 1.0, 1.1, 1),
                                               ([2, 2, 2, 4], 0.01, 0.0, 1), ([5, 3, 7, 9], 1.0, 0.0, 0),
                                               ([1, 4, 2, 3], 2.5, 0.0, 0), ([4, 6, 4, 8], 1.0, 0.0, 0)])
@pytest.mark.parametrize("prec", ["fp64", "mixed_fp32", "mixed_bf16"])
def test_solve_near_the_fp64_floor(pt, ctx, dims, scale, csw, eo, prec):
    N = int(np.prod(dims))
    U = inputs.gauge_links(dims, 77) * scale
    kappa = 0.11 / scale
    op = pt.wilson(ctx, dims, _t(U), kappa, True)
    if csw:
        pt.set_clover(op, csw)
    pt.set_tuning(op, prec, evenodd=eo)
    rng = np.random.default_rng(8)
    B = np.zeros((4, N, 4, 3), np.complex128)
    B[0, N // 3, 1, 2] = 1.0                                        # an even or odd point, and its neighbour
    B[1, N // 3 + 1, 2, 0] = 1j
    B[2] = rng.standard_normal((N, 4, 3)) + 1j * rng.standard_normal((N, 4, 3))
    B[3] = B[2] * 10.0 ** rng.uniform(-8, 0, (N, 1, 1))
    X, _, relres, _ = pt.solve(op, _t(B), prec, 1e-14, 20000)
    pt.set_tuning(op, prec, reset=True)
    X = X.cpu().numpy()
    for j in range(4):
        ax = OC.clover_apply(X[j], U, kappa, csw, dims, True) if csw else OO.wilson_apply(X[j], U, kappa, dims, True)
        assert relres[j] <= 1e-14
        assert np.linalg.norm(B[j] - ax) <= 3e-14 * np.linalg.norm(B[j]), j


def test_scaled_sources_in_fp64(pt, ctx):
    """The site exponents follow the data: a source scaled by a power of two
    far from one gives the same solution, scaled, bit for bit."""
    dims, kappa = [4, 4, 2, 6], 0.12
    N = int(np.prod(dims))
    op = pt.wilson(ctx, dims, _t(inputs.gauge_links(dims, 5)), kappa, True)
    rng = np.random.default_rng(3)
    b = rng.standard_normal((1, N, 4, 3)) + 1j * rng.standard_normal((1, N, 4, 3))
    X1 = pt.solve(op, _t(b), "fp64", 1e-12, 2000)[0].cpu().numpy()
    for e in (-100, 100):
        X2 = pt.solve(op, _t(b * 2.0 ** e), "fp64", 1e-12, 2000)[0].cpu().numpy()
        assert np.array_equal(X2, X1 * 2.0 ** e), e
