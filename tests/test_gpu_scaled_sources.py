"""Mixed-precision solves of a source and of the same source times a power of two
give the same solution, scaled, bit for bit: no sum of squares or product of
the outer and inner steps leaves the normal range of its type for sources of
moderate size (|b| from 1e-5 to 1e5 and residuals down to 1e-8 |b|: squares of
1e-26 and more, entries a thousand times smaller still 1e-32)."""
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


@pytest.mark.parametrize("kind", ["wilson", "laplacian", "laplacian, batched"])
@pytest.mark.parametrize("dims", [[4, 4, 2, 6], [3, 5, 2, 4], [8, 4, 6, 12]])
@pytest.mark.parametrize("prec", ["mixed_fp32", "mixed_bf16"])
def test_scaled_sources(pt, kind, dims, prec):
    import torch
    N = int(np.prod(dims))
    ctx = pt.Context(0)
    rng = np.random.default_rng(3)
    if kind == "wilson":
        op = pt.wilson(ctx, dims, torch.as_tensor(inputs.gauge_links(dims, 5)).cuda(), 0.12, True)
        b = rng.standard_normal((2, N, 4, 3)) + 1j * rng.standard_normal((2, N, 4, 3))
    else:
        op = pt.laplacian(ctx, dims, 0.3)
        if kind.endswith("batched"):
            pt.set_tuning(op, prec, graph_iters=4)
        b = rng.standard_normal((2, N))
    want, _, rel, _ = pt.solve(op, torch.as_tensor(b).cuda(), prec, 1e-8, 2000)
    assert max(rel) <= 1e-8
    for e in (-17, 17):
        got = pt.solve(op, torch.as_tensor(b * 2.0 ** e).cuda(), prec, 1e-8, 2000)[0]
        assert torch.equal(got, want * 2.0 ** e), e
