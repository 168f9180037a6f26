"""The device memory that a Wilson trace, solve or gradient takes stays within
the context's budget, with the link copies of the fixed-point outer step in it."""
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


@pytest.mark.parametrize("prec", ["fp64", "mixed_fp32", "mixed_bf16"])
@pytest.mark.parametrize("call", ["grad", "trace"])
def test_within_the_budget(pt, prec, call):
    """A budget of two FP64 solution pairs (8 vectors each) and no more.  2 MiB of slack for the work lists, partial sums
    and graphs, and 2 MiB for the allocator's pages; the link copies alone are 9.7 MB."""
    import torch
    dims = [8, 8, 16, 16]
    N = int(np.prod(dims))
    U = torch.as_tensor(inputs.gauge_links(dims, 5)).cuda()
    col = torch.zeros(N, dtype=torch.int32, device="cuda")
    budget = 2 * 2 * N * 24 * 64 + (1 << 18)

    def run(nbytes):
        ctx = pt.Context(0)
        ctx.set_memory_budget(nbytes)
        op = pt.wilson(ctx, dims, U, 0.11, True)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        if call == "grad":
            pt.grad(op, col, 1, 2, 1, "z4", 3, 0, 1, True, prec, 1e-6, 500)
        else:
            pt.trace(op, col, 1, 2, [0, 1], "z4", 3, 0, 8, True, prec, 1e-6, 500)
        torch.cuda.synchronize()
        return free - torch.cuda.mem_get_info()[0]

    run(1 << 24)                                     # kernels are loaded
    assert run(budget) <= budget + (1 << 22)
