"""The Wilson gradient on the even-odd engine against the full system: the same
probes through both (each solve to 1e-10), every output, with several tasks,
an undiluted set, a side of 2, periodic time and every storage precision."""
import numpy as np
import pytest

from oracle.colouring import greedy_colour
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


@pytest.mark.parametrize("dims,antip,dilute", [([4, 4, 4, 8], True, True), ([2, 6, 4, 4], False, True),
                                               ([4, 2, 4, 6], True, False)])
@pytest.mark.parametrize("prec", ["fp64", "mixed_fp32", "mixed_bf16"])
def test_gradient_matches_the_full_system(pt, dims, antip, dilute, prec):
    import torch
    ctx = pt.Context(0)
    U = torch.as_tensor(inputs.gauge_links(dims, 21)).cuda()
    op = pt.wilson(ctx, dims, U, 0.12, antip)
    col, m = greedy_colour(dims, 2, [1], 1, 0)
    col = torch.as_tensor(col).cuda()
    got = pt.grad(op, col, m, 2, 1, "z4", 5, 0, 2, dilute, prec, 1e-10, 5000, links=True)
    pt.set_tuning(op, prec, evenodd=0)
    want = pt.grad(op, col, m, 2, 1, "z4", 5, 0, 2, dilute, prec, 1e-10, 5000, links=True)
    assert got[4]["inner_iters"] < want[4]["inner_iters"]           # the even system took its place
    assert np.allclose(got[0], want[0], rtol=1e-8, atol=1e-8 * np.abs(want[0]).max())
    assert abs(got[1] - want[1]) <= 1e-8 * abs(want[1]) + 1e-8 * np.abs(want[0]).max()
    for a, b in zip(got[2:4], want[2:4]):
        assert (a - b).abs().max() <= 1e-8 * b.abs().max()
