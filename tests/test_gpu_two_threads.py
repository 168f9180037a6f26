"""Two host threads, each with a context of its own (one thread per context at
a time is what the interface asks for), run calls whose lattices share a kernel
but not the shared memory that it is launched with.  Every call succeeds and
gives the bits that it gives alone."""
import ctypes
import threading

import numpy as np
import pytest

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


def _both(pt, make, calls):
    """`make(ctx, which)` gives a call; its result alone, then `calls` times beside the other thread's."""
    ctxs = [pt.Context(0) for _ in range(2)]
    fns = [make(c, i) for i, c in enumerate(ctxs)]
    alone = [f() for f in fns]
    wrong = []
    start = threading.Barrier(2)

    def work(i):
        start.wait()
        for _ in range(calls):
            try:
                if not np.array_equal(fns[i](), alone[i]):
                    wrong.append((i, "another result"))
            except Exception as e:              # a PtraceError, kept for the assertion in the main thread
                wrong.append((i, repr(e)))

    ts = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not wrong, (len(wrong), wrong[0])


@pytest.mark.parametrize("prec", ["mixed_fp32", "fp64"])
def test_laplacian_solves(pt, prec):
    """16^3 x 8 (256 threads a CTA) and 32 x 40 x 4 x 2 (160; two z planes in FP64): one build.
    Through the C interface, with the arguments made beforehand: little of a call holds the interpreter."""
    import torch
    shapes = [[16, 16, 16, 8], [32, 40, 4 if prec == "mixed_fp32" else 2, 2]]

    def make(ctx, i):
        op = pt.laplacian(ctx, shapes[i], 20.0)
        b = torch.as_tensor(np.random.default_rng(i).standard_normal((1, int(np.prod(shapes[i]))))).cuda()
        x = torch.empty_like(b)
        torch.cuda.synchronize()
        run = pt.lib().pt_solve
        args = (ctx.handle, op._h, ctypes.c_void_p(b.data_ptr()), ctypes.c_void_p(x.data_ptr()), 1, pt.PREC[prec],
                1e-2, 100, None, None, None)

        def call(op=op, b=b):
            for _ in range(20):
                rc = run(*args)
                if rc:
                    raise RuntimeError("pt_solve: %d" % rc)
            return x.cpu().numpy()

        return call

    _both(pt, make, 300)


# 8-bit colours in shared memory (4^4 and 16 x 16 x 8 x 8), the extended array (sides beyond 127) and the walk of one
# node at a time (a stencil beyond the window's shared memory) against itself at another size
@pytest.mark.parametrize("shapes,k", [(([4, 4, 4, 4], [16, 16, 8, 8]), 1), (([130, 2, 2, 2], [150, 3, 2, 2]), (1, 6)),
                                      (([9, 9, 9, 9], [10, 10, 8, 9]), 12)])
def test_colourings(pt, shapes, k):
    ks = k if isinstance(k, tuple) else (k, k)

    def make(ctx, i):
        return lambda: pt.colour(ctx, shapes[i], 0, [1], ks[i], "natural")[0].cpu().numpy()

    _both(pt, make, 200 if max(ks) < 12 else 12)
