"""A call whose launches are refused part way (no fault: the legacy stream is refused
while a blocking stream is being captured) must fail alone: the next call on the
context works and runs nothing that the failed one left behind."""

import ctypes
import threading

import numpy as np
import pytest

from paper_1807_11560_gb300 import Context, LddmmError, inputs

from helpers import ALPHA, S, SIGMA, torch_dev

pytestmark = pytest.mark.gpu

NS, KS, NT = (8, 8), (4, 4), 4000       # a shoot of 8000 evaluations: tens of milliseconds of launches


def _refused_then(ctx, v, out, then):
    """Runs ctx.shoot in a thread, captures a blocking stream once some hundred kernels
    are launched, so that the rest is refused, ends the capture, and runs `then` in the
    same thread (CUDA keeps the last error of a thread); returns both calls' errors."""
    import torch
    torch.cuda.synchronize()
    cu = ctypes.CDLL("libcuda.so.1")
    stream, graph, errors, over = ctypes.c_void_p(), ctypes.c_void_p(), [None, None], threading.Event()
    assert cu.cuStreamCreate(ctypes.byref(stream), 0) == 0          # blocking with respect to the legacy stream
    failed = threading.Event()

    def calls():
        for i, call in enumerate((lambda: ctx.shoot(v, out), then)):
            try:
                call()
            except LddmmError as e:
                errors[i] = e
            failed.set()
            over.wait()

    before = ctx.kernel_count
    worker = threading.Thread(target=calls)
    worker.start()
    while not failed.is_set() and ctx.kernel_count < before + 500:
        pass
    began = cu.cuStreamBeginCapture_v2(stream, 2)                    # relaxed: forbids nothing else
    failed.wait()
    cu.cuStreamEndCapture(stream, ctypes.byref(graph))
    if graph:
        cu.cuGraphDestroy(graph)
    cu.cuStreamDestroy_v2(stream)
    torch.cuda.synchronize()
    over.set()
    worker.join()
    assert began == 0 and errors[0] is not None, "the launches were over before the capture began"
    assert errors[0].code == 3
    return errors


@pytest.fixture
def context():
    """(context with a linearisation point, v, p, H p, kernels of a product)"""
    import torch
    v = torch_dev(inputs.random_bl(KS, 2, 3, 1.0, NS), "fp32")
    p = torch_dev(inputs.random_bl(KS, 2, 4, 1.0, NS), "fp32")
    I0, I1 = inputs.make_pair("blobs", NS, 5, max_disp=1.0)
    with Context(NS, KS, ALPHA, S, SIGMA, NT, precision="fp32", use_graphs=False) as ctx:
        ctx.set_images(torch_dev(I0, "fp32"), torch_dev(I1, "fp32"))
        ref = torch.empty_like(v)
        ctx.gradient(v, ref)
        before = ctx.kernel_count
        ctx.hessvec(p, ref)
        yield ctx, v, p, ref, ctx.kernel_count - before


def test_the_call_after_a_refused_one_works(context):
    import torch
    ctx, v, p, ref, _ = context
    out = torch.empty_like(p)
    errors = _refused_then(ctx, v, torch.empty_like(v), lambda: ctx.hessvec(p, out))
    assert errors[1] is None
    np.testing.assert_array_equal(out.cpu().numpy(), ref.cpu().numpy())


def test_the_call_after_a_refused_one_launches_its_own_kernels_only(context):
    import torch
    ctx, v, p, ref, kernels = context
    counts = []

    def then():
        counts.append(ctx.kernel_count)
        ctx.hessvec(p, torch.empty_like(p))
        counts.append(ctx.kernel_count)

    errors = _refused_then(ctx, v, torch.empty_like(v), then)
    assert errors[1] is None
    assert counts[1] - counts[0] == kernels
