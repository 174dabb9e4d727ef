"""The allocation-free transform entry point, lddmm_iota_noalloc.

It serves callers that cannot let a library allocate device memory (a host
framework whose allocator owns the device memory, latency-bound loops that
cannot absorb cudaFree's synchronisation, plugin hosts that forbid it).  It
must give the same grid values as the context-based lddmm_iota, call after
call, although every call reuses one fixed scratch array.

This file is collected last on purpose; it must pass on its own in a fresh
process and after every other test.
"""

import ctypes

import numpy as np
import pytest

from paper_1807_11560_gb300 import Context, inputs, lddmm

pytestmark = pytest.mark.gpu

ALPHA, S, SIGMA = 0.0025, 2, 0.03
TOL = 2e-6            # the FP32 transform tolerance of the other GPU tests


def _rel(a, b):
    """The larger of the relative l2 error and max |a - b| / max |b|."""
    norm = float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel()))
    return max(norm, float(np.abs(a - b).max() / np.abs(b).max()))


# 128^3 crosses the size from which the context's transform runs on the tensor
# cores (3xTF32), so that case compares the two arithmetic paths as well
@pytest.mark.parametrize("Ns,Ks", [((64, 64, 64), (16, 16, 16)), ((33, 17), (10, 6)),
                                   ((128, 128, 128), (16, 16, 16))])
def test_noalloc_iota_matches_context_iota_on_two_calls(Ns, Ks):
    import torch
    d = len(Ns)
    stream = torch.cuda.current_stream().cuda_stream
    with Context(Ns, Ks, ALPHA, S, SIGMA, 2, precision="fp32") as ctx:
        for seed in (3, 4):           # two calls in a row, different inputs
            a = torch.as_tensor(inputs.random_bl(Ks, d, seed, 2.0, Ns), dtype=torch.complex64,
                                device="cuda")
            ref = torch.empty((d,) + Ns, dtype=torch.float32, device="cuda")
            ctx.iota(a, d, ref)
            out = torch.full((d,) + Ns, float("nan"), dtype=torch.float32, device="cuda")
            rc = lddmm.iota_noalloc(Ns, Ks, a, d, out, stream)
            assert rc == 0
            torch.cuda.synchronize()
            assert _rel(out.cpu().numpy(), ref.cpu().numpy()) < TOL


def test_noalloc_rejects_sizes_beyond_its_scratch_and_host_pointers():
    import torch
    L = lddmm.lib()
    arr = ctypes.c_int * 3
    a = torch.zeros(8, dtype=torch.complex64, device="cuda")
    f = torch.zeros(8, dtype=torch.float32, device="cuda")
    # 36 fields on 512^3 with band 64^3 need far more than the fixed scratch
    assert L.lddmm_iota_noalloc(3, arr(512, 512, 512), arr(64, 64, 64), a.data_ptr(), 36,
                                f.data_ptr(), None) == 2        # LDDMM_ENOMEM
    # an odd band is an argument error
    assert L.lddmm_iota_noalloc(3, arr(16, 16, 16), arr(7, 8, 8), a.data_ptr(), 1,
                                f.data_ptr(), None) == 1        # LDDMM_EINVAL
    host = np.zeros(4 * 4 * 4, np.complex64)
    out = torch.zeros((4, 4, 4), dtype=torch.float32, device="cuda")
    assert L.lddmm_iota_noalloc(3, arr(4, 4, 4), arr(2, 2, 2), host.ctypes.data, 1,
                                out.data_ptr(), None) == 1      # host input refused


def test_noalloc_calls_allocate_no_device_memory():
    """After one warm-up call (which loads the kernels), further calls leave the
    device's free memory and torch's allocator untouched."""
    import torch
    Ns, Ks = (96, 80, 64), (16, 16, 16)
    d = 3
    stream = torch.cuda.current_stream().cuda_stream
    a = torch.as_tensor(inputs.random_bl(Ks, d, 5, 2.0, Ns), dtype=torch.complex64, device="cuda")
    out = torch.empty((d,) + Ns, dtype=torch.float32, device="cuda")
    assert lddmm.iota_noalloc(Ns, Ks, a, d, out, stream) == 0
    torch.cuda.synchronize()
    free0, _ = torch.cuda.mem_get_info()
    held0 = torch.cuda.memory_allocated()
    for _ in range(5):
        assert lddmm.iota_noalloc(Ns, Ks, a, d, out, stream) == 0
    torch.cuda.synchronize()
    free1, _ = torch.cuda.mem_get_info()
    assert free1 >= free0
    assert torch.cuda.memory_allocated() == held0


def test_noalloc_binding_checks_extents():
    """The C call cannot see array extents; the binding refuses mismatched sizes."""
    import torch
    a = torch.zeros((3, 8, 8, 8), dtype=torch.complex64, device="cuda")
    out = torch.zeros((3, 16, 16, 16), dtype=torch.float32, device="cuda")
    with pytest.raises(ValueError):
        lddmm.iota_noalloc((16, 16, 16), (8, 8, 8), a[:2], 3, out)
    with pytest.raises(ValueError):
        lddmm.iota_noalloc((16, 16, 16), (8, 8, 8), a, 3, out[:2])
    with pytest.raises(ValueError):
        lddmm.iota_noalloc((16, 16, 16), (8, 8), a, 3, out)


@pytest.mark.parametrize("Ns,Ks", [((32, 32, 32), (8, 8, 8)), ((64, 64, 64), (32, 32, 32)), ((48, 48, 49), (16, 48, 48))])
def test_noalloc_calls_in_a_row_keep_their_order(Ns, Ks):
    """The kernels of a call overlap their predecessors' ends (small items and large
    ones), and a call follows the one before on the same scratch without a
    synchronisation: every result is its own input's."""
    import torch
    stream = torch.cuda.current_stream().cuda_stream
    a = [torch.as_tensor(inputs.random_bl(Ks, 3, seed, 2.0, Ns), dtype=torch.complex64, device="cuda")
         for seed in range(6)]
    out = [torch.full((3,) + Ns, float("nan"), dtype=torch.float32, device="cuda") for _ in a]
    torch.cuda.synchronize()
    for x, y in zip(a, out):
        assert lddmm.iota_noalloc(Ns, Ks, x, 3, y, stream) == 0
    torch.cuda.synchronize()
    with Context(Ns, Ks, ALPHA, S, SIGMA, 2, precision="fp32") as ctx:
        ref = torch.empty((3,) + Ns, dtype=torch.float32, device="cuda")
        for x, y in zip(a, out):
            ctx.iota(x, 3, ref)
            assert _rel(y.cpu().numpy(), ref.cpu().numpy()) < TOL
