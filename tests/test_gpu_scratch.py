"""Images with a long first axis and a thin band: the image-grid transforms run in groups
of velocities and in serial parts, so that the scratch does not grow with the first axis;
against the FP64 oracle, with the tolerances of the transform and product tests."""

import numpy as np
import pytest

from oracle import bl
from paper_1807_11560_gb300 import Context, inputs

from helpers import ALPHA, S, SIGMA, host, problem, quantise, rel_2, rel_V, torch_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("recompute", [False, True])
def test_the_scratch_stays_small_beside_the_image(recompute):
    """One time step keeps about 34 values a voxel on the image grid; with the scratch of
    33 fields at once a context of this shape held 71."""
    Ns = (4096, 16, 16)
    with Context(Ns, (2, 16, 16), ALPHA, S, SIGMA, 1, precision="fp32", recompute=recompute) as ctx:
        assert ctx.device_bytes < 50 * 4 * int(np.prod(Ns))


# several items of row pairs one after another into one partial plane
@pytest.mark.parametrize("Ns,Ks,precision", [((1024, 300, 40), (4, 200, 40), "fp32"),
                                             ((2048, 120, 24), (2, 116, 24), "fp64"),
                                             ((2500, 120, 23), (2, 116, 22), "fp32")])
def test_transforms_in_serial_parts(Ns, Ks, precision):
    import torch
    tol = 1e-11 if precision == "fp64" else 2e-6
    a = quantise(inputs.random_bl(Ks, 3, 3, 2.0, Ns)[:1], precision)
    f = quantise(np.random.default_rng(5).normal(size=(1,) + Ns), precision)
    wide = precision == "fp64"
    with Context(Ns, Ks, ALPHA, S, SIGMA, 1, precision=precision, recompute=True) as ctx:
        out = torch.empty((1,) + Ns, device="cuda", dtype=torch.float64 if wide else torch.float32)
        outk = torch.empty((1,) + Ks, device="cuda", dtype=torch.complex128 if wide else torch.complex64)
        ctx.iota(torch_dev(a, precision), 1, out)
        assert rel_2(host(out), bl.iota(a, Ns)) < tol
        ctx.pi(torch_dev(f, precision), 1, outk)
        assert rel_2(host(outk), bl.pi(f, Ks)) < tol


def test_product_with_velocities_in_groups():
    """11 levels of velocities in groups of 9 and 2."""
    import torch
    Ns, Ks = (1500, 20, 20), (4, 20, 20)
    ctx, P, v0, p = problem("ellipsoids", Ns, Ks, 11, 10, "fp32")
    g, Hp = (torch.empty(v0.shape, device="cuda", dtype=torch.complex64) for _ in range(2))
    lin = P.gradient(v0)
    ctx.gradient(torch_dev(v0, "fp32"), g)
    ctx.hessvec(torch_dev(p, "fp32"), Hp)
    assert rel_V(host(g), lin.g, Ks) < 1e-5
    assert rel_V(host(Hp), P.hessvec(lin, p), Ks) < 1e-5
    ctx.close()
