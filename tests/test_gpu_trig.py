"""The folded cosine/sine transforms at the sizes where their kernels switch: every
row-tile height of the plane phase, columns that need several passes, band items one
and two to an SM, the image-grid kernels' edges of tiles, the 2D kernels, and device
pointers used in place; against the FP64 oracle.  Tolerances are those of the
per-transform and per-product tests of the other modules."""

import gc

import numpy as np
import pytest

from oracle import bl, deformation
from paper_1807_11560_gb300 import Context, inputs

from helpers import ALPHA, S, SIGMA, host, problem, quantise, rel_2, rel_V, torch_dev

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-11, "fp32": 2e-6}
GRAD_TOL = {"fp64": 1e-9, "fp32": 1e-5}

# band -> what it reaches: plane items of 1, 3, 5 and 9 row pairs, more pairs than one
# pass takes, thin and long axes, band items two to an SM, K2/2 below and above 16
BANDS = [(2, 2, 2), (4, 8, 6), (6, 34, 2), (16, 16, 16), (24, 24, 24), (64, 6, 10), (60, 14, 22), (26, 30, 34),
         (32, 32, 32), (40, 40, 40), (64, 30, 44)]


@pytest.fixture(autouse=True, scope="module")
def _no_garbage():
    """Tracebacks of the tests before keep device tensors in reference cycles; drop
    them here, so that they are not freed in the middle of a later memory check."""
    gc.collect()
    yield
    gc.collect()


def _empty(shape, precision, cplx):
    import torch
    wide = precision == "fp64"
    dt = (torch.complex128 if wide else torch.complex64) if cplx else (torch.float64 if wide else torch.float32)
    return torch.empty(shape, device="cuda", dtype=dt)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("Ks", BANDS + [(2, 2), (14, 10), (40, 32), (64, 64)])
def test_brackets_at_the_switches(Ks, precision):
    d, Ns = len(Ks), Ks
    v = quantise(inputs.random_bl(Ks, d, 7, 3.0, Ns), precision)
    u = quantise(inputs.random_bl(Ks, d, 8, 3.0, Ns), precision)
    with Context(Ns, Ks, ALPHA, S, SIGMA, 1, precision=precision) as ctx:
        out = _empty((d,) + Ks, precision, True)
        for got, ref in ((ctx.ad_dagger, bl.ad_dagger(v, u, ALPHA, S)), (ctx.ad, bl.ad(v, u))):
            got(torch_dev(v, precision), torch_dev(u, precision), out)
            if np.abs(ref).max() < 1e-12:     # two slots an axis: the constant mode alone, whose bracket is 0
                assert np.abs(host(out)).max() < 1e-6
            else:
                assert rel_2(host(out), ref) < 10 * TOL[precision]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("Ns,Ks", [((2, 2, 2), (2, 2, 2)), ((9, 64, 66), (6, 20, 10)), ((33, 63, 65), (32, 6, 30)),
                                   ((31, 127, 33), (4, 32, 32)), ((64, 34, 129), (64, 2, 16)),
                                   ((70, 12, 258), (40, 12, 40)), ((3, 3), (2, 2)), ((65, 31), (40, 30))])
def test_image_transforms_at_tile_edges(Ns, Ks, precision):
    d = len(Ns)
    a = quantise(inputs.random_bl(Ks, d, 3, 2.0, Ns), precision)
    f = quantise(np.random.default_rng(5).normal(size=(d,) + Ns), precision)
    with Context(Ns, Ks, ALPHA, S, SIGMA, 1, precision=precision) as ctx:
        for n in (1, d):
            out = _empty((n,) + Ns, precision, False)
            ctx.iota(torch_dev(a[:n], precision), n, out)
            assert rel_2(host(out), bl.iota(a[:n], Ns)) < TOL[precision]
            outk = _empty((n,) + Ks, precision, True)
            ctx.pi(torch_dev(f[:n], precision), n, outk)
            assert rel_2(host(outk), bl.pi(f[:n], Ks)) < TOL[precision]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("Ns,Ks", [((17, 35, 9), (6, 34, 4)), ((24, 24, 24), (24, 24, 24)),
                                   ((64, 14, 23), (60, 14, 22)), ((40, 41, 42), (40, 40, 40)),
                                   ((31, 29), (14, 10)), ((48, 33), (40, 32))])
def test_products_at_the_switches(Ns, Ks, precision):
    ctx, P, v0, p = problem("ellipsoids" if len(Ns) == 3 else "blobs", Ns, Ks, 11, 2, precision)
    g, Hp = _empty(v0.shape, precision, True), _empty(v0.shape, precision, True)
    lin = P.gradient(v0)
    ctx.gradient(torch_dev(v0, precision), g)
    ctx.hessvec(torch_dev(p, precision), Hp)
    assert rel_V(host(g), lin.g, Ks) < GRAD_TOL[precision]
    assert rel_V(host(Hp), P.hessvec(lin, p), Ks) < GRAD_TOL[precision]
    ctx.close()


@pytest.mark.parametrize("Ns,Ks", [((24, 24, 24), (24, 24, 24)), ((40, 41, 42), (40, 40, 40)), ((48, 33), (40, 32))])
def test_deformation_products_at_the_switches(Ns, Ks):
    I0, I1 = inputs.make_pair("ellipsoids" if len(Ns) == 3 else "blobs", Ns, 11, max_disp=2.0)
    I0, I1 = quantise(I0, "fp32"), quantise(I1, "fp32")
    v0 = quantise(inputs.random_bl(Ks, len(Ns), 12, 2.0, Ns), "fp32")
    P = deformation.DeformationProblem(I0, I1, Ks, ALPHA, S, SIGMA, 2)
    with Context(Ns, Ks, ALPHA, S, SIGMA, 2, precision="fp32", state="deformation") as ctx:
        ctx.set_images(torch_dev(I0, "fp32"), torch_dev(I1, "fp32"))
        g = _empty(v0.shape, "fp32", True)
        ctx.gradient(torch_dev(v0, "fp32"), g)
        assert rel_V(host(g), P.gradient(v0).g, Ks) < GRAD_TOL["fp32"]


def test_device_arrays_of_any_offset_equal_host_arrays():
    import torch
    Ns, Ks = (20, 18, 15), (8, 6, 4)
    a = np.concatenate([inputs.random_bl(Ks, 3, 3, 2.0, Ns), inputs.random_bl(Ks, 3, 4, 2.0, Ns)[:1]]).astype(np.complex64)
    f = np.random.default_rng(5).normal(size=(4,) + Ns).astype(np.float32)
    with Context(Ns, Ks, ALPHA, S, SIGMA, 2, precision="fp32") as ctx:
        grid, band = np.empty((4,) + Ns, np.float32), np.empty((4,) + Ks, np.complex64)
        ctx.iota(a, 4, grid)
        ctx.pi(f, 4, band)
        for off in (0, 1, 3):
            def view(x):
                flat = torch.empty(x.size + off, device="cuda", dtype=torch.as_tensor(x).dtype)
                flat[off:] = torch.as_tensor(x).cuda().reshape(-1)
                return flat[off:].view(x.shape)
            out = view(np.zeros_like(grid))
            ctx.iota(view(a), 4, out)
            np.testing.assert_array_equal(out.cpu().numpy(), grid)
            out = view(np.zeros_like(band))
            ctx.pi(view(f), 4, out)
            np.testing.assert_array_equal(out.cpu().numpy(), band)
            both = view(a[:3])
            ref = np.empty((3,) + Ks, np.complex64)
            ctx.ad_dagger(a[:3], a[:3], ref)
            ctx.ad_dagger(both, both, both)       # the result over its own inputs
            np.testing.assert_array_equal(both.cpu().numpy(), ref)
