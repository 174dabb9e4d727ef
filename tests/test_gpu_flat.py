"""2D problems whose second axis is long and whose first is short: a plane is cut into
several items (parts), in the evaluations and in the image-grid projection.  Against the
FP64 oracle, with the tolerances of the transform and product tests."""

import numpy as np
import pytest

from oracle import bl
from paper_1807_11560_gb300 import Context, inputs

from helpers import ALPHA, S, SIGMA, host, problem, quantise, rel_2, rel_V, torch_dev

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-11, "fp32": 2e-6}
GRAD_TOL = {"fp64": 1e-9, "fp32": 1e-5}


def _empty(shape, precision, cplx):
    import torch
    wide = precision == "fp64"
    dt = (torch.complex128 if wide else torch.complex64) if cplx else (torch.float64 if wide else torch.float32)
    return torch.empty(shape, device="cuda", dtype=dt)


def test_few_planes_keep_the_device_busy():
    """12 padded planes of 385 row pairs: at least one item per two SMs."""
    with Context((8, 512), (8, 512), ALPHA, S, SIGMA, 1, precision="fp32") as ctx:
        assert 12 * ctx.tiles[1] >= 76


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("Ks", [(2, 90), (8, 60), (4, 302), (8, 512)])
def test_brackets(Ks, precision):
    v = quantise(inputs.random_bl(Ks, 2, 7, 3.0, Ks), precision)
    u = quantise(inputs.random_bl(Ks, 2, 8, 3.0, Ks), precision)
    with Context(Ks, Ks, ALPHA, S, SIGMA, 1, precision=precision) as ctx:
        out = _empty((2,) + Ks, precision, True)
        for got, ref in ((ctx.ad_dagger, bl.ad_dagger(v, u, ALPHA, S)), (ctx.ad, bl.ad(v, u))):
            got(torch_dev(v, precision), torch_dev(u, precision), out)
            assert rel_2(host(out), ref) < 10 * TOL[precision]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("Ns,Ks", [((5, 128), (4, 64)), ((4, 513), (4, 300)), ((9, 1000), (8, 34))])
def test_image_transforms(Ns, Ks, precision):
    a = quantise(inputs.random_bl(Ks, 2, 3, 2.0, Ns), precision)
    f = quantise(np.random.default_rng(5).normal(size=(2,) + Ns), precision)
    with Context(Ns, Ks, ALPHA, S, SIGMA, 1, precision=precision) as ctx:
        out, outk = _empty((2,) + Ns, precision, False), _empty((2,) + Ks, precision, True)
        ctx.iota(torch_dev(a, precision), 2, out)
        assert rel_2(host(out), bl.iota(a, Ns)) < TOL[precision]
        ctx.pi(torch_dev(f, precision), 2, outk)
        assert rel_2(host(outk), bl.pi(f, Ks)) < TOL[precision]


@pytest.mark.parametrize("persistent", [False, True])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("Ns,Ks", [((12, 200), (8, 120)), ((15, 131), (6, 130))])
def test_products(Ns, Ks, precision, persistent):
    ctx, P, v0, p = problem("blobs", Ns, Ks, 11, 2, precision, persistent=persistent)
    g, Hp = _empty(v0.shape, precision, True), _empty(v0.shape, precision, True)
    lin = P.gradient(v0)
    ctx.gradient(torch_dev(v0, precision), g)
    ctx.hessvec(torch_dev(p, precision), Hp)
    assert rel_V(host(g), lin.g, Ks) < GRAD_TOL[precision]
    assert rel_V(host(Hp), P.hessvec(lin, p), Ks) < GRAD_TOL[precision]
    ctx.close()
