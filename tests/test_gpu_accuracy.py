"""FP32 rounding errors against the FP64 oracle, as means over seeded inputs: the bracket
ad~^dagger on small bands and the projection of smooth images, whose sums of like signs
round the most.  The bounds are what complex half-spectrum sums gave on the same inputs
(ERRORS below, with 5% for the spread of the means)."""

import math

import numpy as np
import pytest

from oracle import bl
from paper_1807_11560_gb300 import Context, inputs

from helpers import ALPHA, S, SIGMA, host, quantise, torch_dev

pytestmark = pytest.mark.gpu

ERRORS = {"ad_dagger": 1.347e-7, "pi": 7.397e-8}


def _rel(a, b):
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel()))


def _mean(x):
    return math.exp(sum(math.log(v) for v in x) / len(x))


def ad_dagger_error():
    import torch
    Ks, errors = (16, 16, 16), []
    with Context(Ks, Ks, ALPHA, S, SIGMA, 1, precision="fp32") as ctx:
        out = torch.empty((3,) + Ks, device="cuda", dtype=torch.complex64)
        for seed in range(16):
            v, u = (quantise(inputs.random_bl(Ks, 3, 100 + 2 * seed + i, 2.0, (64, 64, 64)), "fp32") for i in range(2))
            ctx.ad_dagger(torch_dev(v, "fp32"), torch_dev(u, "fp32"), out)
            errors.append(_rel(host(out), bl.ad_dagger(v, u, ALPHA, S)))
    return _mean(errors)


def pi_error():
    import torch
    Ns, Ks, errors = (64, 64, 64), (16, 16, 16), []
    with Context(Ns, Ks, ALPHA, S, SIGMA, 1, precision="fp32") as ctx:
        out = torch.empty((3,) + Ks, device="cuda", dtype=torch.complex64)
        for seed in range(8):
            I0, I1 = inputs.make_pair("ellipsoids", Ns, 50 + seed, max_disp=2.0)
            f = quantise(np.stack([I0, I1, I0 * I1]), "fp32")
            ctx.pi(torch_dev(f, "fp32"), 3, out)
            errors.append(_rel(host(out), bl.pi(f, Ks)))
    return _mean(errors)


def test_bracket_of_a_small_band():
    assert ad_dagger_error() < 1.05 * ERRORS["ad_dagger"]


def test_projection_of_smooth_images():
    assert pi_error() < 1.05 * ERRORS["pi"]


@pytest.mark.parametrize("Ks", [(24, 24, 24), (8, 64, 64), (40, 40, 40)])
def test_persistent_sweeps_equal_launches_on_larger_bands(Ks):
    """Bands whose items share an SM sum in another order than the others: in both forms."""
    import torch
    v = quantise(inputs.random_bl(Ks, 3, 3, 2.0, Ks), "fp32")
    got = []
    for persistent in (False, True):
        with Context(Ks, Ks, ALPHA, S, SIGMA, 1, precision="fp32", persistent=persistent) as ctx:
            out = torch.empty((3,) + Ks, device="cuda", dtype=torch.complex64)
            ctx.shoot(torch_dev(v, "fp32"), out)
            got.append(out.cpu().numpy())
    np.testing.assert_array_equal(got[0], got[1])
