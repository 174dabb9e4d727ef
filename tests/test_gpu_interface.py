"""The reporting calls of the C interface: work split, probe and launch counter."""

import numpy as np
import pytest

from oracle import bl
from paper_1807_11560_gb300 import Context, inputs

from helpers import ALPHA, S, SIGMA, rel_2, torch_dev

pytestmark = pytest.mark.gpu


# (grid = band, plane parts per x1 column, quads per band item): the padded row pairs of
# the second axis (13 at band 16, 25 at 32) in items of at most 3 and 9; one plane item in 2D
@pytest.mark.parametrize("Ks,parts,quads", [((16, 16, 16), 5, 1), ((32, 32, 32), 3, 2), ((16, 16), 1, 1)])
def test_tiles_are_parts_and_quads(Ks, parts, quads):
    with Context(Ks, Ks, ALPHA, S, SIGMA, 1, precision="fp32") as ctx:
        assert ctx.tiles == (2, parts, quads)


def _probed(ctx, kernel_class, call):
    """(ms, launches, work) of one kernel class during call()."""
    ctx.probe(kernel_class)
    call()
    got = ctx.probe_read()
    ctx.probe(None)
    return got


@pytest.mark.parametrize("persistent", [False, True])
def test_probe_counts_the_operations_of_2d_evaluations(persistent):
    """A 2D shoot evaluation transforms 9 fields in and 3 out over two axes (K/2 products
    of two sums a point and axis) and takes 10 operations a point for the products."""
    import torch
    (K1, K2), Nt = (14, 10), 3
    M1, M2 = 21, 15
    band, plane = 12 * K1 * M1 * K2, 12 * M1 * K2 * M2 + 10 * M1 * M2
    v = torch_dev(inputs.random_bl((K1, K2), 2, 3, 1.0, (K1, K2)), "fp32")
    with Context((K1, K2), (K1, K2), ALPHA, S, SIGMA, Nt, precision="fp32", persistent=persistent) as ctx:
        shoot = lambda: ctx.shoot(v, torch.empty_like(v))
        if persistent:
            expect = {"sweep": (1, 2 * Nt * (band + plane))}
        else:
            expect = {"pi_ba": (2 * Nt + 1, 2 * Nt * band), "cpw": (2 * Nt, 2 * Nt * plane)}
        for kernel_class, (launches, work) in expect.items():
            ms, n, w = _probed(ctx, kernel_class, shoot)
            assert n == launches and ms > 0
            assert w == pytest.approx(work, rel=1e-12)


def test_probe_times_deformation_evaluations():
    """A deformation gradient: 2 Nt evaluations of the sweep and one of the terminal
    product, each sweep ended by a projection; 12 fields in and 3 out of each."""
    import torch
    Ns, (K1, K2, K3), Nt = (12, 12, 12), (8, 6, 4), 3
    M1, M2, M3 = 12, 9, 6
    v = torch_dev(inputs.random_bl((K1, K2, K3), 3, 3, 1.0, Ns), "fp32")
    I0, I1 = inputs.make_pair("ellipsoids", Ns, 5, max_disp=1.0)
    with Context(Ns, (K1, K2, K3), ALPHA, S, SIGMA, Nt, precision="fp32", state="deformation") as ctx:
        ctx.set_images(torch_dev(I0, "fp32"), torch_dev(I1, "fp32"))
        ms, n, work = _probed(ctx, "deform", lambda: ctx.gradient(v, torch.empty_like(v)))
        assert n == (2 * Nt + 1) + (1 + 1) and ms > 0
        transforms = 15 * (K1 * M1 * K2 * K3 + M1 * K2 * M2 * K3 + M1 * M2 * K3 * M3)
        assert work == pytest.approx((2 * Nt + 1) * transforms + (2 * Nt * 21 + 18) * M1 * M2 * M3, rel=1e-12)
        # the classes of the bracket kernels leave them out
        assert _probed(ctx, "cpw", lambda: ctx.gradient(v, torch.empty_like(v)))[1] == 2 * (2 * Nt)


@pytest.mark.parametrize("Ns,Ks", [((12, 10, 9), (8, 6, 4)), ((12, 10), (6, 2)), ((40, 40, 40), (4, 40, 36))])
def test_pi_writes_the_hermitian_array_in_its_two_kernels(Ns, Ks):
    """The projection's second kernel writes every slot of the caller's array, the zero
    Nyquist slots among them, without a launch of its own for that."""
    import torch
    d = len(Ns)
    f = np.random.default_rng(5).normal(size=(d,) + Ns).astype(np.float32)
    with Context(Ns, Ks, ALPHA, S, SIGMA, 1, precision="fp32") as ctx:
        for out in (np.full((d,) + Ks, np.nan, np.complex64),
                    torch.full((d,) + Ks, float("nan"), dtype=torch.complex64, device="cuda")):
            before = ctx.kernel_count
            ctx.pi(f, d, out)
            assert ctx.kernel_count - before == 2
            got = np.asarray(out if isinstance(out, np.ndarray) else out.cpu())
            assert rel_2(got.astype(np.complex128), bl.pi(f.astype(np.float64), Ks)) < 2e-6
            for axis, k in enumerate(Ks):
                assert not np.take(got, k // 2, axis + 1).any()


@pytest.mark.parametrize("state", ["image", "deformation"])
def test_probe_changes_no_result(state):
    """Gradient and product (captured and replayed) with every class probed and with none."""
    import torch
    Ns, Ks, Nt = (20, 18, 15), (8, 6, 4), 3
    v = torch_dev(inputs.random_bl(Ks, 3, 3, 1.0, Ns), "fp32")
    p = torch_dev(inputs.random_bl(Ks, 3, 4, 1.0, Ns), "fp32")
    I0, I1 = (torch_dev(x, "fp32") for x in inputs.make_pair("ellipsoids", Ns, 5, max_disp=1.0))
    with Context(Ns, Ks, ALPHA, S, SIGMA, Nt, precision="fp32", state=state) as ctx:
        ctx.set_images(I0, I1)

        def results():
            g, h = torch.empty_like(v), torch.empty_like(v)
            E = ctx.gradient(v, g)
            for _ in range(2):
                ctx.hessvec(p, h)
            return E, g.cpu().numpy(), h.cpu().numpy()

        ref = results()
        for kernel_class in ("cpw", "pi_ba", "deform", "transport", "inc_step", "iota_full", "pi_full", "sweep"):
            ctx.probe(kernel_class)
            got = results()
            ctx.probe_read()
            assert got[0] == ref[0]
            np.testing.assert_array_equal(got[1], ref[1])
            np.testing.assert_array_equal(got[2], ref[2])
