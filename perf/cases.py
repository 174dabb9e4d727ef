"""What the speed of this library is measured on: calls of its public entry
points over the sizes, options and directions that users run.

The sizes are those of the benchmark workloads (2D 64^2, 64^3 / 16^3, 96^3 /
24^3, 160x192x160 / 32^3), of the paper's band tables (band sizes 40 and 64,
grid 180x210x180) and of the batched population.  Inputs are seeded synthetic
phantoms made on the GPU: smoothed nested ellipsoidal shells (or Gaussian blobs
in 2D) and an analytically warped copy, with random band-limited velocities of
at most two voxels.

``exact`` restates the method in 64 bits with torch's FFTs (array-wide, no code
of the library): band-limited EPDiff with Heun steps, semi-Lagrangian transport,
the reduced adjoint Jacobi sweep and the Gauss-Newton product.
"""

import itertools
import math

import numpy as np
import torch

from paper_1807_11560_gb300 import Context, batch_gn_solve, inputs
from paper_1807_11560_gb300.autograd import shoot_transport

ALPHA, S, SIGMA = 0.0025, 2, 0.03
DEV = "cuda"


def _case(name, kind, grid, band, Nt=10, **more):
    d = {"name": name, "kind": kind, "Nt": Nt, "precision": "fp32", "state": "image"}
    d.update({f"n{j + 1}": n for j, n in enumerate(grid)})
    d.update({f"k{j + 1}": k for j, k in enumerate(band)})
    d.update(more)
    return d


def listed():
    return [
        # one bracket pair on a small band: the shortest calls, latency alone
        _case("brackets_64", "brackets", (64, 64, 64), (16, 16, 16)),
        # the 2D double-precision configuration: PCG's inner call on a tiny problem
        _case("product_2d_fp64", "product", (64, 64), (16, 16), precision="fp64"),
        # PCG's inner call on the 64^3 workload
        _case("product_64", "product", (64, 64, 64), (16, 16, 16)),
        # a whole Gauss-Newton-Krylov call: gradients, PCG and line searches
        _case("solve_64", "solve", (64, 64, 64), (16, 16, 16), n_gn=2, n_pcg=3),
        # training through the registration: m(1) and the gradient of a loss of it
        _case("autograd_96", "autograd", (96, 96, 96), (24, 24, 24), Nt=16, adjoint="jacobi"),
        # a small population solved at once, one stream each
        _case("population_96", "population", (96, 96, 96), (24, 24, 24), pairs=4, n_gn=1, n_pcg=3),
        # both transforms of a velocity on the large image grid
        _case("transforms_160", "transforms", (160, 192, 160), (32, 32, 32)),
        # the headline workload: the Gauss-Newton product, and its gradient
        _case("product_160", "product", (160, 192, 160), (32, 32, 32)),
        _case("gradient_160", "gradient", (160, 192, 160), (32, 32, 32)),
        # the same product subject to the deformation state equation
        _case("product_160_deformation", "product", (160, 192, 160), (32, 32, 32), state="deformation"),
        # the paper's grid (ragged sizes) with a band of its tables
        _case("product_180_band40", "product", (180, 210, 180), (40, 40, 40)),
        # the largest band of the paper's tables
        _case("product_160_band64", "product", (160, 192, 160), (64, 64, 64)),
    ]


def draw(rng):
    kind = rng.choice(["product"] * 5 + ["gradient"] * 2 + ["brackets", "transforms", "autograd"])

    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if kind == "product" and rng.random() < 0.2:
        grid, dims, precision = [size(32, 160) for _ in range(2)], 2, "fp64"
    else:
        grid, dims, precision = [size(24, 168) for _ in range(3)], 3, "fp32"
    k0 = size(8, 64)
    band = [min(64, max(6, int(round(k0 * rng.uniform(0.8, 1.2))))) for _ in range(dims)]
    band = [max(2, min(b, n) // 2 * 2) for b, n in zip(band, grid)]
    if dims == 2:
        band = [min(b, 32) for b in band]
    case = _case("", kind, grid, band, Nt=rng.choice([4, 6, 8, 10]), precision=precision)
    del case["name"]
    if kind == "product" and dims == 3:
        case["state"] = rng.choice(["image", "image", "image", "deformation"])
        if case["state"] == "image":
            case["recompute"] = rng.random() < 0.2
    if kind in ("product", "gradient") and dims == 3:
        case["precision"] = rng.choice(["fp32", "fp32", "fp32", "3xtf32", "bf16x3"])
    if kind == "autograd":
        case["adjoint"] = rng.choice(["jacobi", "exact"])
    return case


def _sizes(case):
    dims = 3 if "n3" in case else 2
    return (tuple(case[f"n{j + 1}"] for j in range(dims)), tuple(case[f"k{j + 1}"] for j in range(dims)))


# ---- inputs ------------------------------------------------------------------
def _phantom(X, grid, ph):
    """Nested shells with a folded boundary (3D), Gaussian blobs (2D)."""
    if len(grid) == 2:
        img = torch.zeros(grid, dtype=torch.float64, device=DEV)
        for b in range(8):
            r2 = 0.0
            for j, n in enumerate(grid):
                d = (X[j] - ph[b, j] * n + n / 2) % n - n / 2
                r2 = r2 + d * d
            img = img + ph[b, 2] * torch.exp(-r2 / (2 * ((3 + 5 * ph[b, 3]) * min(grid) / 64) ** 2))
        return img.clamp(0, 1)
    y = [(X[j] - n / 2) / (a * n) for j, (n, a) in enumerate(zip(grid, (0.40, 0.47, 0.36)))]
    r = torch.sqrt(y[0] ** 2 + y[1] ** 2 + y[2] ** 2)
    theta = torch.acos((y[2] / r.clamp_min(1e-12)).clamp(-1, 1))
    phi = torch.atan2(y[1], y[0])
    rho = 1 + 0.06 * torch.sin(7 * theta + 6.28 * ph[0, 0]) * torch.sin(9 * phi + 6.28 * ph[0, 1])
    img = 0.2 * (r < rho) + 0.3 * (r < 0.8 * rho) + 0.3 * (r < 0.55 * rho)
    w = torch.exp(-0.5 * torch.arange(-3, 4, device=DEV, dtype=torch.float64) ** 2)
    w = w / w.sum()
    for ax in range(3):
        img = sum(float(wt) * torch.roll(img, o, ax) for o, wt in zip(range(-3, 4), w))
    return img


def _images(grid, seed):
    """An image pair in 64 bits: a phantom and its copy under a smooth periodic warp."""
    rng = np.random.default_rng(seed)
    ph = rng.uniform(0.1, 1.0, size=(8, 4))
    X = torch.meshgrid(*[torch.arange(n, dtype=torch.float64, device=DEV) for n in grid], indexing="ij")
    warped = []
    for j in range(len(grid)):
        u = 0.0
        for _ in range(4):
            k = rng.integers(0, 3, size=len(grid))
            k[rng.integers(len(grid))] = 1
            arg = sum(2 * math.pi * float(k[i]) * X[i] / n for i, n in enumerate(grid))
            u = u + float(rng.normal()) * torch.sin(arg + float(rng.uniform(0, 2 * math.pi)))
        warped.append(X[j] - u * (2.0 / u.abs().max()))
    return _phantom(X, grid, ph), _phantom(warped, grid, ph)


def _data(case, seed):
    """Seeded inputs of a case at the precision of its context."""
    grid, band = _sizes(case)
    real = torch.float64 if case["precision"] == "fp64" else torch.float32
    cplx = torch.complex128 if case["precision"] == "fp64" else torch.complex64
    d = {}
    if case["kind"] not in ("brackets", "transforms", "population"):
        d["I0"], d["I1"] = (im.to(real) for im in _images(grid, seed))

    def field(k, disp):
        return torch.as_tensor(inputs.random_bl(band, len(grid), seed + k, disp, grid), device=DEV).to(cplx)

    d["v"], d["p"] = field(1, 2.0), field(2, 1.0)
    if case["kind"] in ("transforms", "autograd"):
        gen = torch.Generator(device=DEV).manual_seed(seed)
        shape = ((len(grid),) if case["kind"] == "transforms" else ()) + grid
        d["f"] = torch.randn(shape, generator=gen, device=DEV, dtype=torch.float32).to(real)
    return d


def _context(case, stream=None):
    grid, band = _sizes(case)
    return Context(grid, band, ALPHA, S, SIGMA, case["Nt"], precision=case["precision"], state=case["state"],
                   recompute=bool(case.get("recompute", False)), stream=stream)


def prepare(case, seed):
    st = dict(case)
    if case["kind"] == "population":
        st["streams"] = [torch.cuda.Stream() for _ in range(case["pairs"])]
        st["ctx"], st["v0"] = [], []
        for i, stream in enumerate(st["streams"]):
            ctx = _context(case, stream.cuda_stream)
            grid, band = _sizes(case)
            I0, I1 = (im.float() for im in _images(grid, seed + 101 * i))
            torch.cuda.synchronize()
            ctx.set_images(I0, I1)
            st["ctx"].append(ctx)
            st["v0"].append(torch.zeros((len(grid),) + band, dtype=torch.complex64, device=DEV))
        torch.cuda.synchronize()
        return st
    st.update(_data(case, seed))
    ctx = st["ctx"] = _context(case)
    if "I0" in st:
        ctx.set_images(st["I0"], st["I1"])
    if case["kind"] == "product":              # PCG multiplies at a linearisation point
        ctx.gradient(st["v"], torch.empty_like(st["v"]))
    return st


def run(st):
    kind, ctx = st["kind"], st["ctx"]
    if kind == "population":
        vs = [v.clone() for v in st["v0"]]
        torch.cuda.current_stream().synchronize()   # the contexts run on streams of their own
        reports = batch_gn_solve(ctx, vs, st["n_gn"], st["n_pcg"])
        return {"v": vs, "E": [r["E_final"] for r in reports]}
    v, p = st["v"], st["p"]
    if kind == "product":
        out = torch.empty_like(p)
        ctx.hessvec(p, out)
        return out
    if kind == "gradient":
        g = torch.empty_like(v)
        return {"E": ctx.gradient(v, g), "g": g}
    if kind == "solve":
        w = torch.zeros_like(v)
        rep = ctx.gn_solve(w, st["n_gn"], st["n_pcg"])
        return {"v": w, "E": rep["E_final"]}
    if kind == "autograd":
        w = v.clone().requires_grad_(True)
        m1 = shoot_transport(ctx, w, st["adjoint"])
        (g,) = torch.autograd.grad(m1, w, st["f"])
        return {"m1": m1.detach(), "g": g}
    if kind == "brackets":
        a, b = torch.empty_like(v), torch.empty_like(v)
        ctx.ad_dagger(v, p, a)
        ctx.ad(v, p, b)
        return {"ad_dagger": a, "ad": b}
    grid = torch.empty_like(st["f"])
    band = torch.empty_like(v)
    ctx.iota(v, ctx.ndim, grid)
    ctx.pi(st["f"], ctx.ndim, band)
    return {"iota": grid, "pi": band}


# ---- what a pass cannot do without -------------------------------------------
def work(case):
    """Bytes: images, velocities and results once, and per time step of a sweep on
    the image grid one read and one write of the transported image (and one read of
    the other image it needs).  Operations: the separable truncated transforms of
    the scalar fields that each bracket and each grid velocity needs, as real
    cosine and sine sums over half an axis each."""
    grid, band = _sizes(case)
    Nt, dims, kind = case["Nt"], len(grid), case["kind"]
    size = 8 if case["precision"] == "fp64" else 4
    N, K = float(np.prod(grid)), float(np.prod(band))
    pad = [math.ceil(1.5 * k) for k in band]

    def transform(out):                         # one scalar field, band to grid or back
        n, total = list(band), 0.0
        for j in range(dims):
            n[j] = out[j]
            total += float(np.prod(n)) * band[j]
        return total

    per = 14.0 if dims == 3 else 8.0            # fields of one ad_dagger bracket, in and out
    pair = 28.0 if dims == 3 else 15.0          # and of the bracket triple of the adjoint sweep
    shoot = 2 * Nt * per * transform(pad)
    adjoint = 2 * Nt * pair * transform(pad)
    levels = dims * (Nt + 1) * transform(grid)  # a velocity history on the image grid
    back = dims * transform(grid)
    vec = 2 * dims * K * size
    if kind == "brackets":
        return {"bytes": 4 * vec, "flops": (per + pair / 2) * transform(pad)}
    if kind == "transforms":
        return {"bytes": 2 * vec + 2 * dims * N * size, "flops": 2 * back}
    forward = {"bytes": 2 * Nt * N * size, "flops": shoot + levels}
    product = {"bytes": (3 * Nt + 2) * N * size + 2 * vec, "flops": shoot + levels + back + adjoint}
    gradient = {"bytes": forward["bytes"] + 3 * N * size + 2 * vec, "flops": forward["flops"] + back + adjoint}
    if case["state"] == "deformation":
        product = {"bytes": 8 * N * size + 2 * vec, "flops": 2 * shoot + 2 * back + adjoint}
        forward = {"bytes": 8 * N * size, "flops": 2 * shoot + back}
    if kind == "product":
        return product
    if kind == "gradient":
        return gradient
    if kind == "autograd":
        return {"bytes": forward["bytes"] + gradient["bytes"] + 2 * N * size, "flops": forward["flops"] + gradient["flops"]}
    n, m, pairs = case["n_gn"], case["n_pcg"], case.get("pairs", 1)
    return {k: pairs * n * (gradient[k] + m * product[k]) for k in ("bytes", "flops")}


# ---- the same results in 64 bits ----------------------------------------------
class _Exact:
    """The method in double precision on whole arrays (torch.fft for every transform)."""

    def __init__(self, case):
        self.grid, self.band = _sizes(case)
        self.d, self.Nt = len(self.grid), case["Nt"]
        self.dt = 1.0 / self.Nt
        self.pad = tuple(math.ceil(1.5 * k) for k in self.band)
        f = [torch.where(torch.arange(k) < k / 2, torch.arange(k), torch.arange(k) - k) for k in self.band]
        F = torch.meshgrid(*f, indexing="ij")
        self.F = [x.to(DEV, torch.float64) for x in F]
        self.mask = torch.ones(self.band, device=DEV, dtype=torch.float64)
        for x, k in zip(F, self.band):
            self.mask[(2 * x == -k).to(DEV)] = 0.0
        self.L = (1 + 4 * math.pi ** 2 * ALPHA * sum(x * x for x in self.F)) ** S
        self.f = f

    def _index(self, Ns):
        return torch.meshgrid(*[(x % n).to(DEV) for x, n in zip(self.f, Ns)], indexing="ij")

    def iota(self, a, Ns):
        S_ = torch.zeros(tuple(Ns), dtype=torch.complex128, device=DEV)
        S_[self._index(Ns)] = a * self.mask
        return torch.fft.ifftn(S_).real * float(np.prod(Ns))

    def pi(self, f):
        return torch.fft.fftn(f)[self._index(f.shape)] * self.mask / f.numel()

    def D(self, a, j):
        return 2j * math.pi * self.F[j] * a

    def hermitian(self, a):
        b = a
        for ax, k in enumerate(self.band, start=1):
            b = b.index_select(ax, (-torch.arange(k, device=DEV)) % k)
        return 0.5 * (a + b.conj()) * self.mask

    def fields(self, a):
        d, M = self.d, self.pad
        return ([self.iota(a[i], M) for i in range(d)],
                [[self.iota(self.D(a[i], j), M) for j in range(d)] for i in range(d)])

    def star(self, v, m):
        """sum_j (d_i v_j) m_j + (d_j m_i) v_j + m_i div v from (values, Jacobian) pairs."""
        (vv, dv), (mm, dm), d = v, m, self.d
        div = sum(dv[j][j] for j in range(d))
        return torch.stack([self.pi(mm[i] * div + sum(dv[j][i] * mm[j] + dm[i][j] * vv[j] for j in range(d)))
                            for i in range(d)]) / self.L

    def bracket(self, v, w):
        (vv, dv), (ww, dw), d = v, w, self.d
        return torch.stack([self.pi(sum(dv[i][j] * ww[j] - dw[i][j] * vv[j] for j in range(d))) for i in range(d)])

    # a stage point's fields: (v, L v)
    def point(self, v):
        return self.fields(v), self.fields(self.L * v)

    def shoot(self, v0):
        vs, stars, pts = [v0], [], []
        for _ in range(self.Nt):
            v, k = vs[-1], []
            for x in (v, None):
                if x is None:
                    x = v + self.dt * k[0]
                    stars.append(x)
                pts.append(self.point(x))
                k.append(-self.star(*pts[-1]))
            vs.append(v + 0.5 * self.dt * (k[0] + k[1]))
        return vs, stars, pts

    def tangent(self, pts, p):
        out, stars = [p], []
        for n in range(self.Nt):
            d0, k = out[-1], []
            for r, x in enumerate((d0, None)):
                if x is None:
                    x = d0 + self.dt * k[0]
                    stars.append(x)
                (v, m), (dv, dm) = pts[2 * n + r], self.point(x)
                k.append(-self.star(dv, m) - self.star(v, dm))
            out.append(d0 + 0.5 * self.dt * (k[0] + k[1]))
        return out, stars

    def adjoint(self, pts, U, sources=None):
        """The reduced adjoint Jacobi sweep from (U, 0), or with a band source per level."""
        dt = self.dt
        W = torch.zeros_like(U) if sources is None else sources[-1]

        def G(pt, U, W):
            (v, m), w = pt, self.fields(W)
            a = self.star(w, m) - self.bracket(v, w)
            return (self.star(v, self.fields(self.L * U)), a + U) if sources is None else (U, a)

        for n in range(self.Nt - 1, -1, -1):
            aU, aW = G(pts[2 * n + 1], U, W)
            bU, bW = G(pts[2 * n], U + dt * aU if sources is None else U, W + dt * aW)
            if sources is None:
                U = U + 0.5 * dt * (aU + bU)
            W = W + 0.5 * dt * (aW + bW)
            if sources is not None:
                W = W + sources[n]
        return W

    # ---- the image grid
    def cells(self, disp):
        """Corner indices (per axis) and weights of x - disp (index units)."""
        cell = []
        for j, n in enumerate(self.grid):
            x = torch.arange(n, device=DEV).reshape([-1 if i == j else 1 for i in range(self.d)])
            fl = torch.floor(-disp[j])
            c = (x + fl.long()) % n
            cell.append((c, (c + 1) % n, -disp[j] - fl))
        return cell

    def corners(self, cell):
        for bits in itertools.product((0, 1), repeat=self.d):
            idx, w = 0, 1.0
            for b, n, (c0, c1, f) in zip(bits, self.grid, cell):
                idx = idx * n + (c1 if b else c0)
                w = w * (f if b else 1 - f)
            yield bits, idx, w

    def at(self, f, cell):
        flat = f.reshape(-1)
        return sum(w * flat[idx] for _, idx, w in self.corners(cell))

    def slope(self, f, cell):
        """Derivatives of the interpolant with respect to the index coordinates."""
        flat, out = f.reshape(-1), []
        for j in range(self.d):
            one = [(c0, c1, torch.ones_like(w) if i == j else w) for i, (c0, c1, w) in enumerate(cell)]
            g = 0.0
            for bits, idx, w in self.corners([(c0, c1, w) for c0, c1, w in one]):
                weight = 1.0
                for i, b in enumerate(bits):
                    if i != j:
                        weight = weight * (cell[i][2] if b else 1 - cell[i][2])
                g = g + (weight if bits[j] else -weight) * flat[idx]
            out.append(g)
        return out

    def scatter(self, f, cell, into):
        for _, idx, w in self.corners(cell):
            into.view(-1).index_add_(0, idx.reshape(-1), (w * f).reshape(-1))

    def grad(self, m):
        return torch.stack([(torch.roll(m, -1, j) - torch.roll(m, 1, j)) * (0.5 * n)
                            for j, n in enumerate(self.grid)])

    def velocity(self, a):
        return torch.stack([self.iota(a[i], self.grid) for i in range(self.d)])

    def transport(self, I0, vs):
        n = torch.tensor(self.grid, device=DEV, dtype=torch.float64).reshape([-1] + [1] * self.d)
        ms, feet, cur = [I0], [], self.velocity(vs[0])
        for v in vs[1:]:
            nxt = self.velocity(v)
            mid = self.cells(self.dt * n * nxt)
            u = torch.stack([self.at(cur[j], mid) for j in range(self.d)])
            feet.append(self.cells(0.5 * self.dt * n * (nxt + u)))
            ms.append(self.at(ms[-1], feet[-1]))
            cur = nxt
        return ms, feet

    def project(self, f3):
        return torch.stack([self.pi(f) for f in f3])

    def linearise(self, I0, v0):
        vs, stars, pts = self.shoot(v0)
        ms, feet = self.transport(I0, vs)
        return {"v0": v0, "vs": vs, "stars": stars, "pts": pts, "ms": ms, "feet": feet}

    def energy(self, v0, m1, I1):
        reg = 0.5 * float((self.L * (v0.abs() ** 2)).sum())
        return reg + float(((m1 - I1) ** 2).sum()) / I1.numel() / SIGMA ** 2

    def gradient(self, lin, I1):
        m1 = lin["ms"][-1]
        U = self.project(-2 / SIGMA ** 2 * (m1 - I1) * self.grad(m1)) / self.L
        return self.energy(lin["v0"], m1, I1), lin["v0"] + self.adjoint(lin["pts"], U)

    def product(self, lin, p):
        dvs, _ = self.tangent(lin["pts"], p)
        dm, src = None, (self.grad(lin["ms"][0]) * self.velocity(dvs[0])).sum(0)
        for n in range(self.Nt):
            new = (self.grad(lin["ms"][n + 1]) * self.velocity(dvs[n + 1])).sum(0)
            moved = self.at(src, lin["feet"][n]) + new
            dm = (0.0 if dm is None else self.at(dm, lin["feet"][n])) - 0.5 * self.dt * moved
            src = new
        U = self.project(-2 / SIGMA ** 2 * dm * self.grad(lin["ms"][-1])) / self.L
        return p + self.adjoint(lin["pts"], U)

    # ---- the deformation state equation
    def convolve(self, Du, v, transpose=False):
        return torch.stack([self.pi(sum((Du[j][i] if transpose else Du[i][j]) * v[j] for j in range(self.d)))
                            for i in range(self.d)])

    def product_deformation(self, I0, v0, p):
        vs, stars, pts = self.shoot(v0)
        dvs, dstars = self.tangent(pts, p)
        u, du, dt = torch.zeros_like(v0), torch.zeros_like(v0), self.dt
        for n in range(self.Nt):
            x, dx, k, dk = u, du, [], []
            for v, dv in ((vs[n], dvs[n]), (stars[n], dstars[n])):
                if k:
                    x, dx = u + dt * k[0], du + dt * dk[0]
                g, dg = self.fields(v)[0], self.fields(dv)[0]
                Dx, Ddx = self.fields(x)[1], self.fields(dx)[1]
                k.append(-v - self.convolve(Dx, g))
                dk.append(-dv - self.convolve(Ddx, g) - self.convolve(Dx, dg))
            u, du = u + 0.5 * dt * (k[0] + k[1]), du + 0.5 * dt * (dk[0] + dk[1])
        n = torch.tensor(self.grid, device=DEV, dtype=torch.float64).reshape([-1] + [1] * self.d)
        cell = self.cells(-n * self.velocity(u))
        gs = torch.stack([self.at(g, cell) for g in self.grad(I0)])
        dm = (gs * self.velocity(du)).sum(0)
        r = self.project(-2 / SIGMA ** 2 * dm * gs)
        U = (r + self.convolve(self.fields(u)[1], self.fields(r)[0], transpose=True)) / self.L
        return p + self.adjoint(pts, U)

    # ---- vector-Jacobian products of v0 -> m(1)
    def vjp_jacobi(self, lin, gm):
        m1 = lin["ms"][-1]
        U = self.project(-float(np.prod(self.grid)) * gm * self.grad(m1)) / self.L
        return self.L * self.adjoint(lin["pts"], U)

    def vjp_exact(self, lin, gm):
        dt, d = self.dt, self.d
        vg = [self.velocity(v) for v in lin["vs"]]
        G = [torch.zeros_like(vg[0]) for _ in vg]
        lam = gm
        for n in range(self.Nt - 1, -1, -1):
            back = torch.zeros_like(lam)
            self.scatter(lam, lin["feet"][n], back)
            dmdx = self.slope(lin["ms"][n], lin["feet"][n])
            alpha = [-0.5 * dt * self.grid[j] * lam * dmdx[j] for j in range(d)]
            mid = self.cells(torch.stack([dt * self.grid[j] * vg[n + 1][j] for j in range(d)]))
            for j in range(d):
                self.scatter(alpha[j], mid, G[n][j])
            du = [self.slope(vg[n][j], mid) for j in range(d)]
            for i in range(d):
                G[n + 1][i] += alpha[i] - dt * self.grid[i] * sum(alpha[j] * du[j][i] for j in range(d))
            lam = back
        srcs = [self.project(g) * float(np.prod(self.grid)) / self.L for g in G]
        return self.L * self.adjoint(lin["pts"], torch.zeros_like(lin["v0"]), srcs)

    # ---- Gauss-Newton-Krylov
    def dot(self, a, b):
        return float((self.L * (a.conj() * b).real).sum())

    def solve(self, I0, I1, v, n_gn, n_pcg):
        E = None
        for _ in range(n_gn):
            lin = self.linearise(I0, v)
            E, g = self.gradient(lin, I1)
            x, r = torch.zeros_like(g), -g
            dvec, rho = r, self.dot(r, r)
            for _ in range(n_pcg):
                q = self.product(lin, dvec)
                a = rho / self.dot(dvec, q)
                x, r = x + a * dvec, r - a * q
                rho, old = self.dot(r, r), rho
                dvec = r + rho / old * dvec
            slope, eps = self.dot(g, x), 1.0
            for _ in range(11):
                trial = v + eps * x
                Et = self.energy(trial, self.transport(I0, self.shoot(trial)[0])[0][-1], I1)
                if Et <= E + 1e-4 * eps * slope:
                    v, E = trial, Et
                    break
                eps *= 0.5
        return v, E


def exact(case, seed):
    ex = _Exact(case)
    kind = case["kind"]
    if kind == "population":
        got = []
        for i in range(case["pairs"]):
            I0, I1 = (im.float().double() for im in _images(ex.grid, seed + 101 * i))
            zero = torch.zeros((ex.d,) + ex.band, dtype=torch.complex128, device=DEV)
            got.append(ex.solve(I0, I1, zero, case["n_gn"], case["n_pcg"]))
        return {"v": [v for v, _ in got], "E": [E for _, E in got]}
    data = _data(case, seed)
    v, p = (ex.hermitian(data[k].to(torch.complex128)) for k in ("v", "p"))
    if kind == "brackets":
        return {"ad_dagger": ex.star(ex.fields(v), ex.fields(ex.L * p)), "ad": ex.bracket(ex.fields(v), ex.fields(p))}
    if kind == "transforms":
        return {"iota": ex.velocity(v), "pi": ex.project(data["f"].double())}
    I0, I1 = data["I0"].double(), data["I1"].double()
    if kind == "solve":
        w, E = ex.solve(I0, I1, torch.zeros_like(v), case["n_gn"], case["n_pcg"])
        return {"v": w, "E": E}
    if kind == "product" and case["state"] == "deformation":
        return ex.product_deformation(I0, v, p)
    lin = ex.linearise(I0, v)
    if kind == "product":
        return ex.product(lin, p)
    if kind == "gradient":
        E, g = ex.gradient(lin, I1)
        return {"E": E, "g": g}
    vjp = ex.vjp_exact if case["adjoint"] == "exact" else ex.vjp_jacobi
    return {"m1": lin["ms"][-1], "g": vjp(lin, data["f"].double())}
