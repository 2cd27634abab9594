"""Two-step transform plans: a line of N = A B points as B butterflies of radix A, twiddles, and A
butterflies of radix B, restated on the host for every length the kernels ship, and the kernels
themselves on grids that use them.

The kernel lists its lengths in ``csrc/fft2.cuh`` as X(N, A, B); the CPU test reads that list, so a
length added there is checked here.  The forward transform of H psi runs the inverse's two steps
backwards, which is what lets the potential multiply sit between them in registers."""
import os
import re

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1406_7803_gb300", "csrc")
TEXT = open(os.path.join(CSRC, "fft2.cuh")).read()


def plans(prefix):
    lines = re.findall(r"#define %s\d\(X\)((?:.*\\\n)*.*)" % prefix, TEXT)
    return [tuple(map(int, m)) for line in lines for m in re.findall(r"X\((\d+), (\d+), (\d+)\)", line)]


LINES = plans("FDE_SPLIT_SIDES") + plans("FDE_SPLIT_LONG")   # (N, A, B), A <= B: z lines
PLANES = plans("FDE_PLANE_SIDES")                            # (N, R1, R2), R1 >= R2: plane sides, strided axes
SIDES = [p[0] for p in PLANES]


def dft(x, sign):
    k = np.arange(len(x))
    return np.exp(sign * 2j * np.pi * np.outer(k, k) / len(x)) @ x


def indices(n, r1, r2, prime_factor):
    """Input index of (item j, element r) and output index of (item q, element p)."""
    if not prime_factor:
        return (lambda j, r: j + r2 * r), (lambda q, p: q + r1 * p)
    e1 = next(k for k in range(n) if k % r1 == 1 % r1 and k % r2 == 0)
    e2 = next(k for k in range(n) if k % r1 == 0 and k % r2 == 1 % r2)
    return (lambda j, r: (r1 * j + r2 * r) % n), (lambda q, p: (q * e1 + p * e2) % n)


def check(n, r1, r2, prime_factor):
    rng = np.random.default_rng(n)
    x = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    v = rng.standard_normal(n)
    at, to = indices(n, r1, r2, prime_factor)
    ins = np.array([[at(j, r) for r in range(r1)] for j in range(r2)])
    outs = np.array([[to(q, p) for p in range(r2)] for q in range(r1)])
    assert sorted(ins.ravel()) == sorted(outs.ravel()) == list(range(n))
    j, q = np.arange(r2)[:, None], np.arange(r1)[None, :]
    tw = np.ones((r2, r1)) if prime_factor else np.exp(-2j * np.pi * j * q / n)
    A = np.array([dft(x[i], +1) for i in ins]) * tw.conj()          # [j][q]
    y = np.array([dft(A[:, i], +1) for i in range(r1)])             # [q][p]
    flat = np.empty(n, dtype=complex)
    flat[outs] = y
    want = np.fft.ifft(x) * n
    assert np.abs(flat - want).max() < 1e-12 * np.abs(want).max()
    # product on the same registers, then the forward transform backwards through the steps
    B = np.array([dft(y[i] * v[outs[i]], -1) for i in range(r1)]).T * tw
    out = np.empty(n, dtype=complex)
    out[ins] = np.array([dft(B[i], -1) for i in range(r2)])
    want = np.fft.fft(want * v)
    assert np.abs(out - want).max() < 1e-12 * np.abs(want).max()


@pytest.mark.parametrize("n,a,b", LINES)
def test_line_plans(n, a, b):
    assert n == a * b and a <= b
    check(n, a, b, False)


@pytest.mark.parametrize("n,r1,r2", PLANES)
def test_side_plans(n, r1, r2):
    assert n == r1 * r2 and r1 >= r2
    check(n, r1, r2, np.gcd(r1, r2) == 1)


def test_every_side_is_a_line_too():
    assert sorted(SIDES) == sorted(n for n, _, _ in plans("FDE_SPLIT_SIDES"))


gpu = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    torch = pytest.importorskip("torch")
    from paper_1406_7803_gb300 import build, fde
    build.build()
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    return torch, fde


@gpu
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("mixed", 2e-6)])
@pytest.mark.parametrize("n", SIDES)
def test_every_side_transforms(lib, n, prec, tol):
    """A side as x, y and z length of small grids (the other axes have a remainder against the 16
    lines a CTA takes).  FP32: 3 axes of two butterflies, < 2e-6 of the largest output."""
    torch, fde = lib
    rng = np.random.default_rng(n)
    for shape in ((n, 30, 24), (24, n, 30), (30, 24, n)):
        ctx = fde.Context(np.diag([10.0, 11.0, 12.0]), shape, 1.0, 0, 0, prec=prec)
        f = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
        for sign, want in ((-1, np.fft.fftn(f) / f.size), (+1, np.fft.ifftn(f) * f.size)):
            d = torch.from_numpy(f).to("cuda", torch.complex128 if prec == "fp64" else torch.complex64)
            ctx.fft3d(d, sign)
            assert np.abs(d.cpu().numpy() - want).max() < tol * np.abs(want).max(), (shape, sign)
        d = torch.from_numpy(f).to("cuda")
        with pytest.raises(fde.FDEError) as e:  # 30 is not among the lengths it states
            ctx.fft3d_f64(d, -1, 1)
        assert e.value.status == fde.FDE_EUNSUPPORTED


@gpu
@pytest.mark.parametrize("n", [n for n in SIDES if n not in (24, 32, 60, 72, 96, 144)])
def test_mixed_potentials_on_general_sides(lib, n):
    """Potential build of two subsystems (one transform pair) and of three (a pair and a single) in
    double-float and FP32 against the all-FP64 build: 1e-5 of the largest value, the mixed path's bound."""
    torch, fde = lib
    for grid, subs in (((n, 24, 32), 2), ((24, n, 32), 3)):
        L = 0.25 * np.array(grid)
        x, y, z = np.meshgrid(*[2 * np.pi * np.arange(k) / k for k in grid], indexing="ij")
        out = {}
        for prec in ("fp64", "mixed"):
            ctx = fde.Context(np.diag(L), grid, 5.0, 1, 1, prec=prec)
            for i in range(subs):
                ctx.add_subsystem(np.array([[1.0 + i, 2.0, 3.0]]), np.ones(1), 0.5, 2, np.zeros((1, 3)), np.ones(1), 2.0,
                                  0.01)
                rho = 0.02 * (2.5 + np.cos(x + i) * np.cos(y) + 0.5 * np.sin(2 * z - i) + 0.3 * np.cos(x - y + z))
                ctx.set_density(i, np.ascontiguousarray(rho))
            v = torch.zeros((subs,) + grid, dtype=torch.float64, device="cuda")
            ctx.build_vemb(v)
            ctx.sync()
            out[prec] = v.cpu().numpy()
        assert np.abs(out["mixed"] - out["fp64"]).max() < 1e-5 * np.abs(out["fp64"]).max(), grid


@gpu
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-10), ("mixed", 1e-5)])
@pytest.mark.parametrize("grid", [(24, 24, 320), (30, 24, 45), (45, 75, 54), (160, 30, 24), (36, 160, 162), (72, 72, 250),
                                  (90, 54, 32), (50, 40, 300)])
def test_h_psi_and_density_on_general_grids(lib, grid, prec, tol):
    """Planes with equal and different sides, spheres that nearly fill the grid (spans of n - 1) and one
    band or a few: H psi against the plane-wave sum on the grid, and the density of the orbitals."""
    torch, fde = lib
    L = 0.25 * np.array(grid)
    h = 2 * np.pi / L
    ecut = 0.5 * min((n // 2 - 0.75) * b for n, b in zip(grid, h)) ** 2 * (0.96 if max(grid) < 100 else 0.2)
    kf = np.array([0.25, -0.25, 0.1])
    ctx = fde.Context(np.diag(L), grid, ecut, 0, 0, prec=prec)
    nb = 3
    ctx.add_subsystem(np.zeros((0, 3)), np.zeros(0), 0.5, nb, kf[None], np.ones(1), 2.0 * nb, 0.01)
    mil = ctx.basis(0, 0)
    rng = np.random.default_rng(grid[0])
    c = (rng.standard_normal((nb, len(mil))) + 1j * rng.standard_normal((nb, len(mil))))
    c /= np.linalg.norm(c, axis=1)[:, None]
    v = rng.uniform(-1, 1, grid)
    ctx.set_veff(0, torch.from_numpy(v).cuda())
    psi = torch.from_numpy(c).to("cuda", torch.complex128 if prec == "fp64" else torch.complex64)
    out = torch.zeros_like(psi)
    ctx.apply_h(0, 0, psi, out, nb)
    at = tuple((mil % np.array(grid)).T)
    kin = 0.5 * (((mil + kf) * h) ** 2).sum(1)
    u = np.zeros((nb,) + grid, dtype=complex)
    for b in range(nb):
        u[b][at] = c[b]
    u = np.fft.ifftn(u, axes=(1, 2, 3)) * v.size
    want = np.array([(np.fft.fftn(x * v) / v.size)[at] for x in u]) + kin * c
    got = out.cpu().numpy()
    assert (np.abs(got - want).max(1) < tol * np.abs(want).max(1)).all()
    # density of the block: no iteration (Ritz rotation only), every band occupied alike
    ctx.set_orbitals(0, 0, torch.from_numpy(c).cuda())
    ctx.subspace_solve(0, 0, 1e-30, 0)
    ctx.update_density(0)
    rho = torch.zeros(grid, dtype=torch.float64, device="cuda")
    ctx.get_density(0, rho)
    x = np.zeros_like(c)
    xt = torch.zeros((nb, len(mil)), dtype=torch.complex128, device="cuda")
    eig, occ = ctx.get_orbitals(0, 0, xt, nb)
    x = xt.cpu().numpy()
    u = np.zeros((nb,) + grid, dtype=complex)
    for b in range(nb):
        u[b][at] = x[b]
    u = np.abs(np.fft.ifftn(u, axes=(1, 2, 3)) * v.size) ** 2
    want = (2 * occ[:, None, None, None] / np.prod(L) * u).sum(0)
    assert np.abs(rho.cpu().numpy() - want).max() < tol * want.max()
