"""Block eigensolver when its search directions depend on each other (a Cholesky pivot fails): the failing
direction is replaced by the last one, its H- and S-images alike, and the solve goes on.

Seven plane waves and four bands: the four residuals make eight vectors in a space of seven, so one
direction depends on the others in every first iteration.  Its pivot is the rounding of the Gram matrix,
~1e-7 of the diagonal in FP32 and ~1e-16 in FP64, of either sign and far below the least accepted one (1e-5
and 1e-13)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_1406_7803_gb300 import fde  # noqa: E402

L, GRID, ECUT, NB = 6.0, (24, 24, 24), 0.6, 4
SIGMA, D, Q = (0.5, 1.0), ((0.5, 0.0), (0.0, -0.25)), ((0.25, 0.05), (0.05, 0.10))


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1406_7803_gb300 import build
    build.build()
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")


def columns(ctx, apply, n, dt):
    """The operator as a dense matrix, from its action on the unit vectors."""
    e = torch.eye(n, dtype=dt, device="cuda")
    out = torch.zeros_like(e)
    torch.cuda.synchronize()
    apply(0, 0, e, out, n)
    ctx.sync()
    return out.to(torch.complex128).cpu().numpy().T


# Errors: pivots above the least accepted one scale rounding by its inverse root: 1e-16 by 3e6 in FP64, the
# products' 1e-6 by 300 in FP32, a few times over in 40 iterations.
@pytest.mark.parametrize("uspp", [False, True])
@pytest.mark.parametrize("prec,tol,image", [("fp64", 1e-6, 1e-5), ("mixed", 3e-3, 3e-3)])
def test_dependent_directions_are_dropped(prec, tol, image, uspp):
    ctx = fde.Context(np.diag([L, L, L]), GRID, ECUT, 0, 0, prec=prec)
    aug = dict(proj_Q=Q, aug_sigma=0.7) if uspp else {}
    ctx.add_subsystem(np.array([[1.0, 2.0, 2.5]]), np.ones(1), 0.5, NB, np.zeros((1, 3)), np.ones(1), 2.0, 0.01, SIGMA,
                      D, **aug)
    npw = len(ctx.basis(0, 0))
    assert npw == 7 and npw < 2 * NB
    rng = np.random.default_rng(3)
    x, y, z = np.meshgrid(*[2 * np.pi * np.arange(n) / n for n in GRID], indexing="ij")
    v = sum(a * np.cos(p + b) for a, b, p in zip(rng.uniform(0.1, 0.4, 6), rng.uniform(0, 6, 6),
                                                 (x, y, z, x + y, y - z, x - z)))
    ctx.set_veff(0, torch.from_numpy(v).cuda())
    dt = torch.complex128 if prec == "fp64" else torch.complex64
    H = columns(ctx, ctx.apply_h, npw, dt)
    S = columns(ctx, ctx.apply_s, npw, dt)
    H, S = 0.5 * (H + H.conj().T), 0.5 * (S + S.conj().T)
    Li = np.linalg.inv(np.linalg.cholesky(S))
    want = np.linalg.eigvalsh(Li @ H @ Li.conj().T)[:NB]
    for seed in range(24):
        r = np.random.default_rng([seed, 1])
        c = r.standard_normal((npw, NB)) + 1j * r.standard_normal((npw, NB))
        m = np.linalg.cholesky(c.conj().T @ S @ c)
        c = np.ascontiguousarray((c @ np.linalg.inv(m).conj().T).T)  # S-orthonormal rows
        for iters in (1, 40):
            ctx.set_orbitals(0, 0, torch.from_numpy(c).cuda())
            status, it = ctx.subspace_solve(0, 0, tol, iters)
            X = torch.zeros((NB, npw), dtype=torch.complex128, device="cuda")
            HX = torch.zeros_like(X)
            torch.cuda.synchronize()
            eig, _ = ctx.get_orbitals(0, 0, X, NB)
            ctx.get_hpsi(0, 0, HX)
            X, HX = X.cpu().numpy(), HX.cpu().numpy()
            assert np.abs(X.conj() @ S @ X.T - np.eye(NB)).max() < image, (seed, iters)
            assert np.abs(HX - X @ H.T).max() < image * np.abs(HX).max(), (seed, iters)
            assert (eig > want - image).all(), (seed, iters)
        assert status == fde.FDE_OK, (seed, it)
        assert np.abs(eig - want).max() < image, (seed, eig - want)
