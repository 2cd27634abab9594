"""Transforms on every kind of length: those without a two-step plan (the runtime-length kernels of grid.cu
and hpsi.cu, the FP64 transforms of a mixed potential build), planes of different sides whose sphere does
not fit the two-step plane pass, and the long z lines of every two-step length, in FP32, FP64 and
double-float."""
import numpy as np
import pytest

import test_two_step_plans as plans

from test_two_step_plans import lib  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

PLANLESS = [(20, 27, 25), (24, 25, 30), (18, 24, 40), (27, 30, 81), (30, 24, 243), (125, 24, 20), (2, 3, 5)]


def transforms(lib, shape):
    """FP64 to 1e-12 (potential build's form 1e-13), FP32 to 2e-6 of the largest output: the bounds of the
    compiled lengths."""
    torch, fde = lib
    rng = np.random.default_rng(sum(shape))
    f = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
    for prec, tol in (("fp64", 1e-12), ("mixed", 2e-6)):
        ctx = fde.Context(np.diag([10.0, 11.0, 12.0]), shape, 0.05, 0, 0, prec=prec)
        for sign, want in ((-1, np.fft.fftn(f) / f.size), (+1, np.fft.ifftn(f) * f.size)):
            d = torch.from_numpy(f).to("cuda", torch.complex128 if prec == "fp64" else torch.complex64)
            torch.cuda.synchronize()
            ctx.fft3d(d, sign)
            ctx.sync()
            assert np.abs(d.cpu().numpy() - want).max() < tol * np.abs(want).max(), (prec, sign)
            d = torch.from_numpy(f).cuda()
            torch.cuda.synchronize()
            ctx.fft3d_f64(d, sign, 0)
            ctx.sync()
            assert np.abs(d.cpu().numpy() - want).max() < 1e-13 * np.abs(want).max(), (prec, sign)
            with pytest.raises(fde.FDEError):  # a length that form does not state
                ctx.fft3d_f64(d, sign, 1)


@pytest.mark.parametrize("shape", PLANLESS)
def test_transforms_without_a_plan(lib, shape):  # noqa: F811
    transforms(lib, shape)


# 45 x 45 lines: a remainder against the 16 or 8 lines a CTA takes
@pytest.mark.parametrize("n", [n for n, _, _ in plans.LINES])
def test_z_lines_of_every_plan(lib, n):  # noqa: F811
    transforms(lib, (45, 45, n))


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-10), ("mixed", 1e-5)])
@pytest.mark.parametrize("grid", [g for g in PLANLESS if min(g) > 5] + [(72, 72, 81), (96, 90, 24), (90, 96, 30)])
def test_h_psi_and_density_without_a_plan(lib, grid, prec, tol):  # noqa: F811
    plans.test_h_psi_and_density_on_general_grids(lib, grid, prec, tol)


@pytest.mark.parametrize("n", [18, 20, 25, 27, 81, 125])
def test_mixed_potentials_without_a_plan(lib, n):  # noqa: F811
    plans.test_mixed_potentials_on_general_sides(lib, n)


@pytest.mark.parametrize("n", [n for n, _, _ in plans.LINES])
def test_double_float_lines_in_the_hartree_energy(lib, n):  # noqa: F811
    """A mixed context's Hartree energies come from double-float transforms of the densities and FP64 sums:
    transforms good to 2e-13 of their largest output leave 1e-11 of the energy, FP32 ones 1e-7.  V_eff to
    1e-5 of its largest value (gradients and the functionals in FP32)."""
    torch, fde = lib
    for grid in ((30, 24, n), (n, 24, 30), (24, n, 45)) if n <= 160 else ((30, 24, n),):
        L = 0.25 * np.array(grid)
        x, y, z = np.meshgrid(*[2 * np.pi * np.arange(k) / k for k in grid], indexing="ij")
        out = {}
        for prec in ("fp64", "mixed"):
            ctx = fde.Context(np.diag(L), grid, 5.0, 1, 1, prec=prec)
            for i in range(2):
                ctx.add_subsystem(np.array([[1.0 + i, 2.0, 3.0]]), np.ones(1), 0.5, 2, np.zeros((1, 3)), np.ones(1), 2.0,
                                  0.01)
                rho = 0.02 * (3.0 + np.cos(x + i) * np.cos(y) + np.sin(2 * z - i) * np.cos(3 * x) + 0.3 * np.cos(5 * z + y))
                ctx.set_density(i, np.ascontiguousarray(rho))
            v = torch.zeros((2,) + grid, dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()
            e = ctx.build_vemb(v, energies=True)
            ctx.sync()
            out[prec] = (e["E_H"], e["E_H_nad"], v.cpu().numpy())
        for k in range(2):
            assert abs(out["mixed"][k] - out["fp64"][k]) < 1e-11 * abs(out["fp64"][0]), (grid, k)
        assert np.abs(out["mixed"][2] - out["fp64"][2]).max() < 1e-5 * np.abs(out["fp64"][2]).max(), grid
