"""Performance cases of the embedded plane-wave library: what its users have it compute.

An SCF or freeze-and-thaw run spends its time in four calls, and every case is one of them:

* ``apply_h``   H_I psi of one block of orbitals (``Context.apply_h``);
* ``potential`` new subsystem densities in, every V_eff^I out (``set_density``, ``build_vemb``);
* ``hot_step``  one pass over a whole cell: new densities in, the potentials built, H psi of
  every band of every (subsystem, k) out (``set_density``, ``hot_step``, ``get_hpsi``);
* ``solve``     the block eigensolver on one (subsystem, k) and the density of its orbitals
  (``set_orbitals``, ``subspace_solve``, ``update_density``, ``get_density``).

``mixed`` contexts compute in single precision (their FP64 buffers carry single-precision
results, so those results are handed on as FP32 here, as a caller that keeps working on them
would); ``fp64`` contexts, and the refinement that ends every mixed SCF, in double.

Grids are the 2-3-5 sizes plane-wave codes choose, from 24 points a side to the largest planes
the library takes; bands from one to a slab's; cells with and without projectors; LDA with
Thomas-Fermi and PBE with either GGA kinetic functional.  Lattices have the grid spacing and
cutoff of the library's own cells: h = L / n, ecut = 20 Ha (0.222 / h)^2, unless a case says
otherwise.
"""
import math

import numpy as np
import torch

from paper_1406_7803_gb300 import fde

KB_SIGMA = (0.5, 1.0)              # two Gaussian projectors an atom
KB_D = ((0.5, 0.0), (0.0, -0.25))
RC = 0.5                           # width of the erf-regularised nuclei
RHO_CUT = 1e-10
SMEAR = 0.01                       # Fermi smearing of the slab (Ha)
CHUNK = 16                         # bands a batch of the 64-bit reference


# ---- the cases -----------------------------------------------------------------------------
def listed():
    slab = dict(n1=72, n2=72, n3=180, l1=16.0, l2=16.0, l3=40.0, ecut=20.0)
    small = dict(n1=24, n2=24, n3=60, l1=8.0, l2=8.0, l3=20.0, ecut=6.0)
    cube = dict(n1=32, n2=32, n3=32, l1=10.0, l2=10.0, l3=10.0, ecut=15.0)
    return [
        # the smallest call: two atoms' orbitals in a small box, local potential only
        dict(name="apply_h_box_fp64", op="apply_h", prec="fp64", bands=4, atoms=0, **cube),
        # a molecule's residual block late in a solve: a few unconverged bands, launches count
        dict(name="apply_h_few_bands_mixed", op="apply_h", prec="mixed", bands=3, atoms=4, **small),
        # the eigensolver's ordinary call: all bands of one k-point of a 36-atom slab
        dict(name="apply_h_slab_mixed", op="apply_h", prec="mixed", bands=64, atoms=36, **slab),
        # the same cell in the FP64 refinement, with the bands that are still unconverged
        dict(name="apply_h_slab_fp64", op="apply_h", prec="fp64", bands=17, atoms=36, **slab),
        # a cell of general shape: different sides, an odd number of bands
        dict(name="apply_h_general_mixed", op="apply_h", prec="mixed", bands=31, atoms=20,
             n1=60, n2=54, n3=135, l1=13.3, l2=12.0, l3=30.0, ecut=20.0),
        # the largest grid: one molecule of the 30 x 30 x 60 bohr cell, planes that fill an SM
        dict(name="apply_h_large_mixed", op="apply_h", prec="mixed", bands=32, atoms=8,
             n1=144, n2=144, n3=288, l1=30.0, l2=30.0, l3=60.0, ecut=25.0),
        # potentials after a density exchange, slab and molecule, in either precision
        dict(name="potential_slab_mixed", op="potential", prec="mixed", atoms=36, molecules=1, mol_atoms=6,
             gga=1, kedf=1, **slab),
        dict(name="potential_slab_fp64", op="potential", prec="fp64", atoms=36, molecules=1, mol_atoms=6,
             gga=1, kedf=1, **slab),
        # the whole hot path on the slab and molecule
        dict(name="hot_step_slab_mixed", op="hot_step", prec="mixed", bands=64, kpoints=2, atoms=36, molecules=1,
             mol_atoms=6, mol_bands=12, gga=1, kedf=1, **slab),
        # and on a cube with a slab and several molecules of uneven size
        dict(name="hot_step_fragments_mixed", op="hot_step", prec="mixed", bands=48, kpoints=1, atoms=27,
             molecules=4, mol_atoms=7, mol_bands=14, gga=1, kedf=1,
             n1=96, n2=96, n3=96, l1=24.0, l2=24.0, l3=24.0, ecut=20.0),
        # a molecule solved to the refinement's tolerance, FP64: many small steps
        dict(name="solve_small_fp64", op="solve", prec="fp64", bands=12, atoms=4, tol=1e-10, iters=200, **small),
        # the first iterations on the slab, where an SCF of the mixed path spends its time
        dict(name="solve_slab_mixed", op="solve", prec="mixed", bands=64, atoms=36, tol=1e-12, iters=4, **slab),
    ]


_SIDES = (24, 30, 32, 36, 40, 45, 48, 54, 60, 64, 72, 75, 80, 90, 96, 100, 108, 120, 128, 135, 144)
_DEPTHS = _SIDES + (150, 160, 162, 180, 192, 200, 216, 225, 240, 250, 256, 270, 288)


def draw(rng):
    """One more case: call, precision, grid and bands over the ranges the listed ones span."""
    op = rng.choice(("apply_h", "apply_h", "apply_h", "potential", "hot_step", "solve"))
    prec = rng.choice(("mixed", "mixed", "fp64"))
    while True:
        n1 = int(math.exp(rng.uniform(math.log(24), math.log(150))))
        n1 = min(_SIDES, key=lambda s: abs(s - n1))
        n2 = n1 if rng.random() < 0.5 else min(_SIDES, key=lambda s: abs(s - n1 * rng.uniform(0.7, 1.4)))
        n3 = min(_DEPTHS, key=lambda s: abs(s - n1 * rng.uniform(0.9, 2.6)))
        if prec == "fp64" and max(n1, n2) > 96:
            continue
        nr = n1 * n2 * n3
        if op != "apply_h" and nr > (1500000 if prec == "mixed" else 950000):
            continue
        if op == "solve" and nr > 400000:
            continue
        break
    h = rng.uniform(0.20, 0.30)
    case = dict(op=op, prec=prec, n1=n1, n2=n2, n3=n3, l1=round(n1 * h, 3), l2=round(n2 * h, 3),
                l3=round(n3 * h, 3), ecut=round(20.0 * (0.222 / h) ** 2, 3))
    npw = _npw(case)
    most = max(1.0, min(96.0, (4e6 if prec == "mixed" else 7e5) / npw))
    case["bands"] = max(1, int(math.exp(rng.uniform(0.0, math.log(most)))))
    case["atoms"] = rng.randint(0, max(1, min(36, int(1.5e6 / npw)))) if op == "apply_h" else rng.randint(2, max(3, min(30, int(1e6 / npw))))
    if op in ("potential", "hot_step"):
        case["molecules"] = rng.randint(0, 3)
        case["mol_atoms"] = rng.randint(1, 6)
        case["gga"] = int(rng.random() < 0.75)
        case["kedf"] = rng.choice((1, 2)) if case["gga"] else 0
    if op == "hot_step":
        case["kpoints"] = rng.randint(1, 2)
        case["mol_bands"] = rng.randint(1, 9) + 2 * case["mol_atoms"]
    if op == "solve":
        case["bands"] = max(2, case["bands"])
        case["tol"], case["iters"] = 1e-12, rng.randint(1, 4)
    return case


# ---- cells, inputs ---------------------------------------------------------------------------
def _npw(case):
    """Plane waves under the cutoff (the sphere's volume over that of a reciprocal point)."""
    return case["l1"] * case["l2"] * case["l3"] * (2 * case["ecut"]) ** 1.5 / (6 * math.pi ** 2)


def _grid(case):
    return (case["n1"], case["n2"], case["n3"])


def _lengths(case):
    return np.array([case["l1"], case["l2"], case["l3"]])


def _kpoints(case):
    """A q x 1 x 1 Monkhorst-Pack mesh; single blocks stand for a general point of one."""
    q = case.get("kpoints", 1)
    if case["op"] in ("apply_h", "solve") and case["prec"] == "mixed":
        return np.array([[0.25, -0.25, 0.0]]), np.ones(1)
    return np.array([[(2 * r - q - 1) / (2.0 * q), 0.0, 0.0] for r in range(1, q + 1)]), np.full(q, 1.0 / q)


def _place(rng, n, lengths, lo, hi, taken):
    """n positions at heights lo..hi of the cell, 1.4 bohr apart where there is room."""
    out = []
    for _ in range(n):
        for _ in range(200):
            p = rng.uniform(size=3) * lengths * np.array([1, 1, hi - lo]) + np.array([0, 0, lo * lengths[2]])
            d = np.array(taken + out) - p if taken or out else np.zeros((0, 3))
            d = d - lengths * np.round(d / lengths)
            if d.size == 0 or (d * d).sum(1).min() >= 1.4 ** 2:
                break
        out.append(p)
    return out


def _subsystems(case, seed):
    """[(positions, Z, bands, kpts, wk, nelec, smearing)]: a slab in the lower half, molecules above."""
    rng = np.random.default_rng([seed, 1])
    L = _lengths(case)
    whole = case["op"] in ("apply_h", "solve")
    pos = _place(rng, case["atoms"], L, 0.0, 1.0 if whole else 0.45, [])
    kp, wk = _kpoints(case)
    bands = case.get("bands", 1)
    nelec = 1.2 * bands if whole else 3.0 * len(pos)
    subs = [(np.array(pos).reshape(-1, 3), 3.0, bands, kp, wk, nelec, SMEAR)]
    taken = list(pos)
    for m in range(case.get("molecules", 0)):
        na = max(1, case["mol_atoms"] - m)
        p = _place(rng, na, L, 0.5, 0.75, taken)
        taken += p
        nb = max(2 * na, case.get("mol_bands", 2 * na) - m)
        subs.append((np.array(p), 4.0, nb, np.zeros((1, 3)), np.ones(1), 4.0 * na, 0.0))
    return subs


def _context(case, subs):
    gga = case.get("gga", 1)
    ctx = fde.Context(np.diag(_lengths(case)), _grid(case), case["ecut"], gga, case.get("kedf", 1), RHO_CUT,
                      case["prec"])
    for pos, z, nb, kp, wk, nelec, smear in subs:
        kb = len(pos) > 0
        ctx.add_subsystem(pos, np.full(len(pos), z), RC, nb, kp, wk, nelec, smear, KB_SIGMA if kb else (),
                          KB_D if kb else ())
    return ctx


def _density(case, pos, z, nelec):
    """Sharp atomic Gaussians with a tenth of the charge in slowly decaying tails, nelec electrons."""
    L, n = _lengths(case), _grid(case)
    rho = torch.zeros(n, dtype=torch.float64, device="cuda")
    for alpha, share in ((2.0, 0.9), (0.35, 0.1)):
        axes = []
        for c in range(3):
            x = np.arange(n[c]) / n[c] * L[c]
            d = x[None, None, :] - pos[:, c][:, None, None] - np.array([-1, 0, 1])[None, :, None] * L[c]
            axes.append(torch.from_numpy(np.exp(-alpha * d * d).sum(1)).cuda())
        xy = (axes[0][:, :, None] * axes[1][:, None, :]).reshape(len(pos), -1)
        rho += (z * share * (alpha / math.pi) ** 1.5 * (xy.T @ axes[2])).reshape(n)
    return rho * (nelec / (float(rho.sum()) * L.prod() / rho.numel()))


def _potential_well(case, seed):
    """A cell potential of atomic depth: wells on seeded centres over a gentle background."""
    rng = np.random.default_rng([seed, 2])
    L = _lengths(case)
    pos = rng.uniform(size=(max(4, case["atoms"]), 3)) * L
    rho = _density(case, pos, 1.0, 3.0 * len(pos))
    return 0.2 - 1.5 * rho ** (1.0 / 3.0)


def _sphere(case, kfrac):
    """Miller indices [npw, 3], sorted, and |k + G|^2 / 2, of the plane-wave sphere."""
    b = 2 * math.pi / _lengths(case)
    m = [np.arange(-(n // 2), n // 2 + 1) for n in _grid(case)]
    q = [(m[c] + kfrac[c]) * b[c] for c in range(3)]
    e = 0.5 * (q[0][:, None, None] ** 2 + q[1][None, :, None] ** 2 + q[2][None, None, :] ** 2)
    at = np.argwhere(e <= case["ecut"])
    return np.stack([m[c][at[:, c]] for c in range(3)], 1), e[tuple(at.T)]


def _orbitals(case, seed, tag, nb, miller, kfrac, dtype):
    """Normalised seeded orbitals with the decay of bound states in reciprocal space."""
    g = torch.Generator(device="cuda").manual_seed(1000003 * seed + tag)
    b = 2 * math.pi / _lengths(case)
    kin = torch.from_numpy(0.5 * (((miller + np.asarray(kfrac)) * b) ** 2).sum(1)).cuda()
    c = torch.randn((nb, len(miller), 2), dtype=torch.float64, device="cuda", generator=g)
    c = torch.view_as_complex(c) / (1.0 + kin)
    return (c / torch.linalg.norm(c, dim=1, keepdim=True)).to(dtype)


def _inputs(case, seed, miller_of):
    """What the calls take, the same for the library and for the 64-bit reference."""
    subs = _subsystems(case, seed)
    work = torch.complex64 if case["prec"] == "mixed" else torch.complex128
    s = {"subs": subs}
    if case["op"] in ("apply_h", "solve"):
        s["veff"] = _potential_well(case, seed)
    else:
        s["rho"] = [_density(case, p, z, ne) for p, z, _, _, _, ne, _ in subs]
    if case["op"] == "apply_h":
        s["psi"] = _orbitals(case, seed, 0, case["bands"], miller_of(0, 0), subs[0][3][0], work)
    elif case["op"] in ("solve", "hot_step"):
        # stored orbitals are given in FP64; a mixed context keeps them rounded to FP32
        s["blocks"] = [(i, k, _orbitals(case, seed, 64 * i + k, u[2], miller_of(i, k), u[3][k], work)
                        .to(torch.complex128)) for i, u in enumerate(subs) for k in range(len(u[3]))]
    return s


def prepare(case, seed):
    ctx = _context(case, _subsystems(case, seed))
    s = _inputs(case, seed, ctx.basis)
    s["ctx"], s["case"] = ctx, case
    if "veff" in s:
        ctx.set_veff(0, s["veff"])
    if case["op"] == "apply_h":
        s["hpsi"] = torch.zeros_like(s["psi"])
    elif case["op"] == "potential":
        s["out"] = torch.zeros((len(s["subs"]),) + _grid(case), dtype=torch.float64, device="cuda")
    elif case["op"] == "hot_step":
        for i, k, psi in s["blocks"]:
            ctx.set_orbitals(i, k, psi)
        s["hpsi"] = [torch.zeros_like(psi) for _, _, psi in s["blocks"]]
    else:
        s["out"] = torch.zeros(_grid(case), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    return s


def run(s):
    ctx, case = s["ctx"], s["case"]
    mixed = case["prec"] == "mixed"
    if case["op"] == "apply_h":
        ctx.apply_h(0, 0, s["psi"], s["hpsi"], case["bands"])
        return s["hpsi"]
    if case["op"] == "potential":
        for i, rho in enumerate(s["rho"]):
            ctx.set_density(i, rho)
        ctx.build_vemb(s["out"])
        return s["out"].float() if mixed else s["out"]
    if case["op"] == "hot_step":
        for i, rho in enumerate(s["rho"]):
            ctx.set_density(i, rho)
        ctx.hot_step()
        for (i, k, _), out in zip(s["blocks"], s["hpsi"]):
            ctx.get_hpsi(i, k, out)
        return [out.to(torch.complex64) if mixed else out for out in s["hpsi"]]
    for i, k, psi in s["blocks"]:
        ctx.set_orbitals(i, k, psi)
    ctx.subspace_solve(0, 0, case["tol"], case["iters"])
    ctx.update_density(0)
    ctx.get_density(0, s["out"])
    eig, _ = ctx.get_orbitals(0, 0, None, case["bands"])
    return {"eig": eig.astype(np.float32) if mixed else eig, "rho": s["out"].float() if mixed else s["out"]}


# ---- bytes and operations no implementation does without ------------------------------------
def _hpsi_work(case, bands, nproj, size):
    """Orbitals in, H psi out; lines of the sphere along z, its rows along y, every line along x, both
    ways; projections and their expansion."""
    n1, n2, n3 = _grid(case)
    npw = _npw(case)
    r = [math.sqrt(2 * case["ecut"]) * x / (2 * math.pi) for x in _lengths(case)]
    cols, rows = math.pi * r[0] * r[1], 2 * r[0] + 1
    line = [5.0 * n * math.log2(n) for n in (n1, n2, n3)]
    fft = 2 * (cols * line[2] + n3 * (rows * line[1] + n2 * line[0])) + 2.0 * n1 * n2 * n3
    return {"bytes": 2 * bands * npw * size, "flops": bands * (fft + 16.0 * nproj * npw)}


def _potential_work(case, nsub):
    nr = float(case["n1"] * case["n2"] * case["n3"])
    fields = 10 if case.get("gga", 1) else 2  # density, gradients, divergence and potential of a subsystem
    return {"bytes": 16.0 * nsub * nr, "flops": nsub * nr * (fields * 2.5 * math.log2(nr) + 200.0)}


def work(case):
    size = 8 if case["prec"] == "mixed" else 16
    nr = float(case["n1"] * case["n2"] * case["n3"])
    npw, nproj = _npw(case), 2 * case["atoms"]
    if case["op"] == "apply_h":
        w = _hpsi_work(case, case["bands"], nproj, size)
        return {"bytes": w["bytes"] + (nr * size / 2 + nproj * npw * size), "flops": w["flops"]}
    nmol = case.get("molecules", 0)
    if case["op"] == "potential":
        return _potential_work(case, 1 + nmol)
    if case["op"] == "hot_step":
        w = _potential_work(case, 1 + nmol)
        parts = [_hpsi_work(case, case["bands"] * case["kpoints"], nproj, size)]
        for m in range(nmol):
            na = max(1, case["mol_atoms"] - m)
            parts.append(_hpsi_work(case, max(2 * na, case["mol_bands"] - m), 2 * na, size))
        return {k: w[k] + sum(p[k] for p in parts) for k in ("bytes", "flops")}
    nb, w = case["bands"], _hpsi_work(case, case["bands"], nproj, size)
    # an iteration: H of the block, Gram and subspace matrices of three blocks, two rotations
    steps = min(case["iters"], 20) + 1
    return {"bytes": steps * w["bytes"], "flops": steps * (w["flops"] + 8.0 * npw * (9 * nb * nb + 6 * nb * nb))}


# ---- the same in 64 bits, from torch and numpy alone ------------------------------------------
def _gvectors(case):
    n, b = _grid(case), 2 * math.pi / _lengths(case)
    m = [np.fft.fftfreq(x, 1.0 / x) for x in n]
    g = torch.meshgrid(*[torch.from_numpy(m[c] * b[c]).cuda() for c in range(3)], indexing="ij")
    nyq = torch.zeros(n, dtype=torch.bool, device="cuda")
    for c in range(3):
        if n[c] % 2 == 0:
            nyq.index_fill_(c, torch.tensor([n[c] // 2], device="cuda"), True)
    return g, nyq


def _gga(rho, grad, energy):
    """(de/drho, de/dgrad) of an energy density of (rho, |grad rho|^2), zero below the density cut."""
    keep = rho >= RHO_CUT
    r = torch.where(keep, rho, torch.ones_like(rho)).requires_grad_()
    sig = torch.where(keep, grad[0] ** 2 + grad[1] ** 2 + grad[2] ** 2, torch.ones_like(rho)).requires_grad_()
    er, es = torch.autograd.grad(energy(r, sig).sum(), (r, sig), allow_unused=True)
    es = torch.zeros_like(er) if es is None else es
    zero = torch.zeros_like(rho)
    er, es = torch.where(keep, er, zero), torch.where(keep, es, zero)
    return er.detach(), [(2 * es * d).detach() for d in grad]


def _exc(case):
    def e(rho, sig):
        kf = (3 * math.pi ** 2 * rho) ** (1 / 3)
        ex = -0.75 * (3 / math.pi) ** (1 / 3) * rho ** (4 / 3)
        rs = (3 / (4 * math.pi * rho)) ** (1 / 3)
        den = 2 * 0.031091 * (7.5957 * rs ** 0.5 + 3.5876 * rs + 1.6382 * rs ** 1.5 + 0.49294 * rs * rs)
        ec = -2 * 0.031091 * (1 + 0.21370 * rs) * torch.log1p(1 / den)
        if not case.get("gga", 1):
            return ex + rho * ec
        beta, gamma = 0.06672455060314922, (1 - math.log(2.0)) / math.pi ** 2
        fx = 1 + 0.804 - 0.804 / (1 + 0.2195149727645171 * sig / (4 * kf * kf * rho * rho) / 0.804)
        t2 = sig * math.pi / (16 * kf * rho * rho)
        x = beta / gamma / torch.expm1(-ec / gamma) * t2
        p = torch.where(x > 1, (1 / x + 1) / x / (1 + 1 / x + 1 / (x * x)), (1 + x) / (1 + x + x * x))
        return ex * fx + rho * (ec + gamma * torch.log1p(beta / gamma * t2 * p))
    return e


def _ekin(case):
    kind = case.get("kedf", 1)

    def e(rho, sig):
        base = 0.3 * (3 * math.pi ** 2) ** (2 / 3) * rho ** (5 / 3)
        if kind == 0:
            return base
        s = torch.sqrt(sig + 1e-300) / (2 * (3 * math.pi ** 2) ** (1 / 3) * rho ** (4 / 3))
        if kind == 1:
            return base * (1 + 1.245 - 1.245 / (1 + 0.23889 * s * s / 1.245))
        a = 0.093907 * s * torch.asinh(76.32 * s)
        top = 1 + a + (0.26608 - 0.0809615 * torch.exp(-100 * s * s)) * s * s
        return base * top / (1 + a + 0.000057767 * s ** 4)
    return e


def _veff64(case, s):
    """v_loc + v_H[rho] + v_xc[rho] + v_kin[rho] - v_kin[rho_I] for every subsystem."""
    g, nyq = _gvectors(case)
    g2 = g[0] ** 2 + g[1] ** 2 + g[2] ** 2
    inv = torch.where((g2 > 0) & ~nyq, 1 / torch.where(g2 > 0, g2, torch.ones_like(g2)), torch.zeros_like(g2))
    omega = float(np.prod(_lengths(case)))
    real = lambda f: torch.fft.ifftn(f).real  # noqa: E731
    flt = lambda f: torch.where(nyq, torch.zeros_like(f), f)  # noqa: E731
    grad_of = lambda r: [real(flt(1j * g[c] * torch.fft.fftn(r))) for c in range(3)]  # noqa: E731
    div_of = lambda h: real(flt(1j * sum(g[c] * torch.fft.fftn(h[c]) for c in range(3))))  # noqa: E731
    rho = sum(s["rho"][1:], s["rho"][0])
    f = torch.zeros(_grid(case), dtype=torch.complex128, device="cuda")
    z0 = 0.0
    damp = -4 * math.pi * inv * torch.exp(-g2 * RC * RC / 4)
    for pos, z, *_ in s["subs"]:
        for p in pos:
            f += z * damp * torch.exp(-1j * (g[0] * p[0] + g[1] * p[1] + g[2] * p[2]))
            z0 += z * math.pi * RC * RC
    f[0, 0, 0] = z0
    common = real(f) * (rho.numel() / omega) + real(4 * math.pi * inv * torch.fft.fftn(rho))
    del f, damp, inv, g2
    gt = grad_of(rho)

    def functional(r, gr, e):
        er, h = _gga(r, gr, e)
        return er - div_of(h)
    common = common + functional(rho, gt, _exc(case)) + functional(rho, gt, _ekin(case))
    return [common - functional(r, grad_of(r), _ekin(case)) for r in s["rho"]]


def _projectors64(case, pos, miller, kfrac):
    b, omega = 2 * math.pi / _lengths(case), float(np.prod(_lengths(case)))
    q = torch.from_numpy((miller + np.asarray(kfrac)) * b).cuda()
    q2, rows = (q * q).sum(1), []
    for p in pos:
        phase = torch.exp(-1j * (q @ torch.from_numpy(np.asarray(p)).cuda()))
        for sg in KB_SIGMA:
            amp = omega ** -0.5 * (math.pi ** 1.5 * sg ** 3) ** -0.5 * (2 * math.pi * sg * sg) ** 1.5
            rows.append(amp * torch.exp(-q2 * sg * sg / 2) * phase)
    return torch.stack(rows)


def _hpsi64(case, sub, k, psi, veff):
    """H psi of a block: kinetic, local potential on the grid, Gaussian projectors."""
    pos, kfrac = sub[0], sub[3][k]
    miller, kin = _sphere(case, kfrac)
    n = _grid(case)
    at = [torch.from_numpy(miller[:, c] % n[c]).cuda() for c in range(3)]
    flat = (at[0] * n[1] + at[1]) * n[2] + at[2]
    kin = torch.from_numpy(kin).cuda()
    out = torch.empty(psi.shape, dtype=torch.complex128, device="cuda")
    for b0 in range(0, len(psi), CHUNK):
        c = psi[b0:b0 + CHUNK].to(torch.complex128)
        box = torch.zeros((len(c),) + n, dtype=torch.complex128, device="cuda")
        box.view(len(c), -1)[:, flat] = c
        box = torch.fft.fftn(torch.fft.ifftn(box, dim=(1, 2, 3)) * veff, dim=(1, 2, 3))
        out[b0:b0 + CHUNK] = box.view(len(c), -1)[:, flat] + kin * c
    if len(pos):
        beta = _projectors64(case, pos, miller, kfrac)
        c = psi.to(torch.complex128)
        p = (beta.conj() @ c.T).view(len(pos), 2, -1)
        d = torch.tensor(KB_D, dtype=torch.complex128, device="cuda")
        out += torch.einsum("ij,ajb->aib", d, p).reshape(beta.shape[0], -1).T @ beta
    return out


def exact(case, seed):
    s = _inputs(case, seed, lambda i, k: _sphere(case, _subsystems(case, seed)[i][3][k])[0])
    if case["op"] == "apply_h":
        return _hpsi64(case, s["subs"][0], 0, s["psi"], s["veff"])
    if case["op"] == "potential":
        return torch.stack(_veff64(case, s))
    if case["op"] == "hot_step":
        v = _veff64(case, s)
        return [_hpsi64(case, s["subs"][i], k, psi, v[i]) for i, k, psi in s["blocks"]]
    if case["iters"] < 100:
        return None  # a fixed number of iterations: the iterate has no value outside the solver
    sub = s["subs"][0]
    miller, _ = _sphere(case, sub[3][0])
    h = _hpsi64(case, sub, 0, torch.eye(len(miller), dtype=torch.complex128, device="cuda"), s["veff"]).T
    w, v = torch.linalg.eigh(0.5 * (h + h.conj().T))
    eig, nelec = w[:case["bands"]].cpu().numpy(), sub[5]
    lo, hi = eig[0] - 1.0, eig[-1] + 1.0
    for _ in range(200):
        mu = 0.5 * (lo + hi)
        occ = 1 / (1 + np.exp((eig - mu) / SMEAR))
        lo, hi = (mu, hi) if 2 * occ.sum() < nelec else (lo, mu)
    n = _grid(case)
    box = torch.zeros((len(eig),) + n, dtype=torch.complex128, device="cuda")
    flat = [torch.from_numpy(miller[:, c] % n[c]).cuda() for c in range(3)]
    box.view(len(eig), -1)[:, (flat[0] * n[1] + flat[1]) * n[2] + flat[2]] = v[:, :len(eig)].T
    u2 = torch.fft.ifftn(box, dim=(1, 2, 3)).abs() ** 2 * float(np.prod(n)) ** 2
    occ = torch.from_numpy(2 * occ / float(np.prod(_lengths(case)))).cuda()
    return {"eig": eig, "rho": (occ[:, None, None, None] * u2).sum(0)}
