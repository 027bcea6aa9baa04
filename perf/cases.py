"""The work that the library is timed on: whole calls through its public entry points.

A case names the microstructures (grid, filter rule, phase contrast), the load cases, the precision
and scheme, and whether the call starts at the geometry ("build": filter build, solve, effective
stiffness) or at a filtered material in hand (a parameter study over loads or reference media).

FP32 solves run a fixed number of Green-operator applications (`iters`, tol = 0), in the range that
tolerances of 1e-3 to 1e-6 take at these contrasts: run to a tolerance near the FP32 rounding floor,
a load case may stop one iterate sooner or later by rounding alone, and two fields of different
iterates say nothing about each other's accuracy.  The FP64 study runs to its tolerance.  Mean
stresses and stiffnesses of FP32 solves are kept in FP32, the accuracy they have.
"""
import math

import numpy as np
import torch

import hom_inputs as H
import paper_1412_3228_gb300 as hom

RULES = {"none": H.RULE_NONE, "voigt": H.RULE_VOIGT, "reuss": H.RULE_REUSS, "2-layers": H.RULE_TWO_LAYER}
SWEEP_SIZES = (45, 135, 405, 1215)
ENSEMBLE_SIZES = (45, 75, 135, 225, 405)
STUDY_SIZES = (9, 15, 21, 25, 27, 35, 45, 63, 75, 81, 105, 125)


def listed():
    return [
        # an interactive call, or one member of an optimisation loop: the smallest work, where latency counts
        dict(name="disk2d_45", kind="disk", n=45, count=1, loads=3, rule="2-layers", contrast=10.0, iters=40, fp=32,
             scheme="basic", graph=False, build=False),
        # a ragged grid, 11 x 13 voxels per side, of the sizes without a dedicated radix plan
        dict(name="disk2d_143", kind="disk", n=143, count=2, loads=3, rule="voigt", contrast=10.0, iters=40, fp=32,
             scheme="basic", graph=False, build=False),
        # a power-of-two image, the grid most users of FFT solvers bring
        dict(name="disk2d_512", kind="disk", n=512, count=2, loads=3, rule="reuss", contrast=0.1, iters=40, fp=32,
             scheme="basic", graph=False, build=True),
        # the resolution sweep of the benchmark: 32 cells of four grids in one batch, from the geometry to C_eff
        dict(name="sweep2d", kind="sweep", n=1215, count=32, loads=3, rule="all", contrast=10.0, iters=30, fp=32,
             scheme="basic", graph=False, build=True),
        # random-disk ensemble with log-uniform contrasts, uneven grids, accelerated scheme, one graph launch
        dict(name="ensemble2d_em", kind="ensemble", n=405, count=64, loads=3, rule="mixed", contrast=100.0, iters=18,
             fp=32, scheme="em", graph=True, build=False),
        # the paper's convergence study: 60 small grids and a reference grid, one load, double precision, e < 1e-4
        dict(name="study2d_fp64", kind="study", n=405, count=61, loads=1, rule="study", contrast=10.0, iters=0, fp=64,
             scheme="basic", graph=False, build=True),
        # high contrast in double precision by conjugate gradients
        dict(name="cg2d_405_fp64", kind="cg", n=405, count=2, loads=3, rule="2-layers", contrast=1000.0, iters=40, fp=64,
             scheme="cg", graph=False, build=False),
        # a small volume in double precision, six loads
        dict(name="spheres3d_63_fp64", kind="spheres", n=63, count=1, loads=6, rule="2-layers", contrast=10.0, iters=20,
             fp=64, scheme="basic", graph=False, build=False),
        # a power-of-two volume (a cropped tomogram), six loads
        dict(name="spheres3d_64", kind="spheres", n=64, count=1, loads=6, rule="voigt", contrast=0.1, iters=30, fp=32,
             scheme="basic", graph=False, build=False),
        # the random-sphere cell of the benchmark, from the geometry to C_eff
        dict(name="spheres3d_135", kind="spheres", n=135, count=1, loads=6, rule="2-layers", contrast=10.0, iters=30,
             fp=32, scheme="basic", graph=False, build=True),
        # the largest volume of the benchmark
        dict(name="spheres3d_243", kind="spheres", n=243, count=1, loads=6, rule="2-layers", contrast=10.0, iters=12,
             fp=32, scheme="basic", graph=False, build=False),
        # one step of an inverse problem: C_eff and von Mises loss, forward solve and adjoint gradient
        dict(name="gradient3d_81", kind="gradient", n=81, count=1, loads=6, rule="2-layers", contrast=20.0, iters=30,
             fp=32, scheme="basic", graph=False, build=True),
    ]


# ------------------------------------------------------------------ drawn cases
def _supported(n):
    for p in (2, 3, 5, 7, 11, 13):
        while n % p == 0:
            n //= p
    return n == 1


def _grid(rng, lo, hi, own):
    """A grid size: half the time one of the repository's own, else log-uniform over the supported ones."""
    own = [n for n in own if lo <= n <= hi]
    if own and rng.random() < 0.5:
        return rng.choice(own)
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    while not _supported(n):
        n -= 1
    return max(lo, n)


def _cost(c):
    """Voxel iterations of a case, double precision weighed by its arithmetic rate."""
    dim = 3 if c["kind"] in ("spheres", "gradient") else 2
    nvox = float(c["n"]) ** dim * c["count"]
    if c["kind"] == "sweep":
        nvox = 8.0 * sum(n * n for n in SWEEP_SIZES)
    if c["kind"] == "ensemble":
        nvox *= 0.25
    if c["kind"] == "study":
        nvox = float(c["n"]) ** 2 + 5.0 * sum(n * n for n in STUDY_SIZES)
    per = {2: 1.0, 3: 3.0}[dim] * (12.0 if c["fp"] == 64 else 1.0) * (2.0 if c["kind"] == "gradient" else 1.0)
    return nvox * c["loads"] * (c["iters"] or 60) * per


def draw(rng):
    while True:
        kind = rng.choice(["disk", "disk", "disk", "spheres", "spheres", "ensemble", "study", "cg", "gradient"])
        c = dict(kind=kind, n=0, count=1, loads=3, rule=rng.choice(["none", "voigt", "reuss", "2-layers"]),
                 contrast=float("%.3g" % math.exp(rng.choice([-1.0, 1.0]) * rng.uniform(math.log(3.0), math.log(30.0)))),
                 iters=rng.randint(10, 45), fp=32, scheme="basic", graph=rng.random() < 0.3, build=rng.random() < 0.5)
        if kind == "disk":
            c["n"] = _grid(rng, 15, 1215, (45, 75, 135, 225, 405, 1215))
            c["count"], c["loads"] = rng.choice([1, 1, 2, 4, 8, 16]), rng.choice([1, 3, 3])
            c["fp"], c["scheme"] = rng.choice([32, 32, 32, 64]), rng.choice(["basic", "basic", "em"])
            if c["scheme"] == "em" and c["n"] % 2 == 0:
                c["scheme"] = "basic"
        elif kind == "spheres":
            c["n"] = _grid(rng, 15, 162, (27, 45, 81, 135))
            c["loads"] = rng.choice([1, 6, 6])
            c["fp"], c["scheme"] = rng.choice([32, 32, 32, 64]), rng.choice(["basic", "basic", "em"])
            if c["scheme"] == "em" and c["n"] % 2 == 0:
                c["scheme"] = "basic"
        elif kind == "ensemble":
            c.update(n=405, count=rng.randint(8, 128), rule="mixed", contrast=100.0, scheme=rng.choice(["em", "basic"]))
        elif kind == "study":
            c.update(n=rng.choice([135, 225, 315, 405]), count=61, loads=1, rule="study", iters=0, fp=64, graph=False,
                     build=True, contrast=float("%.3g" % math.exp(rng.uniform(math.log(2.0), math.log(20.0)))))
        elif kind == "cg":
            c.update(n=_grid(rng, 27, 405, (45, 75, 135, 225, 405)), count=rng.choice([1, 2, 4]), fp=64, scheme="cg",
                     graph=False, build=False, contrast=rng.choice([100.0, 1000.0]))
            c["iters"] = min(c["iters"], 40)
        else:
            c.update(n=_grid(rng, 15, 81, (27, 45, 81)), loads=6, rule="2-layers", build=True, graph=False)
        if _cost(c) <= 0.25 * _cost(listed()[10]):
            return c


# ------------------------------------------------------------------ inputs
def _disk(n, rng, rule, radius_px=1.0, vf=None):
    """The centred disk of the paper, at a random place of its periodic cell."""
    r = math.sqrt((vf if vf is not None else rng.uniform(0.15, 0.25)) / math.pi)
    centre = (float(rng.uniform(0.3, 0.7)), float(rng.uniform(0.3, 0.7)), 0.0)
    return H.Cell(2, n, 0, [H.Primitive(H.PRIM_DISK, 1, centre, r)], rule, radius_px, 16)


def _geometry(case, seed):
    """Cells, phase table, load cases and reference media of a case."""
    rng = np.random.default_rng(seed)
    kind, n = case["kind"], case["n"]
    cells, phases = [], []

    def add(cell, pair):
        cells.append(H.remap_phases(cell, len(phases)))
        phases.extend(pair)

    if kind in ("disk", "cg"):
        for _ in range(case["count"]):
            add(_disk(n, rng, RULES[case["rule"]]), H.two_phases(case["contrast"]))
    elif kind == "sweep":
        vf = float(rng.uniform(0.18, 0.22))
        for k, contrast in enumerate((case["contrast"], 1.0 / case["contrast"])):
            phases.extend(H.two_phases(contrast))
        for m in SWEEP_SIZES:
            for k in range(2):
                for rule in RULES.values():
                    cells.append(H.remap_phases(_disk(m, rng, rule, vf=vf), 2 * k))
    elif kind == "study":
        vf = float(rng.uniform(0.18, 0.22))
        phases = H.two_phases(case["contrast"])
        for rule, radii in (("none", (1.0,)), ("voigt", (0.55, 1.0)), ("2-layers", (0.55, 1.0))):
            for r in radii:
                cells += [H.centred_disk_cell(m, vf=vf, rule=RULES[rule], radius_px=r) for m in STUDY_SIZES]
        cells.append(H.centred_disk_cell(n, vf=vf, rule=H.RULE_NONE))
    elif kind == "ensemble":
        for i in range(case["count"]):
            cell, pair = H.random_disk_cell(int(rng.integers(1 << 30)), sizes=(ENSEMBLE_SIZES[i % 5],))
            add(cell, pair)
    else:  # spheres, gradient
        cell = None
        while cell is None:
            try:
                cell = H.rsa_spheres_cell(n, int(rng.integers(1 << 30)), vf=float(rng.uniform(0.2, 0.28)),
                                          rule=RULES[case["rule"]], gap_voxels=n / 243)
            except RuntimeError:
                pass
        add(cell, H.two_phases(case["contrast"]))
    dim = cells[0].dim
    E = np.eye(H.ncomp(dim))[:case["loads"]]
    media = []
    for c in cells:
        pair = [phases[c.matrix_phase], phases[c.prims[0].phase]]
        media.append(H.geometric_lame(pair, dim) if case["scheme"] == "em" else H.mean_lame(pair))
    return cells, phases, E, np.array(media)


def prepare(case, seed):
    cells, phases, E, media = _geometry(case, seed)
    st = dict(case=case, cells=cells, phases=phases, E=E, media=media, dim=cells[0].dim)
    prec = hom.HOM_FP32 if case["fp"] == 32 else hom.HOM_FP64
    opts = dict(precision=prec, tol=0.0, max_iter=case["iters"])
    if case["kind"] != "gradient" and case["scheme"] != "cg":
        opts.update(use_graph=case["graph"],
                    scheme=hom.HOM_SCHEME_EYRE_MILTON if case["scheme"] == "em" else hom.HOM_SCHEME_BASIC)
    if case["scheme"] != "cg":
        opts["criterion"] = hom.HOM_CRIT_EN if case["fp"] == 32 else hom.HOM_CRIT_E
    if case["kind"] == "study":
        opts.update(tol=1e-4, max_iter=100000, fields=False)
    st["opts"] = opts
    if case["kind"] == "gradient":
        w = np.random.default_rng([seed, 1]).standard_normal((1, 6, 6))
        st["weights"] = torch.from_numpy(w)
        st["lame"] = torch.tensor(phases, dtype=torch.float64, requires_grad=True)
    elif not case["build"]:
        st["material"] = hom.hom_filter_build(cells, phases)
    return st


# ------------------------------------------------------------------ one pass
def run(st):
    case = st["case"]
    single = np.float32 if case["fp"] == 32 else np.float64
    if case["kind"] == "gradient":
        # weights : C_eff + mean von Mises square over the loads, differentiated through the solve
        lame = st["lame"]
        C, sigma = hom.HomSolve.apply(lame, st["cells"], st["media"], st["opts"])
        s = sigma.view(6, 6, -1)
        dev = torch.cat([s[:, :3] - s[:, :3].mean(1, keepdim=True), s[:, 3:]], 1)
        vm = 1.5 * dev.square().sum(1).mean()
        g, = torch.autograd.grad([C, vm], lame, [st["weights"], torch.ones_like(vm)])
        return {"C": C.detach().float(), "sigma": sigma.detach(), "vm": vm.detach(), "grad": g.float()}
    mat = hom.hom_filter_build(st["cells"], st["phases"]) if case["build"] else st["material"]
    if case["scheme"] == "cg":
        r = hom.hom_solve_cg(mat, st["E"], **st["opts"])
    else:
        r = hom.hom_solve(mat, st["E"], st["media"], **st["opts"])
    out = {"mean_sigma": r["mean_sigma"].astype(single), "iterations": r["iterations"]}
    if r["eps"] is not None:
        out["eps"], out["sigma"] = r["eps"], r["sigma"]
    if len(st["E"]) == H.ncomp(st["dim"]):
        out["C"] = hom.hom_effective_stiffness(st["E"], r["mean_sigma"], st["dim"]).astype(single)
    return out


def work(case):
    """Bytes: labels in, fields out, and, where the batch's state does not fit the chip's 129 MB L2, that state
    (the nc half spectra of every load) read and written for each of an iteration's two sweeps (along the rows
    of x and across them).  Operations: two real transforms of nc components per load and iteration
    (2.5 N log2 N each), the constitutive update (4 nc) and the Green operator (about 60 nc / 3 per bin of the half spectrum)."""
    dim = 3 if case["kind"] in ("spheres", "gradient") else 2
    nc = 3 if dim == 2 else 6
    if case["kind"] == "sweep":
        grids = [m for m in SWEEP_SIZES for _ in range(8)]
    elif case["kind"] == "study":
        grids = [m for m in STUDY_SIZES for _ in range(5)] + [case["n"]]
    elif case["kind"] == "ensemble":
        grids = [ENSEMBLE_SIZES[i % 5] for i in range(case["count"])]
    else:
        grids = [case["n"]] * case["count"]
    size, L, iters = case["fp"] // 8, case["loads"], case["iters"] or 45
    nvox = float(sum(m ** dim for m in grids))
    solves = 2 if case["kind"] == "gradient" else 1
    state = nvox * L * nc * size  # half spectra: n/2 complex values for n reals
    fields = 0.0 if case["kind"] == "study" else 2.0 * state
    per_iter = 4.0 * state if 2.0 * state > 129e6 else 0.0
    flops = sum(m ** dim * (2 * nc * 2.5 * dim * math.log2(m) + 4.0 * nc + 10.0 * nc) for m in grids) * L
    return {"bytes": nvox * 4 + fields * solves + per_iter * iters * solves, "flops": flops * iters * solves}


# ------------------------------------------------------------------ the same in 64 bits, by torch alone
def _cuda64(x):
    return torch.as_tensor(x, dtype=torch.float64, device="cuda")


def _filtered(cell, phases):
    """Filtered stiffness of one cell with one kind of inclusion, from section 2 of the paper: sample counts of the ball
    on the refined grid, then the rule.  Returns (label [nv]: 0 matrix, 1 inclusion, 2 mixed; index and inclusion
    fraction f and normal of the mixed voxels)."""
    n, dim, S = cell.n, cell.dim, cell.subgrid
    nv = n ** dim
    cen = _cuda64([p.centre[:dim] for p in cell.prims])
    rad = _cuda64([p.radius for p in cell.prims])
    reach = cell.radius_px / n if cell.rule != H.RULE_NONE else 0.0
    kmax = min(4, len(cell.prims))
    label = torch.zeros(nv, dtype=torch.int64, device="cuda")
    parts = []
    if cell.rule != H.RULE_NONE:
        t = torch.arange(-int(2 * S * cell.radius_px) - S, int(2 * S * cell.radius_px) + 2 * S, device="cuda")
        D = 2 * t + 1 - S
        ball = torch.cartesian_prod(*([D] * dim))
        ball = ball[(ball * ball).sum(1) <= (2.0 * S * cell.radius_px) ** 2].double() / (2.0 * S * n)
    for v0 in range(0, nv, 1 << 18):
        v = torch.arange(v0, min(nv, v0 + (1 << 18)), device="cuda")
        x = torch.stack([v // n ** d % n for d in range(dim)], 1).double().add_(0.5).div_(n)
        d = x[:, None, :] - cen[None]
        d -= d.round()
        gap = d.square().sum(2).sqrt() - rad  # signed distance to every surface
        inside = (gap <= 0).any(1)
        label[v] = inside.long()
        if cell.rule == H.RULE_NONE:
            continue
        near = (gap.abs().min(1).values <= reach * 1.001).nonzero()[:, 0]
        for c0 in range(0, len(near), 4096):
            q = near[c0:c0 + 4096]
            dist, which = gap[q].abs().topk(kmax, 1, largest=False)
            dd = d[q].gather(1, which[:, :, None].expand(-1, -1, dim))
            far = ((gap[q] < -reach * 1.001)).any(1)
            hit = far[:, None].expand(-1, len(ball)).clone()
            for k in range(kmax):
                hit |= (dd[:, k, None, :] + ball[None]).square().sum(2) <= (rad[which[:, k]] ** 2)[:, None]
            f = hit.double().mean(1)
            normal = dd[:, 0] / dd[:, 0].norm(dim=1, keepdim=True)
            label[v[q]] = torch.where(f == 0, 0, torch.where(f == 1, 1, 2))
            m = (f > 0) & (f < 1)
            parts.append((v[q][m], f[m], normal[m]))
    if not parts:
        e = torch.zeros(0, dtype=torch.float64, device="cuda")
        return label, e.long(), e, e.view(0, dim)
    return (label,) + tuple(torch.cat(z) for z in zip(*parts))


def _iso(lame, dim):
    """Mandel stiffness of an isotropic phase (lambda, mu)."""
    nc = H.ncomp(dim)
    one = torch.zeros(nc, dtype=torch.float64, device="cuda")
    one[:dim] = 1.0
    return lame[0] * one[:, None] * one[None] + 2.0 * lame[1] * torch.eye(nc, dtype=torch.float64, device="cuda")


def _rule(cell, f, normal, Cm, Ci):
    """Stiffness [M, nc, nc] of the mixed voxels: eqs. 3, 4 and 5 (eq. 5 as the closed form of a rank-1 laminate)."""
    f = f[:, None, None]
    if cell.rule == H.RULE_VOIGT:
        return (1 - f) * Cm + f * Ci
    if cell.rule == H.RULE_REUSS:
        return torch.linalg.inv((1 - f) * torch.linalg.inv(Cm) + f * torch.linalg.inv(Ci))
    dim = cell.dim
    r = math.sqrt(0.5)
    N = torch.zeros(len(normal), H.ncomp(dim), dim, dtype=torch.float64, device="cuda")  # a -> sym(a (x) n)
    for i in range(dim):
        N[:, i, i] = normal[:, i]
    for I, (i, j) in enumerate([(0, 1)] if dim == 2 else [(1, 2), (0, 2), (0, 1)]):
        N[:, dim + I, i] = r * normal[:, j]
        N[:, dim + I, j] = r * normal[:, i]
    Nt = N.transpose(1, 2)
    K = Nt @ (f * Cm + (1 - f) * Ci) @ N
    G = N @ torch.linalg.solve(K, Nt)
    dC = Ci - Cm
    return (1 - f) * Cm + f * Ci - f * (1 - f) * (dC @ G @ dC)


class _Problem:
    """One cell's discrete problem on plain torch tensors [nc, nv]."""

    def __init__(self, cell, phases, c0):
        self.cell, self.dim, self.n = cell, cell.dim, cell.n
        self.nc, self.nv = H.ncomp(cell.dim), cell.n ** cell.dim
        self.label, self.at, self.f, self.normal = _filtered(cell, phases)
        inc = cell.prims[0].phase
        self.pair = _cuda64([phases[cell.matrix_phase], phases[inc]])
        lame = self.pair[self.label.clamp(max=1)]
        self.lam, self.mu2 = lame[:, 0].contiguous(), 2.0 * lame[:, 1]
        self.Cx = self.mixed(self.pair)
        self.lam0, self.mu0 = float(c0[0]), float(c0[1])
        n, dim = self.n, self.dim
        a = torch.arange(n, device="cuda")
        a = torch.where(a <= n // 2, a, a - n).double()
        ax = [a[: n // 2 + 1]] + [a] * (dim - 1)  # x last in memory, half spectrum
        self.xi = [2 * math.pi * ax[d].view([-1 if k == dim - 1 - d else 1 for k in range(dim)]) for d in range(dim)]
        self.q2 = sum(x * x for x in self.xi)
        self.live = self.q2 > 0
        self.weight = torch.full((n // 2 + 1,), 2.0, dtype=torch.float64, device="cuda")
        self.weight[0] = 1.0
        if n % 2 == 0:  # wave vectors with a Nyquist component take zero strain
            for x in self.xi:
                self.live = self.live & (x != math.pi * n)
            self.weight[-1] = 1.0
        self.iq = torch.where(self.live, 1.0 / torch.where(self.live, self.q2, torch.ones_like(self.q2)), torch.zeros_like(self.q2))

    def mixed(self, pair):
        return _rule(self.cell, self.f, self.normal, _iso(pair[0], self.dim), _iso(pair[1], self.dim)) if len(self.f) else None

    def stress(self, e, extra=(0.0, 0.0)):
        """(c~ + extra) : e with an isotropic extra (lambda, 2 mu)."""
        s = (self.mu2 + extra[1]) * e
        s[: self.dim] += (self.lam + extra[0]) * e[: self.dim].sum(0)
        if self.Cx is not None:
            C = self.Cx + _iso((extra[0], 0.5 * extra[1]), self.dim)
            s[:, self.at] = torch.einsum("mij,jm->im", C, e[:, self.at])
        return s

    def iso0(self, e):
        s = 2.0 * self.mu0 * e
        s[: self.dim] += self.lam0 * e[: self.dim].sum(0)
        return s

    def strain_of(self, u):
        """(c~ + c0)^-1 : u."""
        m2, l = self.mu2 + 2.0 * self.mu0, self.lam + self.lam0
        e = u / m2
        e[: self.dim] -= l / (m2 * (m2 + self.dim * l)) * u[: self.dim].sum(0)
        if self.Cx is not None:
            C = self.Cx + _iso((self.lam0, self.mu0), self.dim)
            e[:, self.at] = torch.linalg.solve(C, u[:, self.at].T[:, :, None])[:, :, 0].T
        return e

    def hat(self, t):
        return torch.fft.rfftn(t.view((self.nc,) + (self.n,) * self.dim), dim=tuple(range(1, 1 + self.dim)))

    def real(self, t):
        return torch.fft.irfftn(t, s=(self.n,) * self.dim, dim=tuple(range(1, 1 + self.dim))).reshape(self.nc, self.nv)

    def traction(self, th):
        r, dim, xi = math.sqrt(0.5), self.dim, self.xi
        if dim == 2:
            return [xi[0] * th[0] + r * xi[1] * th[2], r * xi[0] * th[2] + xi[1] * th[1]]
        return [xi[0] * th[0] + r * (xi[1] * th[5] + xi[2] * th[4]), xi[1] * th[1] + r * (xi[0] * th[5] + xi[2] * th[3]),
                xi[2] * th[2] + r * (xi[0] * th[4] + xi[1] * th[3])]

    def gamma_hat(self, th):
        """Gamma0 : tau in Fourier space (zero at k = 0 and at Nyquist bins)."""
        v = self.traction(th)
        along = sum(x * a for x, a in zip(self.xi, v)) * ((self.lam0 + self.mu0) / (self.lam0 + 2 * self.mu0)) * self.iq
        u = [(a - x * along) * (self.iq / self.mu0) for x, a in zip(self.xi, v)]
        xi, r = self.xi, math.sqrt(0.5)
        e = [x * a for x, a in zip(xi, u)]
        for i, j in ([(0, 1)] if self.dim == 2 else [(1, 2), (0, 2), (0, 1)]):
            e.append(r * (xi[i] * u[j] + xi[j] * u[i]))
        return torch.stack(e)

    def with_mean(self, eh, m):
        eh[(slice(None),) + (0,) * self.dim] = m.to(eh.dtype) * self.nv
        return eh

    def basic(self, E, iters, tol=0.0, source=None):
        """Iterates of eps <- E - Gamma0 ((c~ - c0) : eps), or of the adjoint's w with a source; returns (eps, count)."""
        e = E[:, None].expand(-1, self.nv).clone()
        cs = self.stress(source) if source is not None else None
        for it in range(iters):
            s = self.stress(e)
            if tol > 0:
                sh = self.hat(s)
                r2 = sum((x.abs() ** 2 * self.weight * self.live).sum() for x in self.traction(sh))
                if float(r2.sqrt() / (s.mean(1).norm() * self.nv)) < tol:
                    return e, it
            t = s - self.iso0(e)
            if cs is not None:
                t -= cs
            e = self.real(self.with_mean(-self.gamma_hat(self.hat(t)), E))
        return e, iters

    def eyre_milton(self, E, iters):
        u = (2.0 * self.iso0(E[:, None])).expand(-1, self.nv).clone()
        add = 2.0 * self.iso0(E[:, None])
        for _ in range(iters):
            e = self.strain_of(u)
            t = self.stress(e) - self.iso0(e)
            g = self.real(self.gamma_hat(self.hat(t)))
            u = t - 2.0 * self.iso0(g) + add
        return self.strain_of(u)

    def conjugate_gradients(self, E, iters):
        """`iters` steps on G(c~ : (E + x)) = 0, G the projection onto compatible zero-mean strains (c0 = identity)."""
        def G(s):
            return self.real(self.gamma_hat(self.hat(s)))
        x = torch.zeros(self.nc, self.nv, dtype=torch.float64, device="cuda")
        r = -G(self.stress(E[:, None].expand(-1, self.nv).clone()))
        p, rr = r.clone(), r.square().sum()
        for _ in range(iters):
            q = G(self.stress(p))
            alpha = rr / (p * q).sum()
            x += alpha * p
            r -= alpha * q
            new = r.square().sum()
            p = r + (new / rr) * p
            rr = new
        return x + E[:, None]


def exact(case, seed):
    cells, phases, E, media = _geometry(case, seed)
    E = _cuda64(E)
    if case["kind"] == "gradient":
        return _exact_gradient(case, seed, cells[0], phases, media[0])
    single = np.float32 if case["fp"] == 32 else np.float64
    eps, sig, mean, count = [], [], [], []
    for cell, c0 in zip(cells, media):
        P = _Problem(cell, phases, (0.0, 0.5) if case["scheme"] == "cg" else c0)
        for El in E:
            it = case["iters"]
            if case["kind"] == "study":
                e, it = P.basic(El, 100000, 1e-4)
            elif case["scheme"] == "cg":
                e = P.conjugate_gradients(El, it)
            elif case["scheme"] == "em":
                e = P.eyre_milton(El, it)
            else:
                e, it = P.basic(El, it)
            s = P.stress(e)
            mean.append(s.mean(1).cpu().numpy())
            count.append(it)
            if case["kind"] != "study":
                eps.append(e.reshape(-1))
                sig.append(s.reshape(-1))
    mean = np.array(mean).reshape(len(cells), len(E), -1)
    out = {"mean_sigma": mean, "iterations": np.array(count, dtype=np.int32).reshape(len(cells), len(E))}
    if eps:
        out["eps"], out["sigma"] = torch.cat(eps), torch.cat(sig)
    if mean.shape[1] == mean.shape[2]:
        out["C"] = np.ascontiguousarray(mean.transpose(0, 2, 1))
    return out


def _exact_gradient(case, seed, cell, phases, c0):
    P = _Problem(cell, phases, c0)
    E = torch.eye(6, dtype=torch.float64, device="cuda")
    W = torch.from_numpy(np.random.default_rng([seed, 1]).standard_normal((6, 6))).cuda()
    eps = [P.basic(E[l], case["iters"])[0] for l in range(6)]
    sig = [P.stress(e) for e in eps]
    C = torch.stack([s.mean(1) for s in sig], 1)
    vm, A = 0.0, torch.zeros(6, 6, P.nv, dtype=torch.float64, device="cuda")
    for l in range(6):
        dev = sig[l].clone()
        dev[:3] -= dev[:3].mean(0)
        vm = vm + 1.5 * dev.square().sum(0).mean() / 6
        S = 3.0 * dev / (6.0 * P.nv)
        w, _ = P.basic(torch.zeros_like(E[0]), case["iters"], source=S)
        A += (S - w)[:, None, :] * eps[l][None]
        for j in range(6):
            A += W[l, j] / P.nv * eps[l][:, None, :] * eps[j][None]
    # dL = sum over voxels of A : dc~, c~ a function of the phase constants through the voxel's rule
    lame = P.pair.clone().requires_grad_(True)
    pure = [A[:, :, P.label == k].sum(2) for k in (0, 1)]
    L = sum((a * _iso(lame[k], 3)).sum() for k, a in enumerate(pure))
    if len(P.f):
        L = L + (A[:, :, P.at].permute(2, 0, 1) * P.mixed(lame)).sum()
    g, = torch.autograd.grad(L, lame)
    return {"C": C[None], "sigma": torch.cat([s.reshape(-1) for s in sig]), "vm": vm, "grad": g}
