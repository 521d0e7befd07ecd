"""What a user of this library has it do, as cases that can be timed and compared.

Every case goes through the public entry points (``paper_1401_7441_gb300.lsw``, the binding
of include/lsw.h).  The systems are the repository's own kinds of system: one support
function filling its box; atoms at the density and radii of the 64-atom, the 1,200-atom
and the 10,000-atom workloads.  Atoms sit at random inside the cells of a cubic lattice
with 1.8 bohr between any two; one or four support functions on each; one Gaussian well
per atom in the potential; coefficients normal with a Gaussian envelope, of unit norm.

A program keeps the system (its handle holds the plans, the workspace and the operator
tables) and the buffers.  The atoms are the case's; potential, functions, prefactors and
matrices come from the seed.

``exact`` holds the same operators in plain torch, in 64 bits: dense boxes, dense 1D filter
matrices and dense matrices of functions, with filters derived here from the 16 low-pass
coefficients of the least-asymmetric Daubechies wavelet of order 16.
"""
import math
from decimal import Decimal, getcontext

import numpy as np
import torch

from paper_1401_7441_gb300 import lsw

H = 0.45                 # coarse grid spacing, bohr
MARGIN = 8.0             # L' reaches this many grid steps beyond L
PAD = 14                 # fine points the filters reach beyond a box, and the kinetic half band
SIGMA = 2.0              # envelope of the support functions, bohr

# kind of system: lattice cell per atom (bohr), locreg radii, fine radius of a locreg radius,
# share of one-function atoms, pair cutoff (0: sum of the two radii)
SYSTEMS = {
    "sparse": dict(cell=7.5, radii=(6.0,), fine=lambda r: 2.0, light=0.25, cutoff=12.0),
    "mixed": dict(cell=5.65, radii=(5.0, 6.0, 7.0, 8.0), fine=lambda r: 0.3 * r, light=0.195, cutoff=0.0),
    "dense": dict(cell=5.1, radii=(7.0,), fine=lambda r: 2.1, light=0.4, cutoff=14.0),
}
PRECISION = {"fp64": lsw.LSW_FP64, "fp32": lsw.LSW_FP32, "bf16x": lsw.LSW_FP32_BF16X}


def listed():
    return [
        # one function on a 24^3 box: the smallest call, a chain of short launches
        dict(name="hphi_one_fp64", op="hphi", system="one", atoms=24, prec="fp64", batch=0, tile=0),
        # a small molecule in double precision, everything a step of the outer loop needs:
        # H phi with both energies, then H and S (library defaults)
        dict(name="step_64_fp64", op="step", system="sparse", atoms=64, prec="fp64", batch=0, tile=0),
        # the same molecule in single precision, library defaults
        dict(name="hphi_64_fp32", op="hphi", system="sparse", atoms=64, prec="fp32", batch=0, tile=0),
        # a nanometre-sized cluster with uneven radii, large batches
        dict(name="hphi_1200_fp32", op="hphi", system="mixed", atoms=1200, prec="fp32", batch=1024, tile=0),
        # a large dense system with the split-bfloat16 z stage, large batches: the production mode
        dict(name="hphi_3000_bf16x", op="hphi", system="dense", atoms=3000, prec="bf16x", batch=1024, tile=0),
        # H and S of given phi and H phi, once per step after the application
        dict(name="matrices_1200_fp32", op="matrices", system="mixed", atoms=1200, prec="fp32", batch=0, tile=8),
        dict(name="matrices_3000_bf16x", op="matrices", system="dense", atoms=3000, prec="bf16x", batch=0, tile=6),
        # the charge density from the density kernel, once per self-consistency cycle
        dict(name="density_300_fp32", op="density", system="mixed", atoms=300, prec="fp32", batch=256, tile=0),
        # re-orthonormalization of updated support functions
        dict(name="lowdin_600_fp32", op="lowdin", system="mixed", atoms=600, prec="fp32", batch=0, tile=6),
        # preconditioning of the support-function gradient: a few conjugate-gradient steps
        dict(name="precondition_20_fp32", op="precondition", system="sparse", atoms=20, prec="fp32", batch=0, tile=0,
             iters=4),
        # H phi of the first outer iterations, with the quartic confining potential
        dict(name="confined_27_fp64", op="confined", system="mixed", atoms=27, prec="fp64", batch=0, tile=0),
        # the density kernel by the Fermi operator expansion
        dict(name="foe_400_fp64", op="foe", system="mixed", atoms=400, prec="fp64", batch=0, tile=0, terms=80),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(["hphi"] * 4 + ["step", "matrices", "matrices", "density", "lowdin", "combine", "precondition",
                                    "confined", "foe"])
    case = dict(op=op, system=rng.choice(["sparse", "mixed", "dense"]), tile=rng.choice([0, 3, 5, 6, 7, 8]),
                batch=rng.choice([0, 0, 64, 200, 512, 1024]), prec="fp32")
    if op == "hphi":
        case["prec"] = rng.choice(["fp32", "bf16x", "bf16x", "fp64"])
        if rng.random() < 0.15:
            case.update(system="one", prec=rng.choice(["fp64", "fp32"]), atoms=rng.randint(13, 31))
        else:
            case["atoms"] = size(8, 60 if case["prec"] == "fp64" else 1400)
        if case["prec"] == "fp64":
            case["batch"] = 0
    elif op == "step":
        case.update(prec="fp64", atoms=size(4, 64), batch=0)
    elif op == "matrices":
        case.update(prec=rng.choice(["fp32", "bf16x"]), atoms=size(10, 1400), batch=0)
    elif op == "density":
        case.update(prec=rng.choice(["fp32", "bf16x"]), atoms=size(10, 300))
    elif op in ("lowdin", "combine"):
        case.update(prec=rng.choice(["fp32", "bf16x", "fp64"]), atoms=size(10, 600), batch=0)
        if case["prec"] == "fp64":
            case["atoms"] = min(case["atoms"], 150)
    elif op == "precondition":
        case.update(prec=rng.choice(["fp32", "bf16x", "fp64"]), atoms=size(2, 9), iters=rng.randint(2, 4), batch=0)
    elif op == "confined":
        case.update(prec=rng.choice(["fp32", "bf16x", "fp64"]), atoms=size(3, 24), batch=0)
    else:
        case.update(prec="fp64", system="mixed", atoms=size(20, 400), terms=rng.randint(25, 90), batch=0)
    return case


# ------------------------------------------------------------------ geometry and inputs


class Geometry:
    """Atoms, grid, locreg members and compressed layout of a case."""

    def __init__(self, case, seed, device):
        self.device = device
        self.gen = torch.Generator(device=device).manual_seed(seed * 7919 + 17)
        rng = np.random.RandomState(1000 * case["atoms"] + len(case["system"]))     # atoms: the case's
        if case["system"] == "one":      # one function, every point of the box a member
            n = case["atoms"]
            self.N = (n, n, n)
            self.pos = np.array([[n // 2 * H] * 3])
            self.r_loc = np.array([100.0])
            self.r_fine = np.array([n / 4.0 * H * (1 + 1e-9)])
            self.nsf = np.array([1], np.int32)
            self.cutoff = 12.0
            box = (n - 1) * H
            centres = box * (0.25 + 0.5 * rng.rand(4, 3))
        else:
            k = SYSTEMS[case["system"]]
            n = case["atoms"]
            m = int(math.ceil(round(n ** (1.0 / 3.0), 9)))
            cube = k["cell"] * n ** (1.0 / 3.0)
            cell = cube / m
            at = np.sort(rng.permutation(m ** 3)[:n])
            idx = np.stack([at % m, at // m % m, at // (m * m)], 1)
            room = max(cell - 1.8, 0.0)
            rmax = max(k["radii"])
            self.pos = rmax + cell * idx + 0.5 * (cell - room) + room * rng.rand(n, 3)
            self.r_loc = np.array(k["radii"])[rng.randint(0, len(k["radii"]), n)]
            self.r_fine = np.array([k["fine"](r) for r in self.r_loc])
            self.nsf = np.where(rng.rand(n) < k["light"], 1, 4).astype(np.int32)
            self.N = (int(math.ceil((cube + 2 * rmax) / H)) + 1,) * 3
            self.cutoff = k["cutoff"]
            centres = self.pos
        rng = np.random.RandomState((seed * 2654435761 + 99) % (1 << 32))           # the rest: the seed's
        self.wells = np.column_stack([centres, 1.0 + 2.0 * rng.rand(len(centres)), 0.5 + rng.rand(len(centres))])
        self.first = np.concatenate([[0], np.cumsum(self.nsf)])
        self.n_sf = int(self.first[-1])
        self.sf_atom = np.repeat(np.arange(len(self.pos)), self.nsf)
        self.rng = rng
        N = self.N
        self.fine = torch.zeros((N[2], N[1], N[0]), dtype=torch.bool, device=device)
        for zyx, _ in self._spheres(self.r_fine):
            self.fine[zyx[:, 1], zyx[:, 2], zyx[:, 3]] = True
        self.L = self._members(self.r_loc)
        self.off_L = self._offsets(self.L)
        self._Lp = None

    @property
    def Lp(self):
        if self._Lp is None:
            self._Lp = self._members(self.r_loc + MARGIN * H)
        return self._Lp

    def _spheres(self, radii):
        """(rows of (atom, z, y, x) of the grid points within `radii`, atoms) in chunks of atoms;
        the rows run along x fastest."""
        N = torch.tensor(self.N, device=self.device)
        W = int(math.ceil(2 * float(np.max(radii)) / H)) + 4
        W = min(W, max(self.N))
        step = max(1, (1 << 26) // W ** 3)
        o = torch.arange(W, device=self.device)
        for a0 in range(0, len(self.pos), step):
            a1 = min(len(self.pos), a0 + step)
            c = torch.tensor(self.pos[a0:a1], device=self.device)
            r = torch.tensor(np.asarray(radii)[a0:a1], device=self.device)
            lo = torch.clamp(torch.floor((c - r[:, None]) / H).long() - 1, min=0)
            g = lo[:, :, None] + o                                   # (atoms, dimension, W)
            d = g.double() * H - c[:, :, None]
            d = d * d
            s = (d[:, 0, None, None, :] + d[:, 1, None, :, None]) + d[:, 2, :, None, None]
            s = s <= (r * r)[:, None, None, None]
            ok = g < N[None, :, None]
            s &= ok[:, 0, None, None, :] & ok[:, 1, None, :, None] & ok[:, 2, :, None, None]
            at = s.nonzero()
            a = at[:, 0]
            yield torch.stack([a + a0, lo[a, 2] + at[:, 1], lo[a, 1] + at[:, 2], lo[a, 0] + at[:, 3]], 1), range(a0, a1)

    def _members(self, radii):
        """Per atom: box origin (x, y, z), extents, and the flat box indices (x fastest) of its
        coarse and of its fine members, in layout order."""
        out = []
        for rows, atoms in self._spheres(radii):
            fine = self.fine[rows[:, 1], rows[:, 2], rows[:, 3]]
            n = len(atoms)
            a = rows[:, 0] - atoms[0]
            big = torch.full((n, 3), 1 << 30, dtype=torch.long, device=self.device)
            ix = a[:, None].expand(-1, 3)
            lo = big.scatter_reduce(0, ix, rows[:, 1:], "amin")
            hi = (-big).scatter_reduce(0, ix, rows[:, 1:], "amax")
            n3 = hi - lo + 1
            l = rows[:, 1:] - lo[a]
            flat = (l[:, 0] * n3[a, 1] + l[:, 1]) * n3[a, 2] + l[:, 2]
            cnt = torch.bincount(a, minlength=n).tolist()
            fcnt = torch.bincount(a[fine], minlength=n).tolist()
            lo, n3 = lo.flip(1).tolist(), n3.flip(1).tolist()
            out += list(zip(lo, n3, flat.split(cnt), flat[fine].split(fcnt)))
        return out

    def _offsets(self, members):
        n = np.array([len(m[2]) + 7 * len(m[3]) for m in members], np.int64)[self.sf_atom]
        return np.concatenate([[0], np.cumsum((n + 63) // 64 * 64)])

    @property
    def off_Lp(self):
        return self._offsets(self.Lp)

    def functions(self, members, off, dtype):
        """Coefficients of every function on `members`: normal, enveloped, of unit norm."""
        v = torch.zeros(int(off[-1]), dtype=torch.float64, device=self.device)
        for a, (lo, n, c, f) in enumerate(members):
            d = [(torch.arange(n[k], device=self.device).double() + lo[k]) * H - self.pos[a][k] for k in range(3)]
            r2 = (d[2] ** 2)[:, None, None] + (d[1] ** 2)[None, :, None] + (d[0] ** 2)[None, None, :]
            e = torch.exp(r2 * (-0.5 / SIGMA ** 2)).reshape(-1)
            k = self.nsf[a]
            w = torch.cat([e[c], e[f].repeat(7)]).repeat(k, 1)
            w = w * torch.randn(w.shape, generator=self.gen, dtype=torch.float64, device=self.device)
            w = w / w.norm(dim=1, keepdim=True)
            o = int(off[self.first[a]])
            v[o:o + k * int((w.shape[1] + 63) // 64 * 64)].view(k, -1)[:, :w.shape[1]] = w
        return v.to(dtype)

    def potential(self, dtype):
        """Wells on the fine grid from index -14, [z, y, x]."""
        w = torch.tensor(self.wells, device=self.device)
        e = []
        for d in range(3):
            x = (torch.arange(2 * self.N[d] + 2 * PAD + 1, device=self.device).double() - PAD) * (H / 2)
            e.append(torch.exp(-((x - w[:, d:d + 1]) ** 2) / (2 * w[:, 4:5] ** 2)))
        V = torch.empty((e[2].shape[1], e[1].shape[1], e[0].shape[1]), dtype=dtype, device=self.device)
        for z in range(0, V.shape[0], 16):
            ez = (-w[:, 3:4] * e[2])[:, z:z + 16]
            V[z:z + 16] = ((ez[:, :, None] * e[1][:, None, :]).reshape(len(w), -1).T @ e[0]).view(-1, *V.shape[1:])
        return V

    def pattern(self):
        """Rows and columns of the pair pattern, row by row with ascending columns."""
        p = torch.tensor(self.pos, device=self.device)
        d = p[:, None, :] - p[None, :, :]
        d = d * d
        r = torch.tensor(self.r_loc, device=self.device)
        c = r[:, None] + r[None, :] if not self.cutoff else torch.full((1, 1), self.cutoff, device=self.device).double()
        near = (d[..., 0] + d[..., 1]) + d[..., 2] <= c * c
        at = torch.tensor(self.sf_atom, device=self.device)
        rows, cols = near[at][:, at].nonzero(as_tuple=True)
        dist = torch.sqrt(((p[at[rows]] - p[at[cols]]) ** 2).sum(1))
        return rows, cols, dist

    def pair_values(self, rows, cols):
        """One uniform value per unordered pair of functions."""
        n = self.n_sf
        u = torch.rand((n, n), generator=self.gen, dtype=torch.float64, device=self.device)
        u = torch.triu(u) + torch.triu(u, 1).T
        return u[rows, cols]


def _matrices(geo):
    """A decaying symmetric Hamiltonian and an overlap near the identity on the pattern, and
    bounds of the spectrum of H c = e S c."""
    rows, cols, dist = geo.pattern()
    diag = rows == cols
    S = (geo.pair_values(rows, cols) - 0.5) * torch.exp(-dist ** 2 / 18)
    S[diag] = 0.0
    total = torch.zeros(geo.n_sf, dtype=torch.float64, device=S.device)
    reach = total.index_add(0, rows, S.abs()).max()
    S = S * (0.3 / reach)
    S[diag] = 1.0
    Hm = (geo.pair_values(rows, cols) - 0.5) * torch.exp(-dist ** 2 / 18)
    top = float(total.index_add(0, rows, Hm.abs()).max()) / 0.7 * 1.05
    return rows, cols, Hm, S, top


def _kernel(geo):
    rows, cols, dist = geo.pattern()
    return rows, cols, (0.5 + geo.pair_values(rows, cols)) * torch.exp(-dist ** 2 / 18)


_KEPT = {}               # the library context and stream that a program keeps


def _context():
    if not _KEPT:
        _KEPT["stream"] = torch.cuda.Stream()
        _KEPT["ctx"] = lsw.lsw_ctx_create(torch.cuda.current_device(), _KEPT["stream"].cuda_stream)
    return _KEPT["ctx"]


def prepare(case, seed):
    dev = torch.device("cuda")
    geo = Geometry(case, seed, dev)
    S = lsw.System(geo.N, H, geo.pos, geo.r_loc, geo.r_fine, geo.nsf, geo.cutoff, 0 if geo.cutoff else 1, MARGIN, 0,
                   PRECISION[case["prec"]], ctx=_context())
    if case["batch"]:
        lsw.lsw_set_option(S.sys, "batch", min(case["batch"], geo.n_sf))
    if case["tile"]:
        lsw.lsw_set_option(S.sys, "tile", case["tile"])
    dt = torch.float64 if case["prec"] == "fp64" else torch.float32
    op = case["op"]
    st = dict(op=op, S=S, sys=S.sys)
    if op != "foe":
        st["phi"] = geo.functions(geo.L, geo.off_L, dt)
        assert st["phi"].numel() == S.total_L
    if op in ("hphi", "step", "confined"):
        st["V"] = geo.potential(dt)
        lsw.lsw_set_potential(S.sys, st["V"], (-PAD,) * 3, tuple(2 * n + 2 * PAD + 1 for n in geo.N))
        st["hphi"] = torch.zeros(S.total_Lp, dtype=dt, device=dev)
        # energies: with the double-precision step; a plain application leaves them out (optional
        # arguments), as a support-function update that takes its energy from Tr(KH) does
        full = case["prec"] == "fp64"
        st["e_kin"] = torch.zeros(geo.n_sf, dtype=torch.float64, device=dev) if full else None
        st["e_pot"] = torch.zeros_like(st["e_kin"]) if full else None
    nnz = len(S.col)
    if op in ("step", "matrices"):
        st["H"] = torch.zeros(nnz, dtype=torch.float64, device=dev)
        st["Sm"] = torch.zeros_like(st["H"])
    if op == "matrices":
        st["hphi"] = geo.functions(geo.Lp, geo.off_Lp, dt)
        assert st["hphi"].numel() == S.total_Lp
    if op == "density":
        st["K"] = _kernel(geo)[2]
        st["lo"], st["dims"] = (-PAD,) * 3, tuple(2 * n + 2 * PAD + 1 for n in geo.N)
        st["rho"] = torch.zeros(st["dims"][::-1], dtype=torch.float64, device=dev)
    if op in ("lowdin", "combine"):
        st["M"] = _matrices(geo)[3] if op == "lowdin" else _kernel(geo)[2]
        st["out"] = torch.zeros_like(st["phi"])
    if op in ("precondition", "confined"):
        u = torch.tensor(geo.rng.rand(2, geo.n_sf), device=dev)
        st["a"] = 2e-3 + 3e-3 * u[0]
        st["eps"] = -0.2 - 0.6 * u[1]
        full = case["prec"] == "fp64"
        if op == "precondition":
            st["iters"] = case["iters"]
            st["out"] = torch.zeros_like(st["phi"])
            st["res"] = torch.zeros((case["iters"], geo.n_sf), dtype=torch.float64, device=dev) if full else None
        else:
            st["e_conf"] = torch.zeros(geo.n_sf, dtype=torch.float64, device=dev) if full else None
    if op == "foe":
        _, _, st["H"], st["Sm"], st["top"] = _matrices(geo)
        st["n_el"], st["terms"] = 0.4 * geo.n_sf, case["terms"]
        st["Kp"] = torch.zeros(nnz, dtype=torch.float64, device=dev)
        st["K"] = torch.zeros_like(st["Kp"])
        assert st["H"].numel() == nnz
    torch.cuda.synchronize()
    return st


def run(st):
    op, s = st["op"], st["sys"]
    if op in ("hphi", "step", "confined"):
        lsw.lsw_apply_hamiltonian(s, st["phi"], st["hphi"], st["e_kin"], st["e_pot"])
        out = [st["hphi"], st["e_kin"], st["e_pot"]]
        if op == "step":
            lsw.lsw_build_matrices(s, st["phi"], st["hphi"], st["H"], st["Sm"])
            out += [st["H"], st["Sm"]]
        if op == "confined":
            lsw.lsw_add_confinement(s, st["a"], st["phi"], st["hphi"], st["e_conf"])
            out.append(st["e_conf"])
        return out
    if op == "matrices":
        lsw.lsw_build_matrices(s, st["phi"], st["hphi"], st["H"], st["Sm"])
        return [st["H"], st["Sm"]]
    if op == "density":
        lsw.lsw_build_density(s, st["phi"], st["K"], st["rho"], st["lo"], st["dims"])
        return [st["rho"]]
    if op == "lowdin":
        lsw.lsw_lowdin_taylor(s, st["M"], st["phi"], st["out"])
        return [st["out"]]
    if op == "combine":
        lsw.lsw_combine(s, st["M"], st["phi"], st["out"])
        return [st["out"]]
    if op == "precondition":
        lsw.lsw_precondition(s, st["a"], st["eps"], st["phi"], st["out"], st["iters"], st["res"])
        return [st["out"], st["res"]]
    mu, ebs, trace = lsw.lsw_foe(s, st["H"], st["Sm"], -st["top"], st["top"], st["n_el"], st["terms"],
                                 0.08 * st["top"], st["Kp"], st["K"])
    return [st["Kp"], st["K"], mu, ebs, trace]


# ------------------------------------------------------------------ work


def work(case):
    """The coefficients, potential, matrices and density in and out once; the multiply-adds of
    the separable passes over the nonzero data of spheres (2 flop per tap), of the pairs'
    common coefficients, of the pairs' common real-space points, of the pattern's products."""
    geo = Geometry(case, 1, torch.device("cuda" if torch.cuda.is_available() else "cpu"))
    es = 8 if case["prec"] == "fp64" else 4
    op = case["op"]
    R = geo.r_loc[geo.sf_atom] / H
    if case["system"] == "one":
        R = np.array([geo.N[0] * (3 / (4 * math.pi)) ** (1.0 / 3.0)])
    ncoef = np.diff(geo.off_L).astype(float)
    nc = np.minimum(4.19 * R ** 3, ncoef)
    fine = np.clip((ncoef / nc - 1) / 7, 0, 1)                          # fine share of the members
    Rp = R + (MARGIN if case["system"] != "one" else 0.0)
    ncp = 4.19 * Rp ** 3
    coefp = ncp * (1 + 7 * fine)
    X = 4 * R + 29
    n_v = float(np.prod([2.0 * n + 2 * PAD + 1 for n in geo.N]))
    fwd = 62.0 * (ncoef + 4 * 3.14 * R ** 2 * X + 2 * 2 * R * X ** 2)
    back = 62.0 * (coefp + 4 * 3.14 * Rp ** 2 * X + 2 * 2 * Rp * X ** 2)
    arm = 2 * 29 * 2.0
    app_b = es * (ncoef.sum() + coefp.sum() + n_v)
    app_f = (fwd + 3 * X ** 3 + back + 3 * arm * ncoef).sum()
    if op == "hphi":
        return {"bytes": app_b, "flops": app_f}
    rows, cols, dist = geo.pattern()
    nnz = len(rows)
    r1, r2, dist = R[rows.cpu().numpy()], R[cols.cpu().numpy()], dist.cpu().numpy() / H

    def lens(a, b, d):       # common volume of two spheres
        d = np.maximum(d, 1e-9)
        cut = np.pi * (a + b - d) ** 2 * (d * d + 2 * d * (a + b) - 3 * (a - b) ** 2) / (12 * d)
        return np.where(d >= a + b, 0.0, np.where(d <= np.abs(a - b), 4.19 * np.minimum(a, b) ** 3, cut))

    per = 1 + 7 * float(fine.mean())
    s_f, h_f = 2 * per * lens(r1, r2, dist).sum(), 2 * per * lens(r1, r2 + MARGIN, dist).sum()
    if op in ("step", "matrices"):
        w = {"bytes": es * (ncoef.sum() + coefp.sum()) + 16.0 * nnz, "flops": s_f + h_f}
        return w if op == "matrices" else {"bytes": w["bytes"] + app_b, "flops": w["flops"] + app_f}
    if op == "density":
        pts = 8 * lens(r1 + 7, r2 + 7, dist).sum() / 2
        return {"bytes": es * ncoef.sum() + 8.0 * (nnz + n_v), "flops": float(fwd.sum() + 2 * pts)}
    if op in ("lowdin", "combine"):
        return {"bytes": 2 * es * ncoef.sum() + 8.0 * nnz, "flops": float(s_f)}
    quartic = 7 * arm        # three X^4, and four X^2 passes give the three cross terms
    if op == "precondition":
        k = case["iters"]
        return {"bytes": 2 * es * ncoef.sum() + 16.0 * geo.n_sf, "flops": float(k * (quartic + 3 * arm + 10) * ncoef.sum())}
    if op == "confined":
        return {"bytes": app_b + es * 2 * coefp.sum(), "flops": float(app_f + quartic * coefp.sum())}
    n = nnz / geo.n_sf
    return {"bytes": 8.0 * 4 * nnz, "flops": 2.0 * nnz * n * 0.6 * (case["terms"] + 4)}


# ------------------------------------------------------------------ 64-bit values

# low-pass filter h_j, j = -7 .. 8, of the least-asymmetric Daubechies wavelet of order 16
LOW_PASS = """
-3.382415951005002595457699235919135128243e-3 -5.421323318000106893478369440173478588246e-4
3.169508781152599143142570752391597485718e-2 7.607487324976608191921008012192383923495e-3
-1.432942383512726628440955443992739699342e-1 -6.127335906781107784304676907365841265563e-2
4.813596512590533915895685802649845258386e-1 7.771857516996280286243335666392108091213e-1
3.644418948361789367595594323842960136511e-1 -5.194583810788180073571072906256342852964e-2
-2.721902991710348632196412421624687935352e-2 4.913717967373028678691098815516544290155e-2
3.808752013894489463071922223049694342708e-3 -1.495225833706219911849029822472598879079e-2
-3.029205147241330812639124399571849886852e-4 1.889950332767689184274432603245581173346e-3
"""
_FILTERS = {}


def _solve(A, b):
    """A x = b by elimination with row pivots, in Decimal."""
    n = len(b)
    A = [list(r) + [y] for r, y in zip(A, b)]
    for k in range(n):
        p = max(range(k, n), key=lambda i: abs(A[i][k]))
        A[k], A[p] = A[p], A[k]
        for i in range(k + 1, n):
            if A[i][k]:
                q = A[i][k] / A[k][k]
                A[i] = [u - q * v for u, v in zip(A[i], A[k])]
    x = [Decimal(0)] * n
    for k in reversed(range(n)):
        x[k] = (A[k][n] - sum(A[k][j] * x[j] for j in range(k + 1, n))) / A[k][k]
    return x


def filters():
    """Combined synthesis and quadrature filters [2][31], kinetic blocks [2][2][29] and the
    moment overlaps [5][29] of the basis, from their two-scale equations."""
    if _FILTERS:
        return _FILTERS
    getcontext().prec = 60
    h = {j: Decimal(t) for j, t in zip(range(-7, 9), LOW_PASS.split())}
    g = {j: (h[1 - j] if j % 2 == 0 else -h[1 - j]) for j in h}
    root2 = Decimal(2).sqrt()
    moments = [Decimal(1)]
    for p in range(1, 16):
        acc = sum(math.comb(p, i) * moments[i] * sum(h[j] * Decimal(j) ** (p - i) for j in h) for i in range(p))
        moments.append(root2 * acc / (2 ** (p + 1) * (1 - Decimal(2) ** -p)))
    # point values from coefficients: the 16 taps with the moments of the scaling function
    taps = _solve([[Decimal(l) ** p if p else Decimal(1) for l in range(-7, 9)] for p in range(16)], moments)
    w = dict(zip(range(-7, 9), taps))
    fwd = [[sum(w.get(m - k, 0) * f[k] for k in f) for m in range(-14, 17)] for f in (h, g)]
    auto = {d: sum(h[i] * h.get(i + d, 0) for i in h) for d in range(-15, 16)}
    band = range(-14, 15)
    A = [[(1 if l == m else 0) - 4 * auto.get(m - 2 * l, Decimal(0)) for m in band] for l in band]
    A[-1] = [Decimal(m * m) for m in band]
    r = dict(zip(band, _solve(A, [Decimal(0)] * 28 + [Decimal(2)])))
    kin = [[[4 * sum(x[k] * y[q] * r.get(2 * l + q - k, 0) for k in x for q in y) for l in band] for y in (h, g)]
           for x in (h, g)]
    over = [{l: Decimal(int(l == 0)) for l in band}]
    for p in range(1, 5):
        s = Decimal(2) ** -p
        A = [[(1 if l == m else 0) - s * auto.get(m - 2 * l, Decimal(0)) for m in band] for l in band]
        b = [s * sum(math.comb(p, q) * Decimal(i) ** (p - q) * h[i] * h[j] * over[q].get(2 * l + j - i, 0)
                     for q in range(p) for i in h for j in h) for l in band]
        over.append(dict(zip(band, _solve(A, b))))

    def f64(v):
        return np.array(v, dtype=object).astype(np.float64)

    _FILTERS.update(fwd=f64(fwd), kin=f64(kin), over=f64([[o[l] for l in band] for o in over]),
                    pair=f64([[h[j] for j in h], [g[j] for j in g]]))
    return _FILTERS


def _toeplitz(table, rows, cols, lead):
    """M[i, j] = table[lead(i, j)], 0 where the index falls outside."""
    i, j = np.meshgrid(np.arange(rows), np.arange(cols), indexing="ij")
    k = lead(i, j)
    ok = (k >= 0) & (k < len(table))
    return np.where(ok, table[np.clip(k, 0, len(table) - 1)], 0.0)


def _quartic(lo, n, centre, m):
    """[2 n, 2 n]: <chi_b,i | (x - centre)^m | chi_b',j> on coarse points lo .. lo + n - 1."""
    F = filters()
    ks = np.arange(-7, 9)
    base = 2.0 * (lo + np.arange(n))[:, None] + ks - 2.0 * centre / H
    out = np.zeros((2, n, 2, n))
    for d in range(-14, 15):
        l = 2 * d + ks[None, :] - ks[:, None]
        ok = np.abs(l) <= 14
        i = np.arange(max(0, -d), min(n, n - d))
        for b in range(2):
            for bp in range(2):
                v = sum(math.comb(m, p) * (base ** (m - p) * F["pair"][b]) @
                        (np.where(ok, F["over"][p][np.clip(l + 14, 0, 28)], 0.0) @ F["pair"][bp]) for p in range(m + 1))
                out[b, i, bp, i + d] = v[i]
    return out.reshape(2 * n, 2 * n) * (H / 2) ** m


class Dense:
    """The operators on one atom's dense boxes; box arrays are [f, bz, by, bx, z, y, x]."""

    def __init__(self, geo, a):
        self.geo, self.a, self.dev = geo, a, geo.device
        self.lo, self.n, self.c, self.f = geo.L[a]

    def t(self, x):
        return torch.tensor(x, dtype=torch.float64, device=self.dev)

    def load(self, members, vec, off):
        lo, n, c, f = members
        k = int(self.geo.nsf[self.a])
        o = int(off[self.geo.first[self.a]])
        size = len(c) + 7 * len(f)
        v = vec[o:o + k * int((size + 63) // 64 * 64)].view(k, -1)
        D = torch.zeros((k, 8, n[0] * n[1] * n[2]), dtype=torch.float64, device=self.dev)
        D[:, 0, c] = v[:, :len(c)].double()
        D[:, 1:, f] = v[:, len(c):size].double().view(k, 7, -1)
        return D.view(k, 2, 2, 2, n[2], n[1], n[0])

    def store(self, members, D, vec, off):
        lo, n, c, f = members
        k = D.shape[0]
        o = int(off[self.geo.first[self.a]])
        size = len(c) + 7 * len(f)
        v = vec[o:o + k * int((size + 63) // 64 * 64)].view(k, -1)
        D = D.reshape(k, 8, -1)
        v[:, :len(c)] = D[:, 0, c]
        v[:, len(c):size] = D[:, 1:, f].reshape(k, -1)

    def along(self, M, D, dim):
        """A [2 n', 2 n] two-level 1D operator along x (0), y (1) or z (2)."""
        k = D.ndim - 1 - dim
        b = 3 - dim
        P = D.movedim((b, k), (-2, -1))
        s = P.shape
        R = P.reshape(-1, s[-2] * s[-1]) @ M.T
        return R.view(*s[:-2], 2, M.shape[0] // 2).movedim((-2, -1), (b, k))

    def realspace(self, D):
        F = filters()["fwd"]
        u = D
        for d in range(3):     # the type axis of each dimension is summed away (kept with extent 1)
            n = self.n[d]
            M = self.t(np.concatenate([_toeplitz(F[b], 2 * n + 29, n, lambda i, j: i - 2 * j) for b in (0, 1)], 1))
            k, b = u.ndim - 1 - d, 3 - d
            P = u.movedim((b, k), (-2, -1))
            s = P.shape
            u = (P.reshape(-1, 2 * n) @ M.T).view(*s[:-2], 1, -1).movedim((-2, -1), (b, k))
        return u

    def coefficients(self, v):
        F = filters()["fwd"]
        lop, np_ = self.geo.Lp[self.a][:2]
        for d in range(3):
            n, dz = self.n[d], lop[d] - self.lo[d]
            M = self.t(np.concatenate([_toeplitz(F[b], 2 * n + 29, np_[d], lambda i, j: i - 2 * (j + dz)).T
                                       for b in (0, 1)], 0))
            k, b = v.ndim - 1 - d, 3 - d
            P = v.movedim((b, k), (-2, -1))
            s = P.shape
            v = (P.reshape(-1, s[-1]) @ M.T).view(*s[:-2], 2, np_[d]).movedim((-2, -1), (b, k))
        return v

    def kinetic(self, n):
        K = filters()["kin"]
        return [self.t(np.block([[_toeplitz(K[b][c], n[d], n[d], lambda i, j: j - i + 14) for c in (0, 1)]
                                 for b in (0, 1)])) * (-0.5 / H ** 2) for d in range(3)]

    def widened(self, D):
        """The box of L placed in the box of L'."""
        lop, np_ = self.geo.Lp[self.a][:2]
        o = [self.lo[d] - lop[d] for d in range(3)]
        n = self.n
        P = torch.zeros(D.shape[:4] + (np_[2], np_[1], np_[0]), dtype=torch.float64, device=self.dev)
        P[..., o[2]:o[2] + n[2], o[1]:o[1] + n[1], o[0]:o[0] + n[0]] = D
        return P

    def hamiltonian(self, D, V):
        lo, n = self.lo, self.n
        Vs = V[2 * lo[2]:2 * lo[2] + 2 * n[2] + 29, 2 * lo[1]:2 * lo[1] + 2 * n[1] + 29,
               2 * lo[0]:2 * lo[0] + 2 * n[0] + 29].double()
        u = self.realspace(D)
        v = Vs * u
        e_pot = (v * u).flatten(1).sum(1)
        P = self.widened(D)
        T = sum(self.along(M, P, d) for d, M in enumerate(self.kinetic(P.shape[:3:-1])))
        return self.coefficients(v) + T, (T * P).flatten(1).sum(1), e_pot

    def confinement(self, P, lo, a):
        n = P.shape[:3:-1]
        c = self.geo.pos[self.a]
        Q4 = [self.t(_quartic(lo[d], n[d], c[d], 4)) for d in range(3)]
        Q2 = [self.t(_quartic(lo[d], n[d], c[d], 2)) for d in range(3)]

        def apply(P):
            z = self.along(Q2[2], P, 2)
            yz = self.along(Q2[1], P, 1) + z
            out = sum(self.along(Q4[d], P, d) for d in range(3))
            out = out + 2 * self.along(Q2[1], z, 1) + 2 * self.along(Q2[0], yz, 0)
            return out * a.view(-1, 1, 1, 1, 1, 1, 1)

        return apply


def _each_atom(geo):
    for a in range(len(geo.pos)):
        if geo.nsf[a]:
            yield a, slice(int(geo.first[a]), int(geo.first[a + 1])), Dense(geo, a)


def _tiles(boxes, T, width, lead):
    """For every tile of T^3 points: the functions whose boxes meet it and their values there
    [function, lead * T^3].  boxes: per atom (origin, extents, functions, [f, lead, z, y, x])."""
    lo = np.array([b[0] for b in boxes])
    hi = lo + np.array([b[1] for b in boxes])
    for tz in range(0, width[2], T):
        for ty in range(0, width[1], T):
            for tx in range(0, width[0], T):
                t0 = np.array([tx, ty, tz])
                meet = np.nonzero(np.all((lo < t0 + T) & (hi > t0), axis=1))[0]
                if not len(meet):
                    continue
                ids = np.concatenate([np.arange(boxes[a][2].start, boxes[a][2].stop) for a in meet])
                P = torch.zeros((len(ids), lead, T, T, T), dtype=torch.float64, device=boxes[0][3].device)
                k = 0
                for a in meet:
                    s = np.maximum(lo[a], t0)
                    e = np.minimum(hi[a], t0 + T)
                    src = tuple(slice(int(s[d] - lo[a][d]), int(e[d] - lo[a][d])) for d in (2, 1, 0))
                    dst = tuple(slice(int(s[d] - t0[d]), int(e[d] - t0[d])) for d in (2, 1, 0))
                    nf = boxes[a][2].stop - boxes[a][2].start
                    P[(slice(k, k + nf), slice(None)) + dst] = boxes[a][3][(slice(None), slice(None)) + src]
                    k += nf
                yield tuple(t0), meet, torch.tensor(ids, device=P.device), P.view(len(ids), -1)


def _boxes(geo, members, vec, off):
    return [(members[a][0], members[a][1], fs, D.load(members[a], vec, off).flatten(1, 3))
            for a, fs, D in _each_atom(geo)]


def _overlaps(geo, phi, hphi, off_Lp):
    """H and S on the pattern, from the functions' values tile by tile."""
    T = 16
    dev = geo.device
    Hd = torch.zeros((geo.n_sf, geo.n_sf), dtype=torch.float64, device=dev)
    Sd = torch.zeros_like(Hd)
    A = {t: (i, P) for t, _, i, P in _tiles(_boxes(geo, geo.L, phi, geo.off_L), T, geo.N, 8)}
    for t, _, j, Q in _tiles(_boxes(geo, geo.Lp, hphi, off_Lp), T, geo.N, 8):
        if t in A:
            i, P = A.pop(t)
            Hd[i[:, None], j[None, :]] += P @ Q.T
            Sd[i[:, None], i[None, :]] += P @ P.T
    rows, cols, _ = geo.pattern()
    return Hd[rows, cols], Sd[rows, cols]


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    geo = Geometry(case, seed, dev)
    dt = torch.float64 if case["prec"] == "fp64" else torch.float32
    op = case["op"]
    full = case["prec"] == "fp64"
    phi = geo.functions(geo.L, geo.off_L, dt) if op != "foe" else None
    if op in ("hphi", "step", "confined"):
        V = geo.potential(dt)
        off = geo.off_Lp
        out = torch.zeros(int(off[-1]), dtype=torch.float64, device=dev)
        e = torch.zeros((3, geo.n_sf), dtype=torch.float64, device=dev)
        a = 2e-3 + 3e-3 * torch.tensor(geo.rng.rand(2, geo.n_sf), device=dev)[0] if op == "confined" else None
        for k, fs, D in _each_atom(geo):
            P = D.load(geo.L[k], phi, geo.off_L)
            R, e[0, fs], e[1, fs] = D.hamiltonian(P, V)
            if op == "confined":
                W = D.widened(P)
                Q = D.confinement(W, geo.Lp[k][0], a[fs])(W)
                e[2, fs] = (Q * W).flatten(1).sum(1)
                R = R + Q
            D.store(geo.Lp[k], R, out, off)
        got = [out, e[0] if full else None, e[1] if full else None]
        if op == "confined":
            got.append(e[2] if full else None)
        if op == "step":
            got += _overlaps(geo, phi, out, off)
        return got
    if op == "matrices":
        if geo.n_sf > 5000:
            return None
        return list(_overlaps(geo, phi, geo.functions(geo.Lp, geo.off_Lp, dt), geo.off_Lp))
    if op == "density":
        rows, cols, K = _kernel(geo)
        Kd = torch.zeros((geo.n_sf, geo.n_sf), dtype=torch.float64, device=dev)
        Kd[rows, cols] = K
        dims = [2 * n + 2 * PAD + 1 for n in geo.N]
        boxes = []
        for k, fs, D in _each_atom(geo):
            u = D.realspace(D.load(geo.L[k], phi, geo.off_L)).flatten(1, 3)
            boxes.append(([2 * x for x in D.lo], [2 * x + 29 for x in D.n], fs, u))
        rho = torch.zeros(dims[::-1], dtype=torch.float64, device=dev)
        for t, _, i, U in _tiles(boxes, 32, dims, 1):
            v = ((Kd[i][:, i] @ U) * U).sum(0).view(32, 32, 32)
            e = [min(32, dims[d] - t[d]) for d in range(3)]
            rho[t[2]:t[2] + e[2], t[1]:t[1] + e[1], t[0]:t[0] + e[0]] = v[:e[2], :e[1], :e[0]]
        return [rho]
    if op in ("lowdin", "combine"):
        if op == "lowdin":
            rows, cols, _, M, _ = _matrices(geo)
            M = 0.5 * (3.0 * (rows == cols).double() - M)
        else:
            rows, cols, M = _kernel(geo)
        Md = torch.zeros((geo.n_sf, geo.n_sf), dtype=torch.float64, device=dev)
        Md[rows, cols] = M
        boxes = _boxes(geo, geo.L, phi, geo.off_L)
        where = {b[2].start: k for k, b in enumerate(boxes)}
        res = [torch.zeros_like(b[3]) for b in boxes]
        for t, meet, i, P in _tiles(boxes, 16, geo.N, 8):
            Z = (Md[i][:, i] @ P).view(-1, 8, 16, 16, 16)
            k = 0
            for b in meet:
                lo, n, fs, _ = boxes[b]
                s = [max(lo[d], t[d]) for d in range(3)]
                e = [min(lo[d] + n[d], t[d] + 16) for d in range(3)]
                dst = tuple(slice(s[d] - lo[d], e[d] - lo[d]) for d in (2, 1, 0))
                src = tuple(slice(int(s[d] - t[d]), int(e[d] - t[d])) for d in (2, 1, 0))
                nf = fs.stop - fs.start
                res[b][(slice(None), slice(None)) + dst] = Z[(slice(k, k + nf), slice(None)) + src]
                k += nf
        out = torch.zeros(int(geo.off_L[-1]), dtype=torch.float64, device=dev)
        for k, fs, D in _each_atom(geo):
            D.store(geo.L[k], res[where[fs.start]], out, geo.off_L)
        return [out]
    if op == "precondition":
        u = torch.tensor(geo.rng.rand(2, geo.n_sf), device=dev)
        a, eps = 2e-3 + 3e-3 * u[0], -0.2 - 0.6 * u[1]
        out = torch.zeros(int(geo.off_L[-1]), dtype=torch.float64, device=dev)
        res = torch.zeros((case["iters"], geo.n_sf), dtype=torch.float64, device=dev)
        for k, fs, D in _each_atom(geo):
            r = -D.load(geo.L[k], phi, geo.off_L)
            lo, n, c, f = geo.L[k]
            mask = torch.zeros((8, n[0] * n[1] * n[2]), dtype=torch.float64, device=dev)
            mask[0, c] = 1.0
            mask[1:, f] = 1.0
            mask = mask.view(r.shape[1:])
            Q, K = D.confinement(r, lo, a[fs]), D.kinetic(n)
            one = (-1,) + (1,) * 6
            x, p = torch.zeros_like(r), r
            rr = (r * r).flatten(1).sum(1)
            for it in range(case["iters"]):
                Ap = (Q(p) + sum(D.along(M, p, d) for d, M in enumerate(K)) - eps[fs].view(one) * p) * mask
                al = (rr / (p * Ap).flatten(1).sum(1)).view(one)
                x, r = x + al * p, r - al * Ap
                new = (r * r).flatten(1).sum(1)
                p = r + (new / rr).view(one) * p
                rr = new
                res[it, fs] = torch.sqrt(new)
            D.store(geo.L[k], x, out, geo.off_L)
        return [out, res if full else None]
    rows, cols, Hm, Sm, top = _matrices(geo)
    n = geo.n_sf
    keep = torch.zeros((n, n), dtype=torch.float64, device=dev)
    keep[rows, cols] = 1.0
    Hd, Sd = torch.zeros_like(keep), torch.zeros_like(keep)
    Hd[rows, cols], Sd[rows, cols] = Hm, Sm
    I = torch.eye(n, dtype=torch.float64, device=dev)
    sigma, terms, de, n_el = 1.0 / top, case["terms"], 0.08 * top, 0.4 * n
    Ht, X = sigma * Hd, 0.5 * (3.0 * I - Sd)
    P = (X @ Ht @ X) * keep
    series = [I, P * keep]
    for _ in range(2, terms + 1):
        series.append((2.0 * (P @ series[-1]) - series[-2]) * keep)
    tr = np.array([float(torch.trace(T)) for T in series])
    th = math.pi * (np.arange(terms + 1) + 0.5) / (terms + 1)
    cosines = np.cos(np.outer(np.arange(terms + 1), th))
    lo, hi = -top, top
    for _ in range(200):
        mu = 0.5 * (lo + hi)
        fx = np.array([0.5 * (1.0 - math.erf((x - sigma * mu) / (sigma * de))) for x in np.cos(th)])
        c = 2.0 / (terms + 1) * (cosines @ fx)
        c[0] *= 0.5
        trace = float(c @ tr)
        if abs(trace - n_el) <= 1e-10:
            break
        lo, hi = (mu, hi) if trace < n_el else (lo, mu)
    Kp = sum(ck * T for ck, T in zip(c, series))
    K = (X @ Kp @ X) * keep
    ebs = float((K * Ht.T).sum()) / sigma
    return [Kp[rows, cols], K[rows, cols], mu, ebs, trace]
