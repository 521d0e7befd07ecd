"""Confinement and preconditioning on the region shapes where the pass kernels can go wrong:
locregs clipped by the box, an output region equal to L or wider than the filters' reach, no
fine members, more functions than one packed group of lines, lines too long for shared
memory.  Against the oracle (oracle/confinement.py); FP64 1e-12 of the largest element, FP32
1e-5 (the precisions' tolerances), the preconditioner's iterate 1e-11 after two iterations
(FP64: two operator applications and dot products)."""
import numpy as np
import pytest

from oracle import confinement as Q
from oracle import geometry as G
from paper_1401_7441_gb300 import lsw
from tests.lib_support import ensure_built

pytestmark = pytest.mark.gpu

H = 0.5
CASES = {
    # name: (N, positions, r_loc, r_fine, n_sf, margin)
    "clipped": ((17, 13, 15), [[0.3, 0.2, 0.4], [7.0, 5.5, 6.6]], [2.6, 3.1], [1.2, 0.9], [2, 1], 8.0),
    "margin_zero": ((19, 18, 17), [[4.1, 4.4, 4.2]], [3.0], [1.4], [3], 0.0),
    "wide_margin": ((41, 39, 40), [[9.9, 9.6, 10.1]], [1.3], [0.8], [2], 17.0),
    "no_fine": ((20, 20, 20), [[4.87, 5.13, 4.91]], [2.9], [0.0], [1], 8.0),
    "one_point": ((16, 16, 16), [[4.0, 4.0, 4.0]], [0.1], [0.1], [1], 8.0),
    "all_fine": ((18, 14, 16), [[4.0, 3.5, 4.0]], [50.0], [50.0], [2], 8.0),
    "long_lines": ((230, 3, 4), [[57.0, 0.5, 0.9]], [80.0], [3.0], [1], 8.0),
}


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()


@pytest.mark.parametrize("prec", [lsw.LSW_FP64, lsw.LSW_FP32])
@pytest.mark.parametrize("name", sorted(CASES))
def test_confinement_and_preconditioner_edges(name, prec):
    import torch
    N, pos, rl, rf, nsf, margin = CASES[name]
    S = lsw.System(N, H, np.array(pos), np.array(rl), np.array(rf), np.array(nsf), 4.0, 0, margin, 0, prec, device=0,
                   stream=torch.cuda.current_stream().cuda_stream)
    try:
        geo = G.build(G.SystemDesc(N, H, np.array(pos), np.array(rl), np.array(rf), np.array(nsf), 4.0, 0,
                                   lprime_margin=margin))
        dt, tol = (torch.float64, 1e-12) if prec == lsw.LSW_FP64 else (torch.float32, 1e-5)
        rng = np.random.default_rng(11)
        phi = torch.tensor(rng.standard_normal(S.total_L), dtype=dt, device="cuda")
        a_h, eps_h = rng.uniform(0.001, 0.01, S.n_sf), -rng.uniform(0.3, 1.0, S.n_sf)
        a, eps = torch.tensor(a_h, device="cuda"), torch.tensor(eps_h, device="cuda")
        base = torch.tensor(rng.standard_normal(S.total_Lp), dtype=dt, device="cuda")
        hphi, e = base.clone(), torch.zeros(S.n_sf, dtype=torch.float64, device="cuda")
        lsw.lsw_add_confinement(S.sys, a, phi, hphi, e)
        gp = torch.zeros_like(phi)
        lsw.lsw_precondition(S.sys, a, eps, phi, gp, 2, None)
        lsw.lsw_sync(S.sys, 60.0)
        pin, got, b, x = (t.double().cpu().numpy() for t in (phi, hphi, base, gp))
        for f in range(S.n_sf):
            n = geo.L[geo.sf_atom[f]].n_coef
            pf = pin[S.off_L[f]:S.off_L[f] + n]
            ref, e_ref = Q.confinement_energy_and_action(geo, f, pf, a_h[f])
            at = slice(S.off_Lp[f], S.off_Lp[f] + len(ref))
            scale = max(np.max(np.abs(ref)), np.max(np.abs(b[at])))
            assert np.max(np.abs(got[at] - b[at] - ref)) <= tol * scale, (name, f)
            assert abs(e[f].item() - e_ref) <= tol * abs(e_ref), (name, f)
            if prec == lsw.LSW_FP64:
                xr, _ = Q.precondition(geo, f, pf, a_h[f], eps_h[f], 2)
                assert np.linalg.norm(x[S.off_L[f]:S.off_L[f] + n] - xr) <= 1e-11 * np.linalg.norm(xr), (name, f)
    finally:
        S.close()


@pytest.mark.parametrize("prec", [lsw.LSW_FP64, lsw.LSW_FP32])
def test_confinement_energy_same_bits_on_every_call(prec):
    # hundreds of rows per function: partial sums added in the order they finish would differ
    import torch
    N, n_sf = (41, 39, 40), 6
    S = lsw.System(N, H, np.array([[9.7, 9.6, 10.1]]), np.array([6.0]), np.array([2.2]), np.array([n_sf]), 4.0, 0, 8.0, 0,
                   prec, device=0, stream=torch.cuda.current_stream().cuda_stream)
    try:
        dt = torch.float64 if prec == lsw.LSW_FP64 else torch.float32
        rng = np.random.default_rng(7)
        phi = torch.tensor(rng.standard_normal(S.total_L), dtype=dt, device="cuda")
        a = torch.tensor(rng.uniform(0.001, 0.01, n_sf), device="cuda")
        hphi = torch.zeros(S.total_Lp, dtype=dt, device="cuda")
        runs = []
        for _ in range(12):
            e = torch.full((n_sf,), float("nan"), dtype=torch.float64, device="cuda")
            lsw.lsw_add_confinement(S.sys, a, phi, hphi, e)
            lsw.lsw_sync(S.sys, 60.0)
            runs.append(e.cpu().numpy())
        assert np.all(np.isfinite(runs[0])) and np.all(runs[0] > 0)
        assert all(np.array_equal(runs[0], r) for r in runs[1:])
    finally:
        S.close()


def test_confinement_of_one_coefficient_is_the_tables_entry_by_entry():
    # phi = one coefficient at the end of L along a dimension, a = 1: H phi on the line through it
    # holds X^4 and the two cross terms' X^2 entries of that dimension, over the whole band
    import torch
    N, h = (44, 43, 45), 0.5
    pos = np.array([[10.37, 10.81, 11.13]])
    S = lsw.System(N, h, pos, np.array([2.6]), np.array([50.0]), np.array([1]), 4.0, 0, 17.0, 0, lsw.LSW_FP64, device=0,
                   stream=torch.cuda.current_stream().cuda_stream)
    try:
        def members(region, part):
            k = S.keys(0, region, part)
            return np.concatenate([np.arange(s, e + 1) for s, e, _ in k])

        Lc, Lf = members(lsw.LSW_REGION_L, lsw.LSW_PART_COARSE), members(lsw.LSW_REGION_L, lsw.LSW_PART_FINE)
        Pc, Pf = members(lsw.LSW_REGION_LP, lsw.LSW_PART_COARSE), members(lsw.LSW_REGION_LP, lsw.LSW_PART_FINE)
        assert np.array_equal(Lc, Lf) and np.array_equal(Pc, Pf)          # fine everywhere
        row = lambda d, m, b, bp, i: lsw.lsw_confinement_row(S.sys, 0, d, m, b, bp, int(i))
        stride = (1, N[0], N[0] * N[1])
        ijk = np.stack([Lc % N[0], Lc // N[0] % N[1], Lc // (N[0] * N[1])], 1)
        mid = np.round(pos[0] / h).astype(int)
        a = torch.ones(1, dtype=torch.float64, device="cuda")
        for d in range(3):
            o = [e for e in range(3) if e != d]
            line = ijk[(ijk[:, o[0]] == mid[o[0]]) & (ijk[:, o[1]] == mid[o[1]])][:, d]
            diag = sum(row(e, 2, 0, 0, mid[e])[14] for e in o)            # <s|X_e^2|s> of the other dimensions
            for j in (line.min(), line.max()):
                g = int(mid[o[0]] * stride[o[0]] + mid[o[1]] * stride[o[1]] + j * stride[d])
                for bp in (0, 1):
                    phi = torch.zeros(S.total_L, dtype=torch.float64, device="cuda")
                    at = int(np.searchsorted(Lc, g))
                    phi[at if bp == 0 else len(Lc) + ((1 << d) - 1) * len(Lf) + at] = 1.0
                    hphi = torch.zeros(S.total_Lp, dtype=torch.float64, device="cuda")
                    lsw.lsw_add_confinement(S.sys, a, phi, hphi, None)
                    lsw.lsw_sync(S.sys, 60.0)
                    out = hphi.cpu().numpy()
                    for b in (0, 1):
                        got, want = [], []
                        for i in range(j - 14, j + 15):
                            p = int(np.searchsorted(Pc, g + (i - j) * stride[d]))
                            assert Pc[p] == g + (i - j) * stride[d]
                            got.append(out[p if b == 0 else len(Pc) + ((1 << d) - 1) * len(Pf) + p])
                            want.append(row(d, 4, b, bp, i)[14 + j - i] + 2.0 * diag * row(d, 2, b, bp, i)[14 + j - i]
                                        + (sum(row(e, 4, 0, 0, mid[e])[14] for e in o)
                                           + 2.0 * row(o[0], 2, 0, 0, mid[o[0]])[14] * row(o[1], 2, 0, 0, mid[o[1]])[14])
                                        * (i == j and b == bp))
                        got, want = np.array(got), np.array(want)
                        assert np.all(np.abs(got - want) <= 1e-13 * np.max(np.abs(want))), (d, j, bp, b)
    finally:
        S.close()
