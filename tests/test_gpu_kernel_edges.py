"""Sizes at which the kernels' splits change: atoms with many functions (cut by the 32-function
chunks of the density, by the 128 coefficients a combination keeps, by the outputs of a
pair's expansion), more functions and atoms on a tile than the density's tables hold, pairs
outside the pattern, boxes that are long in one direction and a few points wide in the
others.  Against the oracles, element by element, at the tolerances of the paths (FP64 1e-12,
FP32 1e-5 of the absolute-term bound; 1e-11 of the largest entry for the expansion)."""
import numpy as np
import pytest

from oracle import density as Dn
from oracle import foe as F
from oracle import geometry as G
from paper_1401_7441_gb300 import inputs as I
from paper_1401_7441_gb300 import lsw
from tests.lib_support import ensure_built, gpu_density, gpu_run
from tests.oracle_support import desc_of, phi_all
from tests.test_gpu_combine import _check, _phi, _run, _system
from tests.test_gpu_parity import check_functions, check_rows, oracle_hphi, phi_fn

pytestmark = pytest.mark.gpu

TOL = {lsw.LSW_FP64: 1e-12, lsw.LSW_FP32: 1e-5}
FLOOR = {lsw.LSW_FP64: 0.0, lsw.LSW_FP32: 1e-34}


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()


def cluster(N, n_atoms, nsf, r_loc, r_fine, cutoff, h=0.45, seed=31, margin=8.0):
    """Atoms at seeded places of a small box, `nsf` repeated over them."""
    u = I.uniform(seed, 9, 5 * n_atoms).reshape(-1)
    pos = (1.0 + u[:3 * n_atoms].reshape(n_atoms, 3) * (np.array(N) - 2.5)) * h
    wells = np.column_stack([pos[:8], 1.0 + 2.0 * u[3 * n_atoms:][:len(pos[:8])], 0.5 + u[4 * n_atoms:][:len(pos[:8])]])
    return I.Workload("cluster", tuple(N), h, pos, np.resize(r_loc, n_atoms).astype(float),
                      np.resize(r_fine, n_atoms).astype(float), np.resize(nsf, n_atoms).astype(np.int64), cutoff, 0, wells,
                      seed, lprime_margin=margin)


MANY_ATOMS = dict(N=(9, 9, 8), n_atoms=150, nsf=[1], r_loc=[1.0, 1.2], r_fine=[0.6], cutoff=1.3)
MANY_FUNCTIONS = dict(N=(9, 8, 9), n_atoms=48, nsf=[1, 4, 3, 9], r_loc=[1.1, 0.9, 1.3], r_fine=[0.6, 0.0], cutoff=1.5)


@pytest.mark.parametrize("prec", [lsw.LSW_FP64, lsw.LSW_FP32])
@pytest.mark.parametrize("shape", [MANY_ATOMS, MANY_FUNCTIONS], ids=["many_atoms", "many_functions"])
def test_density_crowded_tiles(prec, shape):
    wl = cluster(**shape)
    K_of = lambda rp, col, sa: np.random.default_rng(3).uniform(-1.0, 1.0, len(col))
    gpu = gpu_density(wl, prec, kernel=K_of)
    geo = G.build(desc_of(wl))
    assert len(gpu["col"]) < 0.7 * wl.n_sf ** 2               # pairs outside the pattern
    phi = phi_all(wl, geo)
    rho = Dn.density(geo, phi, gpu["K"], wl.V_lo, wl.V_shape)
    bound = Dn.density(geo, phi, gpu["K"], wl.V_lo, wl.V_shape, absolute=True)
    got = gpu["rho"][0]
    assert np.all(np.abs(got - rho) <= TOL[prec] * bound + FLOOR[prec])
    assert np.all(got[bound == 0] == 0)


# tiles of at most 8 functions (one block of coefficients), 9 to 16 (FP32: another width), 17 (tables)
@pytest.mark.parametrize("prec", [lsw.LSW_FP64, lsw.LSW_FP32])
@pytest.mark.parametrize("nsf", [[1], [8], [9], [16], [17], [2, 5]], ids=lambda v: "-".join(map(str, v)))
def test_density_few_functions(prec, nsf):
    wl = cluster((8, 9, 7), len(nsf), nsf, [1.6, 1.1], [0.8, 0.5], 0.9 if len(nsf) > 1 else 5.0)
    gpu = gpu_density(wl, prec, kernel=lambda rp, col, sa: np.random.default_rng(4).uniform(-1.0, 1.0, len(col)))
    geo = G.build(desc_of(wl))
    phi = phi_all(wl, geo)
    rho = Dn.density(geo, phi, gpu["K"], wl.V_lo, wl.V_shape)
    bound = Dn.density(geo, phi, gpu["K"], wl.V_lo, wl.V_shape, absolute=True)
    assert np.all(np.abs(gpu["rho"][0] - rho) <= TOL[prec] * bound + FLOOR[prec])
    assert np.all(gpu["rho"][0][bound == 0] == 0)


@pytest.mark.parametrize("prec", [lsw.LSW_FP64, lsw.LSW_FP32])
@pytest.mark.parametrize("tile", [0, 2, 5])
def test_matrices_and_combination_many_functions_per_tile(prec, tile):
    wl = cluster(**MANY_FUNCTIONS)
    geo = G.build(desc_of(wl))
    rows = [0, 1, 5, 8, 17, 100, wl.n_sf - 1]
    options = {"tile": tile} if tile else {}
    gpu = gpu_run(wl, phi_fn(wl), prec, options=options)
    ref = oracle_hphi(wl, geo, rows, I.potential(wl))
    check_functions(wl, geo, gpu, ref, TOL[prec])
    check_rows(wl, geo, gpu, ref, rows, TOL[prec], h_cols=set(rows))
    S = _system(wl, prec, options)
    try:
        M_v = np.random.default_rng(5).uniform(-1.0, 1.0, len(S.col))
        got, phi_in = _run(S, prec, _phi(wl, S), M_v)
        _check(S, geo, got, M_v, phi_in, rows, prec)
    finally:
        S.close()


BOXES = {
    # N, atoms, functions per atom, r_loc, r_fine, margin
    "long_x": ((61, 3, 4), 2, [9, 2], [40.0], [2.0], 8.0),
    "long_y": ((3, 58, 4), 2, [3, 1], [40.0], [3.0], 8.0),
    "long_z": ((4, 3, 63), 2, [2, 1], [40.0], [2.5], 8.0),
    "few_points": ((12, 11, 13), 2, [1, 2], [0.4], [0.1], 8.0),
    "no_fine": ((13, 12, 11), 2, [2, 1], [1.6], [0.0], 8.0),
    "all_fine_margin_zero": ((9, 7, 8), 2, [3, 2], [20.0], [20.0], 0.0),
    "clipped_wide_margin": ((19, 14, 16), 2, [5, 1], [2.2, 1.4], [0.9], 16.0),
}


@pytest.mark.parametrize("prec", [lsw.LSW_FP64, lsw.LSW_FP32])
@pytest.mark.parametrize("name", sorted(BOXES))
def test_hamiltonian_box_shapes(prec, name):
    N, n_atoms, nsf, r_loc, r_fine, margin = BOXES[name]
    wl = cluster(N, n_atoms, nsf, r_loc, r_fine, 100.0, margin=margin)
    geo = G.build(desc_of(wl))
    gpu = gpu_run(wl, phi_fn(wl), prec)
    check_functions(wl, geo, gpu, oracle_hphi(wl, geo, range(wl.n_sf), I.potential(wl)), TOL[prec])


# 8 atoms of 64: a row block of X A X no longer fits in shared memory
@pytest.mark.parametrize("n_atoms,nsf,n_pl", [(6, [64, 1], 30), (6, [33, 2, 9], 30), (6, [1], 30), (8, [64], 8)])
def test_fermi_expansion_functions_per_atom(n_atoms, nsf, n_pl):
    import torch
    wl = cluster((12, 11, 12), n_atoms, nsf, [1.2], [0.6], 3.0)
    S = lsw.System(wl.N, wl.h, wl.pos, wl.r_loc, wl.r_fine, wl.nsf, wl.pair_cutoff, wl.pair_mode, wl.lprime_margin, 0,
                   lsw.LSW_FP64, device=0, stream=torch.cuda.current_stream().cuda_stream)
    try:
        n = S.n_sf
        rows = np.repeat(np.arange(n), np.diff(S.row_ptr))
        mask = np.zeros((n, n), bool)
        mask[rows, S.col] = True
        rng = np.random.default_rng(17)
        A, B = rng.standard_normal((2, n, n))
        Hd = np.where(mask, (A + A.T) / np.sqrt(8.0 * n), 0.0)
        Sd = np.where(mask, (B + B.T) * 0.1 / np.sqrt(8.0 * n), 0.0) + np.eye(n)
        bounds = F.spectrum_bounds(Hd, Sd)
        n_el = float(max(1, n // 2))
        ref = F.foe(Hd, Sd, n_el, n_pl, 0.1, sinv="taylor", bounds=bounds, pattern=mask)
        Hv, Sv = (torch.tensor(m[rows, S.col], device="cuda") for m in (Hd, Sd))
        Kp = torch.zeros(len(S.col), dtype=torch.float64, device="cuda")
        K = torch.zeros_like(Kp)
        mu, ebs, tr = lsw.lsw_foe(S.sys, Hv, Sv, bounds[0], bounds[1], n_el, n_pl, 0.1, Kp, K)
        assert mu == pytest.approx(ref["mu"], abs=1e-12 * (bounds[1] - bounds[0]))
        for got, want in ((Kp, ref["Kp"]), (K, ref["K"])):
            want = want[rows, S.col]
            assert np.max(np.abs(got.cpu().numpy() - want)) <= 1e-11 * np.max(np.abs(want))
        assert ebs == pytest.approx(ref["E_BS"], rel=1e-11, abs=1e-11)
    finally:
        S.close()
