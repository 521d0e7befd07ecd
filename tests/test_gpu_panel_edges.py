"""H/S panels and the sparse combination where their forms change: tile edges 2 and 3 (a lane holds
a point of each part) against larger ones, tiles of so few functions that every coefficient is
looked up by itself, of more than a CTA holds, items of one and of many blocks of panel entries.
Against the oracle at the paths' tolerances (FP64 1e-12, FP32 1e-5), and between tile edges: a
member's sum runs over the same functions in the same order whatever the tile, so the
combination's bits do not depend on it."""
import numpy as np
import pytest

from oracle import geometry as G
from paper_1401_7441_gb300 import inputs as I
from paper_1401_7441_gb300 import lsw
from tests.lib_support import ensure_built, gpu_run
from tests.oracle_support import desc_of
from tests.test_gpu_combine import _check, _phi, _run, _system
from tests.test_gpu_kernel_edges import MANY_FUNCTIONS, TOL, cluster
from tests.test_gpu_parity import check_functions, check_rows, oracle_hphi, phi_fn

pytestmark = pytest.mark.gpu

SHAPES = {
    # two atoms apart: tiles of one or three functions; all fine / no fine members
    "few": dict(N=(15, 12, 13), n_atoms=2, nsf=[1, 3], r_loc=[2.0], r_fine=[1.0], cutoff=9.0),
    "all_fine": dict(N=(9, 7, 8), n_atoms=3, nsf=[5, 1, 2], r_loc=[20.0], r_fine=[20.0], cutoff=9.0),
    "no_fine": dict(N=(10, 11, 7), n_atoms=4, nsf=[6], r_loc=[1.7], r_fine=[0.0], cutoff=2.0),
    "many": MANY_FUNCTIONS,
}


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()


@pytest.mark.parametrize("prec", [lsw.LSW_FP64, lsw.LSW_FP32])
@pytest.mark.parametrize("tile", [2, 3, 4, 8])
@pytest.mark.parametrize("name", sorted(SHAPES))
def test_matrices_and_combination_by_tile_edge(name, tile, prec):
    wl = cluster(**SHAPES[name])
    geo = G.build(desc_of(wl))
    rows = sorted({0, 1, wl.n_sf // 2, wl.n_sf - 1})
    gpu = gpu_run(wl, phi_fn(wl), prec, options={"tile": tile})
    ref = oracle_hphi(wl, geo, rows, I.potential(wl))
    check_functions(wl, geo, gpu, ref, TOL[prec])
    check_rows(wl, geo, gpu, ref, rows, TOL[prec], h_cols=set(rows))
    S = _system(wl, prec, {"tile": tile})
    try:
        M_v = np.random.default_rng(5).uniform(-1.0, 1.0, len(S.col))
        got, phi_in = _run(S, prec, _phi(wl, S), M_v)
        _check(S, geo, got, M_v, phi_in, rows, prec)
    finally:
        S.close()


@pytest.mark.parametrize("prec,n_atoms", [(lsw.LSW_FP64, 60), (lsw.LSW_FP32, 250)])
def test_combination_same_bits_for_every_tile_edge(prec, n_atoms):
    import torch
    wl = I.scaled("atoms10k", n_atoms, seed=9)
    dt = torch.float64 if prec == lsw.LSW_FP64 else torch.float32
    S = lsw.System(wl.N, wl.h, wl.pos, wl.r_loc, wl.r_fine, wl.nsf, wl.pair_cutoff, wl.pair_mode, wl.lprime_margin, 0,
                   prec, device=0, stream=torch.cuda.current_stream().cuda_stream)
    try:
        gen = torch.Generator(device="cuda").manual_seed(3)
        phi = torch.randn(S.total_L, generator=gen, dtype=dt, device="cuda")
        M = torch.rand(len(S.col), generator=gen, dtype=torch.float64, device="cuda") - 0.5
        outs = []
        for tile in (8, 3, 6, 5, 2):
            lsw.lsw_set_option(S.sys, "tile", tile)
            out = torch.zeros_like(phi)
            lsw.lsw_combine(S.sys, M, phi, out)
            lsw.lsw_sync(S.sys, 60.0)
            outs.append(out)
        assert float(outs[0].abs().max()) > 0.0
        for out in outs[1:]:
            assert torch.equal(out, outs[0])
    finally:
        S.close()
