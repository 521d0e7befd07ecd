"""The forms of the backward plane kernel that its rules take only for large systems or large boxes:
items of several functions of an atom, the z arm's plane read in place, no list of fine members.
Forced by option on small systems, where every form has the default's bits; and on boxes that
leave no other choice, against the oracle (FP64 1e-12, FP32 1e-5)."""
import numpy as np
import pytest

from oracle import geometry as G
from paper_1401_7441_gb300 import inputs as I
from paper_1401_7441_gb300 import lsw
from tests.lib_support import ensure_built, gpu_run, keys_to_g
from tests.oracle_support import desc_of
from tests.test_gpu_kernel_edges import TOL, cluster
from tests.test_gpu_parity import check_functions, oracle_hphi, phi_fn

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()


SYSTEMS = {
    # uneven radii; atoms of one and four functions cut by batches of 5
    "uneven": lambda: I.scaled("atoms1200", 9, seed=21),
    # more fine members than the list holds; no fine members; L' far beyond L (planes without L)
    "all_fine": lambda: cluster((13, 11, 12), 3, [7, 1, 3], [20.0], [20.0], 9.0),
    "no_fine": lambda: cluster((15, 14, 17), 3, [6, 2], [1.9], [0.0], 9.0, margin=5.0),
    "long": lambda: cluster((47, 4, 5), 2, [9, 3], [40.0], [2.0], 9.0),
    "wide_margin": lambda: cluster((33, 30, 31), 2, [4, 5], [1.3], [0.6], 9.0, margin=15.0),
}


@pytest.mark.parametrize("prec", [lsw.LSW_FP64, lsw.LSW_FP32])
@pytest.mark.parametrize("name", sorted(SYSTEMS))
def test_forms_have_the_same_bits(name, prec):
    import torch
    wl = SYSTEMS[name]()
    dt = torch.float64 if prec == lsw.LSW_FP64 else torch.float32
    st = torch.cuda.Stream()
    S = lsw.System(wl.N, wl.h, wl.pos, wl.r_loc, wl.r_fine, wl.nsf, wl.pair_cutoff, wl.pair_mode, wl.lprime_margin, 0,
                   prec, device=0, stream=st.cuda_stream)
    try:
        phi = torch.randn(S.total_L, generator=torch.Generator(device="cuda").manual_seed(2), dtype=dt, device="cuda")
        V = torch.tensor(I.potential(wl), dtype=dt, device="cuda")
        lsw.lsw_set_potential(S.sys, V, wl.V_lo, wl.V_shape)
        base = None
        for persistent, batch, layout, groups in ((0, 5, -1, [0]), (0, 64, 0, [0]), (1, 64, 3, [1, 2, 3, 64]),
                                                  (1, 64, 2, [1, 3, 64]), (1, 64, 0, [1, 64]), (1, 5, -1, [2, 64])):
            lsw.lsw_set_option(S.sys, "persistent", persistent)
            lsw.lsw_set_option(S.sys, "batch", batch)
            lsw.lsw_set_option(S.sys, "bwd_layout", layout)
            for group in groups:
                lsw.lsw_set_option(S.sys, "bwd_group", group)
                hphi = torch.full((S.total_Lp,), -7.0, dtype=dt, device="cuda")
                ek = torch.zeros(S.n_sf, dtype=torch.float64, device="cuda")
                torch.cuda.synchronize()
                for _ in range(2):                                # captured, then replayed
                    lsw.lsw_apply_hamiltonian(S.sys, phi, hphi, ek, None)
                lsw.lsw_sync(S.sys, 60.0)
                if base is None:
                    base = hphi, ek
                    assert float(hphi.abs().max()) > 0.0
                form = (persistent, batch, layout, group)
                assert torch.equal(hphi, base[0]), form
                tol = 1e-12 if prec == lsw.LSW_FP64 else 1e-6       # per-thread sums over other tasks
                assert float((ek - base[1]).abs().max()) <= tol * float(base[1].abs().max()), form
    finally:
        S.close()


# L and L' extents along x and y (three planes) at which only these layouts fit
@pytest.mark.parametrize("prec,n,fits", [(lsw.LSW_FP64, 37, [2, 0]), (lsw.LSW_FP32, 57, [0])], ids=["fp64", "fp32"])
def test_boxes_that_leave_no_room(prec, n, fits):
    import torch
    h, N = 0.45, (n + 16, n + 16, 3)
    c = (n + 15) // 2 * h
    wl = I.Workload("flat", N, h, np.array([[c, c, h]]), np.array([(n // 2) * h + 1e-6]), np.array([3.1 * h]),
                    np.array([3]), 4.0, 0, np.array([[c, c, h, 1.5, 0.8], [0.4 * c, c, 0.0, 1.0, 0.6]]), 3)
    S = lsw.System(wl.N, wl.h, wl.pos, wl.r_loc, wl.r_fine, wl.nsf, wl.pair_cutoff, 0, 8.0, 0, prec, device=0,
                   stream=torch.cuda.current_stream().cuda_stream)
    try:
        g = keys_to_g(S.keys(0, lsw.LSW_REGION_L, lsw.LSW_PART_COARSE))
        assert len(set(g % N[0])) == n and len(set(g // N[0] % N[1])) == n
        for layout in (3, 2, 0):
            if layout in fits:
                lsw.lsw_set_option(S.sys, "bwd_layout", layout)
            else:
                with pytest.raises(lsw.LswError) as e:
                    lsw.lsw_set_option(S.sys, "bwd_layout", layout)
                assert e.value.status == lsw.LSW_ERR_UNSUPPORTED
    finally:
        S.close()
    geo = G.build(desc_of(wl))
    ref = oracle_hphi(wl, geo, range(3), I.potential(wl))
    for options in [{}] + [{"bwd_layout": v, "bwd_group": 3} for v in fits]:
        check_functions(wl, geo, gpu_run(wl, phi_fn(wl), prec, options=options), ref, TOL[prec])
