"""Device buffers that calls keep between them: which calls may allocate, how much stays, and
that a buffer a caller's captured graph holds is not moved."""
import numpy as np
import pytest

from oracle import foe as F
from paper_1401_7441_gb300 import lsw
from tests.lib_support import ensure_built
from tests.test_gpu_kernel_edges import cluster

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()


def _conf_case(prec, stream, n_atoms=3, n_sf=2, seed=11):
    import torch
    rng = np.random.default_rng(seed)
    N, h = (23, 21, 22), 0.5
    S = lsw.System(N, h, rng.uniform(3.0, 7.0, (n_atoms, 3)), np.full(n_atoms, 2.6), np.full(n_atoms, 1.1),
                   np.full(n_atoms, n_sf), 4.0, 0, 8.0, 0, prec, device=0, stream=stream)
    dt = torch.float64 if prec == lsw.LSW_FP64 else torch.float32
    phi = torch.tensor(rng.standard_normal(S.total_L), dtype=dt, device="cuda")
    a = torch.tensor(rng.uniform(0.001, 0.01, S.n_sf), device="cuda")
    eps = torch.tensor(-rng.uniform(0.3, 1.0, S.n_sf), device="cuda")
    return S, phi, a, eps


@pytest.mark.parametrize("prec", [lsw.LSW_FP64, lsw.LSW_FP32])
def test_confinement_and_preconditioner_share_one_buffer(prec):
    # a program that has called one of the two may capture the other, and graphs that hold the
    # buffer's address stay valid: the second kind of call allocates nothing
    import torch
    st = torch.cuda.Stream()
    S, phi, a, eps = _conf_case(prec, st.cuda_stream)
    try:
        gp = torch.zeros_like(phi)
        hphi = torch.zeros(S.total_Lp, dtype=phi.dtype, device="cuda")
        torch.cuda.synchronize()
        lsw.lsw_precondition(S.sys, a, eps, phi, gp, 2, None)
        lsw.lsw_sync(S.sys, 60.0)
        first = gp.clone()
        held = lsw.lsw_workspace_bytes(S.sys)
        g = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(g, stream=st, capture_error_mode="thread_local"):
            lsw.lsw_precondition(S.sys, a, eps, phi, gp, 2, None)
            lsw.lsw_add_confinement(S.sys, a, phi, hphi, None)
        assert lsw.lsw_workspace_bytes(S.sys) == held
        direct = torch.zeros_like(hphi)
        torch.cuda.synchronize()
        lsw.lsw_add_confinement(S.sys, a, phi, direct, None)
        lsw.lsw_sync(S.sys, 60.0)
        gp.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(gp, first)
        assert torch.equal(hphi, direct) and float(direct.abs().max()) > 0.0
        assert lsw.lsw_workspace_bytes(S.sys) == held
        del g
    finally:
        S.close()


def _foe_system(n_atoms, nsf):
    import torch
    wl = cluster((12, 11, 12), n_atoms, nsf, [1.2], [0.6], 3.0)
    S = lsw.System(wl.N, wl.h, wl.pos, wl.r_loc, wl.r_fine, wl.nsf, wl.pair_cutoff, wl.pair_mode, wl.lprime_margin, 0,
                   lsw.LSW_FP64, device=0, stream=torch.cuda.current_stream().cuda_stream)
    n = S.n_sf
    rows = np.repeat(np.arange(n), np.diff(S.row_ptr))
    mask = np.zeros((n, n), bool)
    mask[rows, S.col] = True
    rng = np.random.default_rng(17)
    A, B = rng.standard_normal((2, n, n))
    H = np.where(mask, (A + A.T) / np.sqrt(8.0 * n), 0.0)
    O = np.where(mask, (B + B.T) * 0.1 / np.sqrt(8.0 * n), 0.0) + np.eye(n)
    return S, H, O, mask, rows


@pytest.mark.parametrize("n_pl", [1, 2, 3, 4, 31])
def test_fermi_expansion_with_and_without_kept_matrices(n_pl):
    # the two ways of summing K': from the kept T_j, or with the recursion run twice over three slots
    import torch
    S, H, O, mask, rows = _foe_system(6, [5, 2, 1])
    try:
        bounds = F.spectrum_bounds(H, O)
        n_el = float(S.n_sf // 2)
        ref = F.foe(H, O, n_el, n_pl, 0.1, sinv="taylor", bounds=bounds, pattern=mask)
        Hv, Sv = (torch.tensor(m[rows, S.col], device="cuda") for m in (H, O))
        for keep in (4096, 0, 1):
            lsw.lsw_set_option(S.sys, "foe_keep_mb", keep)
            Kp = torch.zeros(len(S.col), dtype=torch.float64, device="cuda")
            K = torch.zeros_like(Kp)
            mu, ebs, tr = lsw.lsw_foe(S.sys, Hv, Sv, bounds[0], bounds[1], n_el, n_pl, 0.1, Kp, K)
            assert mu == pytest.approx(ref["mu"], abs=1e-12 * (bounds[1] - bounds[0])), keep
            for got, want in ((Kp, ref["Kp"]), (K, ref["K"])):
                want = want[rows, S.col]
                assert np.max(np.abs(got.cpu().numpy() - want)) <= 1e-11 * np.max(np.abs(want)), keep
            assert ebs == pytest.approx(ref["E_BS"], rel=1e-11, abs=1e-11), keep
        for bad in (-1, 1 << 23):
            with pytest.raises(lsw.LswError):
                lsw.lsw_set_option(S.sys, "foe_keep_mb", bad)
    finally:
        S.close()


def test_fermi_expansion_gives_its_matrices_back():
    # 512 functions: the 300 T_j of a call take 450 MB, of which 256 MiB may stay
    import torch
    S, H, O, mask, rows = _foe_system(8, [64])
    try:
        assert len(S.col) * 300 * 8 > (400 << 20)
        Hv, Sv = (torch.tensor(m[rows, S.col], device="cuda") for m in (H, O))
        Kp = torch.zeros(len(S.col), dtype=torch.float64, device="cuda")
        K = torch.zeros_like(Kp)
        lsw.lsw_set_option(S.sys, "foe_keep_mb", 0)
        lsw.lsw_foe(S.sys, Hv, Sv, -4.0, 4.0, 100.0, 300, 0.2, Kp, K)      # the other work buffers
        first = K.clone()
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        lsw.lsw_set_option(S.sys, "foe_keep_mb", 4096)
        for _ in range(3):
            lsw.lsw_foe(S.sys, Hv, Sv, -4.0, 4.0, 100.0, 300, 0.2, Kp, K)
            torch.cuda.synchronize()
            assert free - torch.cuda.mem_get_info()[0] <= (256 << 20) + (8 << 20)
            assert float((K - first).abs().max()) <= 1e-11 * float(first.abs().max())
    finally:
        S.close()
