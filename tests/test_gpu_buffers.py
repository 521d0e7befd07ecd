"""Device buffers that calls keep between them: which calls may allocate, how much stays, and
that a buffer a caller's captured graph holds is not moved."""
import numpy as np
import pytest

from paper_1401_7441_gb300 import lsw
from tests.lib_support import ensure_built

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
