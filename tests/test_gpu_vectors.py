"""Vector kernels that move 16 bytes at a time, where they cannot: prolongation to rows whose length is no multiple of four or
from an odd address (copies, so equal to the last bit), solves whose vectors start 8 bytes off a 16-byte boundary (the stopping
rule is on the true FP64 residual, so the oracle's matrix must agree to the tolerance)."""
import numpy as np
import pytest

from oracle.discrete import Discretization, ppbe_matrix
from oracle.grid import Grid

pytestmark = pytest.mark.gpu

PH = dict(E=1e-3, Ra=100.0, Pr=1.0, Pm=5.0, dt=1e-4)


@pytest.mark.parametrize('kind', [0, 1])
@pytest.mark.parametrize('Ns,Nr', [(8, 4), (10, 6), (36, 4)])
@pytest.mark.parametrize('off', [0, 1])
def test_prolongation_copies(kind, Ns, Nr, off):
    import torch

    from paper_2009_02171_gb300 import fv
    d = 7 if kind == 0 else 2
    g = fv.fv_build_grid(Ns, Nr)
    s = fv.fv_assemble_system(g, kind, **PH, p=(2, 2, 1), overlap=1, levels=2, coarse_maxit=2)
    xc = np.random.default_rng(3).standard_normal((d, 6, Nr // 2, Ns // 2, Ns // 2))
    x = torch.full((d * 6 * Nr * Ns * Ns + 2,), np.nan, dtype=torch.float64, device='cuda')
    fv.fv_prolong_coarse(s, torch.tensor(xc.ravel(), device='cuda'), x[off:])
    got = x.cpu().numpy()
    np.testing.assert_array_equal(got[off:x.numel() - 2 + off], xc.repeat(2, 2).repeat(2, 3).repeat(2, 4).ravel())
    assert np.isnan(np.delete(got, np.s_[off:x.numel() - 2 + off])).all()
    fv.fv_free_system(s)
    fv.fv_free_grid(g)


@pytest.mark.parametrize('Ns,Nr,prec', [(8, 4, 0), (8, 4, 1), (9, 3, 1)])
def test_solve_from_odd_addresses(Ns, Nr, prec):
    import torch

    from paper_2009_02171_gb300 import fv
    A = ppbe_matrix(Discretization(Grid(Ns, Nr)), PH['E'], PH['dt'])
    g = fv.fv_build_grid(Ns, Nr)
    s = fv.fv_assemble_system(g, 1, **PH, p=(2, 2, 1), overlap=1, precision=prec, inner_maxit=6)
    b = A @ np.random.default_rng(5).standard_normal(A.shape[0])
    bd = torch.zeros(b.size + 1, dtype=torch.float64, device='cuda')
    bd[1:] = torch.tensor(b, device='cuda')
    x = torch.zeros(b.size + 1, dtype=torch.float64, device='cuda')
    st = fv.fv_gmres_solve(s, bd[1:], x[1:], restart=30, rtol=1e-9)
    assert st.converged and st.iters > 1
    res = np.linalg.norm(b - A @ x[1:].cpu().numpy()) / np.linalg.norm(b)
    assert res <= 1.01e-9, res
    fv.fv_free_system(s)
    fv.fv_free_grid(g)
