"""The one-launch Gram-Schmidt step (csrc/krylov.cu) at its edges: vectors of one block, vectors whose length is no multiple of
a 16-byte load, a ragged last slice, more basis vectors than a block's 512 threads keep in registers.  The stopping rule is on
the true FP64 residual, so a solve that reports convergence must satisfy the oracle's matrix to the tolerance."""
import numpy as np
import pytest

from oracle.discrete import Discretization, ppbe_matrix, vtbe_matrix
from oracle.grid import Grid

pytestmark = pytest.mark.gpu

PH = dict(E=1e-3, Ra=100.0, Pr=1.0, Pm=5.0, dt=1e-4)


@pytest.mark.parametrize('kind,Ns,Nr,prec,restart', [
    (1, 4, 2, 0, 5),     # 384 values: one block
    (0, 9, 7, 1, 30),    # FP32 vectors of 23,814 values: no 16-byte loads
    (0, 9, 7, 0, 30),
    (1, 13, 11, 0, 31),  # up to 31 basis vectors: 256 threads a block
    (1, 24, 12, 1, 30)])
def test_solves_reach_the_true_residual(kind, Ns, Nr, prec, restart):
    import torch

    from paper_2009_02171_gb300 import fv
    d = Discretization(Grid(Ns, Nr))
    A = vtbe_matrix(d, **PH) if kind == 0 else ppbe_matrix(d, PH['E'], PH['dt'])
    g = fv.fv_build_grid(Ns, Nr)
    s = fv.fv_assemble_system(g, kind, **PH, p=(2, 2, 1), overlap=1, precision=prec, inner_maxit=6)
    b = A @ np.random.default_rng(5).standard_normal(A.shape[0])
    x = torch.zeros(b.size, dtype=torch.float64, device='cuda')
    st = fv.fv_gmres_solve(s, torch.tensor(b, device='cuda'), x, restart=restart, rtol=1e-9)
    assert st.converged and st.iters > 1
    res = np.linalg.norm(b - A @ x.cpu().numpy()) / np.linalg.norm(b)
    assert res <= 1.01e-9, res
    fv.fv_free_system(s)
    fv.fv_free_grid(g)
