"""The tiled operator apply (csrc/apply.cu) against the oracle's matrix at the edges of its tiling: a panel row held by one
thread, rows that are no multiple of a thread's 16 bytes, one and several tiles a panel, chunks that end at the wall, and
vectors that are not 16-byte aligned (the scalar path)."""
import numpy as np
import pytest

from oracle.discrete import Discretization, ppbe_matrix, vtbe_matrix
from oracle.grid import Grid

pytestmark = pytest.mark.gpu

PH = dict(E=1e-3, Ra=100.0, Pr=1.0, Pm=5.0, dt=1e-4)


@pytest.mark.parametrize('kind', [0, 1])
@pytest.mark.parametrize('Ns,Nr', [(4, 2), (5, 3), (12, 7), (17, 2), (36, 5), (65, 3)])
def test_apply_at_tile_edges(kind, Ns, Nr):
    import torch

    from paper_2009_02171_gb300 import fv
    d = Discretization(Grid(Ns, Nr))
    A = vtbe_matrix(d, **PH) if kind == 0 else ppbe_matrix(d, PH['E'], PH['dt'])
    g = fv.fv_build_grid(Ns, Nr)
    n = A.shape[0]
    x = np.random.default_rng(11).standard_normal(n)
    ref = A @ x
    for prec, dtype, bar in ((0, torch.float64, 1e-12), (1, torch.float32, 2e-5)):
        s = fv.fv_assemble_system(g, kind, **PH, precision=prec, inner_maxit=2)
        f = fv.fv_apply_op if prec == 0 else fv.fv_apply_op_fp32
        for shift in (0, 1):  # shift 1: no vector is 16-byte aligned
            xd = torch.zeros(n + 1, dtype=dtype, device='cuda')[shift:shift + n]
            xd.copy_(torch.tensor(x))
            y = f(s, xd, torch.empty(n + 1, dtype=dtype, device='cuda')[shift:shift + n]).cpu().numpy()
            assert np.abs(y - ref).max() <= bar * np.abs(ref).max(), (prec, shift)
        fv.fv_free_system(s)
    fv.fv_free_grid(g)
