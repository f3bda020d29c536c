"""Streamed subdomain sweeps (csrc/sweep.cu) against the oracle's ILU(0) solves at the edges of their scheme: a window of
rows of one warp, of the most a CTA takes and of more (the general sweeps take over), boxes of one layer, steps that
straddle operand chunks, uneven boxes whose tables differ, forward results in shared and in global memory."""
import numpy as np
import pytest

from oracle.discrete import Discretization, ppbe_matrix, vtbe_matrix
from oracle.grid import Grid
from oracle.schwarz import OneLevelRAS

pytestmark = pytest.mark.gpu

PH = dict(E=1e-3, Ra=100.0, Pr=1.0, Pm=5.0, dt=1e-4)


@pytest.mark.parametrize('kind,Ns,Nr,parts,delta', [
    (1, 4, 2, (4, 4, 2), 0),      # boxes of one cell
    (0, 5, 3, (2, 2, 3), 1),      # VTBE, one-warp windows, odd boxes
    (1, 24, 16, (1, 1, 1), 0),    # 9216 cells a box: more chunks than the ring holds, both directions
    (0, 20, 14, (1, 1, 1), 1),    # VTBE with the forward result in global memory
    (1, 28, 26, (1, 1, 1), 0),    # a window of 377 rows: 384 threads
    (1, 28, 32, (1, 1, 1), 0),    # steps of more than 384 cells: the general sweeps
    (1, 11, 7, (3, 2, 2), 2),     # uneven boxes
    (0, 13, 9, (3, 2, 2), 2)])
def test_sweeps_match_oracle(kind, Ns, Nr, parts, delta):
    import torch

    from paper_2009_02171_gb300 import fv
    d = Discretization(Grid(Ns, Nr))
    A = vtbe_matrix(d, **PH) if kind == 0 else ppbe_matrix(d, PH['E'], PH['dt'])
    M = OneLevelRAS(Grid(Ns, Nr), A, 7 if kind == 0 else 2, parts, delta)
    g = fv.fv_build_grid(Ns, Nr)
    s = fv.fv_assemble_system(g, kind, **PH, p=parts, overlap=delta)
    r = np.random.default_rng(3).standard_normal(A.shape[0])
    z = fv.fv_precond_apply(s, torch.tensor(r, device='cuda'), torch.empty(r.size, dtype=torch.float64, device='cuda'))
    ref = M.apply(r)
    assert np.abs(z.cpu().numpy() - ref).max() <= 1e-11 * np.abs(ref).max()
    fv.fv_free_system(s)
    fv.fv_free_grid(g)


def test_sweeps_are_reproducible():
    """Several CTAs an SM, forward results in global memory, the operand ring wrapping many times: the same bits every
    time, other right-hand sides in between (operands are refilled while other warps still solve)."""
    import torch

    from paper_2009_02171_gb300 import fv
    g = fv.fv_build_grid(48, 72)
    s = fv.fv_assemble_system(g, 1, **PH, p=(3, 3, 3), overlap=2)
    n = fv.fv_system_size(s)
    gen = torch.Generator('cuda').manual_seed(1)
    r, q = (torch.randn(n, dtype=torch.float64, device='cuda', generator=gen) for _ in range(2))
    first = fv.fv_precond_apply(s, r, torch.empty_like(r)).clone()
    z, w = torch.empty_like(r), torch.empty_like(r)
    for t in range(60):
        if t % 3 == 0:
            fv.fv_precond_apply(s, q, w)
        assert torch.equal(fv.fv_precond_apply(s, r, z), first)
    fv.fv_free_system(s)
    fv.fv_free_grid(g)
