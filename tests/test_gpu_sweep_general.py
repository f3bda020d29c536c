"""The general sweeps (boxes with more than 384 cells in a step) in every precision: one application against the oracle's ILU(0)
solves, batched solves by groups of right-hand sides (a last group that is not full among them) and mixed solves by the
iterations of FP64 ones."""
import numpy as np
import pytest

torch = pytest.importorskip('torch')
pytestmark = pytest.mark.gpu

from oracle.discrete import Discretization, ppbe_matrix, vtbe_matrix  # noqa: E402
from oracle.grid import Grid  # noqa: E402
from oracle.schwarz import OneLevelRAS  # noqa: E402

PH = dict(E=1e-3, Ra=100.0, Pr=1.0, Pm=5.0, dt=1e-4)
NS, NR = 28, 32  # one box a panel: steps of 440 cells and more


def _matrix(kind):
    d = Discretization(Grid(NS, NR))
    return vtbe_matrix(d, **PH) if kind == 0 else ppbe_matrix(d, PH['E'], PH['dt'])


def _backward_launches(fv, call):
    fv.fv_profile_enable(True)
    call()
    n = sum(fv.fv_profile_read(c)[0] for c in range(fv.K_COUNT) if fv.category_name(c).startswith('ras_bwd'))
    fv.fv_profile_enable(False)
    return n


@pytest.mark.parametrize('kind', [0, 1])
def test_general_sweeps_match_oracle(kind):
    from paper_2009_02171_gb300 import fv
    A = _matrix(kind)
    M = OneLevelRAS(Grid(NS, NR), A, 7 if kind == 0 else 2, (1, 1, 1), 0)
    g = fv.fv_build_grid(NS, NR)
    s = fv.fv_assemble_system(g, kind, **PH, p=(1, 1, 1), overlap=0)
    r = np.random.default_rng(3).standard_normal(A.shape[0])
    rd = torch.tensor(r, device='cuda')
    z = torch.empty_like(rd)
    assert _backward_launches(fv, lambda: fv.fv_precond_apply(s, rd, z)) == 1
    ref = M.apply(r)
    assert np.abs(z.cpu().numpy() - ref).max() <= 1e-11 * np.abs(ref).max()
    fv.fv_free_system(s)
    fv.fv_free_grid(g)


@pytest.mark.parametrize('kind', [0, 1])
def test_general_sweeps_in_solves(kind):
    """Batches of 3 and 5 (groups of up to 4) in FP64 and FP32 take the iterations of single FP64 solves, within one, and
    reach the tolerance on the oracle's matrix; mixed solves of eight inner iterations an outer one take at most half as
    many, BF16 factors two more than FP32 at most."""
    from paper_2009_02171_gb300 import fv
    A = _matrix(kind)
    g = fv.fv_build_grid(NS, NR)
    rng = np.random.default_rng(8)
    b = np.stack([A @ rng.standard_normal(A.shape[0]) for _ in range(5)])
    bd = torch.tensor(b, device='cuda')
    single, its = [], {}
    for prec in (0, 1, 2):
        s = fv.fv_assemble_system(g, kind, **PH, p=(1, 1, 1), overlap=0, precision=prec, inner_maxit=8)
        for r in range(5 if prec == 0 else 1):
            x = torch.zeros_like(bd[0])
            st = fv.fv_gmres_solve(s, bd[r], x, rtol=1e-8)
            assert st.converged and np.linalg.norm(b[r] - A @ x.cpu().numpy()) <= 1.0001e-8 * np.linalg.norm(b[r])
            if prec == 0:
                single.append(st.iters)
            its[prec] = st.iters
        for nrhs in (3, 5) if prec < 2 else ():
            X = torch.zeros_like(bd[:nrhs])
            st = fv.fv_gmres_solve_batch(s, bd[:nrhs].contiguous(), X, rtol=1e-8)
            for r in range(nrhs):
                assert st[r].converged and abs(st[r].iters - single[r]) <= 1, (prec, r, st[r].iters, single)
                assert np.linalg.norm(b[r] - A @ X[r].cpu().numpy()) <= 1.0001e-8 * np.linalg.norm(b[r])
        fv.fv_free_system(s)
    assert its[1] <= max(single[0] // 2, 2) and its[2] <= its[1] + 2, (single, its)
    fv.fv_free_grid(g)
