"""The Gram-Schmidt step's coefficients, Givens rotations and least squares (csrc/krylov.cu): the iterate after exactly m
steps, with no restart to mend it, against the oracle's FGMRES.  m stands at the edges of the register and reduction chunks
(1, 8, 9, 16, 17, 31), the vectors are one block, several with a ragged last one, and (VTBE on odd grids) no multiple of a
16-byte load in FP32."""
import numpy as np
import pytest

torch = pytest.importorskip('torch')
pytestmark = pytest.mark.gpu

from oracle.discrete import Discretization, ppbe_matrix, vtbe_matrix  # noqa: E402
from oracle.grid import Grid  # noqa: E402
from oracle.krylov import fgmres  # noqa: E402
from oracle.schwarz import OneLevelRAS  # noqa: E402

PH = dict(E=1e-3, Ra=100.0, Pr=1.0, Pm=5.0)


@pytest.mark.parametrize('kind,Ns,Nr,parts,dt', [
    (1, 4, 2, (2, 2, 1), 1e-4),    # 384 values
    (0, 5, 3, (2, 2, 1), 1.0),     # 3150, two beyond the last 16 bytes
    (1, 13, 11, (2, 2, 1), 1e-4),
    (0, 9, 7, (3, 3, 2), 1e-2),
    (1, 24, 12, (3, 3, 2), 1e-4)])
def test_iterates_after_m_steps_match_oracle(kind, Ns, Nr, parts, dt):
    """Bars, for ||A (x - x_oracle)|| / ||b||: FP64 1e-11 a step (the bar of one preconditioner application); FP32 16 units of
    roundoff a step, times || |A| |x| || / ||b||, the growth of a product's rounding (an FP32 run of the same steps in numpy
    stays below a fifth of that)."""
    from paper_2009_02171_gb300 import fv
    d = Discretization(Grid(Ns, Nr))
    A = vtbe_matrix(d, dt=dt, **PH) if kind == 0 else ppbe_matrix(d, PH['E'], dt)
    M = OneLevelRAS(Grid(Ns, Nr), A, 7 if kind == 0 else 2, parts, 0)
    b = A @ np.random.default_rng(5).standard_normal(A.shape[0])
    bd = torch.tensor(b, device='cuda')
    g = fv.fv_build_grid(Ns, Nr)
    s = fv.fv_assemble_system(g, kind, dt=dt, **PH, p=parts, overlap=0)
    for m in (1, 2, 8, 9, 16, 17, 31):
        ref = fgmres(lambda v: A @ v, M.apply, b, np.zeros_like(b), restart=m, rtol=1e-14, maxit=m)
        off = lambda x: np.linalg.norm(A @ (x.cpu().numpy() - ref.x)) / np.linalg.norm(b)  # noqa: E731
        x = torch.zeros_like(bd)
        st = fv.fv_gmres_solve(s, bd, x, restart=m, max_it=m, rtol=1e-14, raise_on_noconv=False)
        assert abs(st.iters - ref.iters) <= (0 if ref.rfinal > 1e-12 * ref.r0 else 1) and off(x) <= 1e-11 * (m + 1), (m, off(x))
        bar = 16 * 2.0 ** -24 * (m + 1) * max(1.0, np.linalg.norm(abs(A) @ abs(ref.x)) / np.linalg.norm(b))
        for passes in (1, 2):
            s32 = fv.fv_assemble_system(g, kind, dt=dt, **PH, p=parts, overlap=0, precision=1, inner_maxit=m,
                                        inner_gs_passes=passes)
            z = fv.fv_precond_apply(s32, bd, torch.empty_like(bd))
            assert off(z) <= bar, (m, passes, off(z), bar)
            fv.fv_free_system(s32)
    fv.fv_free_system(s)
    fv.fv_free_grid(g)
