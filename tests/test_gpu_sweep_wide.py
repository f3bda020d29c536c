"""Boxes whose widest step fits a CTA (384 cells) but whose window of rows held a step longer does not, and boxes with more rows
than shared memory holds a table of: streamed like the others (both directions of a box in one launch), against the oracle's
ILU(0) solves and, in FP32 and BF16, by the iterations of FP64 solves."""
import numpy as np
import pytest

torch = pytest.importorskip('torch')
pytestmark = pytest.mark.gpu

from oracle.discrete import Discretization, ppbe_matrix, vtbe_matrix  # noqa: E402
from oracle.grid import Grid  # noqa: E402
from oracle.schwarz import OneLevelRAS  # noqa: E402

PH = dict(E=1e-3, Ra=100.0, Pr=1.0, Pm=5.0, dt=1e-4)


def _backward_launches(fv, call):
    """launches of a backward sweep of its own (the streamed sweeps have none) in call()"""
    fv.fv_profile_enable(True)
    call()
    n = sum(fv.fv_profile_read(c)[0] for c in range(fv.K_COUNT) if fv.category_name(c).startswith('ras_bwd'))
    fv.fv_profile_enable(False)
    return n


@pytest.mark.parametrize('kind,Ns,Nr,parts,delta', [
    (1, 24, 32, (1, 1, 1), 0),   # widest step 376, window 390
    (1, 48, 16, (1, 1, 1), 0),   # 384 and 392: every thread busy, rows begin the step after the last one ends
    (1, 50, 20, (2, 2, 1), 5),   # uneven: corner boxes 30 x 30 x 20 among others
    (0, 24, 32, (1, 1, 1), 0),
    (1, 5, 1023, (5, 1, 1), 0),  # one cell along i; 5115 rows, read from global memory
    (1, 6, 1000, (3, 1, 1), 0),
    (0, 5, 1023, (5, 1, 1), 0)])
def test_wide_and_long_boxes_match_oracle(kind, Ns, Nr, parts, delta):
    from paper_2009_02171_gb300 import fv
    d = Discretization(Grid(Ns, Nr))
    A = vtbe_matrix(d, **PH) if kind == 0 else ppbe_matrix(d, PH['E'], PH['dt'])
    M = OneLevelRAS(Grid(Ns, Nr), A, 7 if kind == 0 else 2, parts, delta)
    g = fv.fv_build_grid(Ns, Nr)
    s = fv.fv_assemble_system(g, kind, **PH, p=parts, overlap=delta)
    r = np.random.default_rng(3).standard_normal(A.shape[0])
    rd = torch.tensor(r, device='cuda')
    z = torch.empty_like(rd)
    assert _backward_launches(fv, lambda: fv.fv_precond_apply(s, rd, z)) == 0
    ref = M.apply(r)
    assert np.abs(z.cpu().numpy() - ref).max() <= 1e-11 * np.abs(ref).max()
    first = z.clone()
    for _ in range(10):
        assert torch.equal(fv.fv_precond_apply(s, rd, z), first)
    fv.fv_free_system(s)
    fv.fv_free_grid(g)


@pytest.mark.parametrize('kind', [0, 1])
def test_wide_boxes_in_lower_precision(kind):
    """FP32 sweeps inside the FP64 batch solver take the iterations of FP64 ones (within one); mixed solves reach the
    tolerance in at most half as many outer iterations (eight inner ones each), BF16 factors within two of FP32."""
    from paper_2009_02171_gb300 import fv
    Ns, Nr = 24, 32
    g = fv.fv_build_grid(Ns, Nr)
    its = {}
    for name, prec in (('f64', 0), ('batch32', 1), ('f32', 1), ('bf16', 2)):
        s = fv.fv_assemble_system(g, kind, **PH, precision=prec, overlap=0, inner_maxit=8)
        n = fv.fv_system_size(s)
        x = torch.randn(n, dtype=torch.float64, device='cuda', generator=torch.Generator('cuda').manual_seed(2))
        b = fv.fv_apply_op(s, x, torch.empty_like(x))
        if name == 'batch32':
            X = torch.zeros(2, n, dtype=torch.float64, device='cuda')
            st = fv.fv_gmres_solve_batch(s, torch.stack([b, -b]), X, rtol=1e-8)
            its[name] = [t.iters for t in st]
        else:
            st = [fv.fv_gmres_solve(s, b, x.zero_(), rtol=1e-8)]
            its[name] = st[0].iters
        assert all(t.converged for t in st)
        assert _backward_launches(fv, lambda: fv.fv_precond_apply(s, b, x)) == 0
        fv.fv_free_system(s)
    assert all(abs(i - its['f64']) <= 1 for i in its['batch32']), its
    assert its['f32'] <= max(its['f64'] // 2, 2) and its['bf16'] <= its['f32'] + 2, its
    fv.fv_free_grid(g)
