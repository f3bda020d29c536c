"""Many small boxes, more than the device runs at once: the sweeps' small operand ring, its widest step, uneven boxes, boxes of
one chunk and of less, and boxes of a cell or a few, which the general sweeps take."""
import numpy as np
import pytest

torch = pytest.importorskip('torch')
pytestmark = pytest.mark.gpu

from oracle.discrete import Discretization, ppbe_matrix, vtbe_matrix  # noqa: E402
from oracle.grid import Grid  # noqa: E402
from oracle.schwarz import OneLevelRAS  # noqa: E402

PH = dict(E=1e-3, Ra=100.0, Pr=1.0, Pm=5.0, dt=1e-4)


@pytest.mark.parametrize('kind,Ns,Nr,parts,delta', [
    (1, 16, 16, (4, 4, 4), 1),
    (0, 16, 12, (4, 4, 3), 1),
    (1, 17, 13, (4, 4, 4), 1),   # uneven
    (0, 17, 13, (5, 4, 4), 2),
    (1, 12, 12, (6, 6, 6), 0),   # 8 cells a box, chunks of 32
    (0, 12, 12, (6, 6, 6), 0),
    (1, 64, 24, (8, 8, 1), 0),   # steps of 64 cells, the widest
    (0, 24, 40, (6, 6, 1), 1),   # long boxes: the ring wraps many times
    (1, 8, 8, (8, 8, 8), 0),     # one cell
    (0, 8, 8, (8, 8, 8), 0)])
def test_small_boxes_match_oracle(kind, Ns, Nr, parts, delta):
    from paper_2009_02171_gb300 import fv
    d = Discretization(Grid(Ns, Nr))
    A = vtbe_matrix(d, **PH) if kind == 0 else ppbe_matrix(d, PH['E'], PH['dt'])
    M = OneLevelRAS(Grid(Ns, Nr), A, 7 if kind == 0 else 2, parts, delta)
    g = fv.fv_build_grid(Ns, Nr)
    s = fv.fv_assemble_system(g, kind, **PH, p=parts, overlap=delta)
    r, q = np.random.default_rng(3).standard_normal((2, A.shape[0]))
    rd, qd = torch.tensor(r, device='cuda'), torch.tensor(q, device='cuda')
    z, w = torch.empty_like(rd), torch.empty_like(rd)
    first = fv.fv_precond_apply(s, rd, z).clone()
    ref = M.apply(r)
    assert np.abs(first.cpu().numpy() - ref).max() <= 1e-11 * np.abs(ref).max()
    for t in range(12):
        if t % 3 == 0:
            fv.fv_precond_apply(s, qd, w)
        assert torch.equal(fv.fv_precond_apply(s, rd, z), first)
    fv.fv_free_system(s)
    fv.fv_free_grid(g)


@pytest.mark.parametrize('kind', [0, 1])
@pytest.mark.parametrize('parts', [(5, 5, 4), (10, 10, 8)])
def test_small_boxes_in_lower_precision(kind, parts):
    """FP32 sweeps inside the FP64 batch solver take the iterations of FP64 ones (within one); mixed solves reach the
    tolerance in at most half as many outer iterations (eight inner ones each), BF16 factors within two of FP32."""
    from paper_2009_02171_gb300 import fv
    g = fv.fv_build_grid(20, 16)
    its = {}
    for name, prec in (('f64', 0), ('batch32', 1), ('f32', 1), ('bf16', 2)):
        s = fv.fv_assemble_system(g, kind, **PH, p=parts, overlap=1, precision=prec, inner_maxit=8)
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
        fv.fv_free_system(s)
    assert all(abs(i - its['f64']) <= 1 for i in its['batch32']), its
    assert its['f32'] <= max(its['f64'] // 2, 2) and its['bf16'] <= its['f32'] + 2, its
    fv.fv_free_grid(g)


@pytest.mark.parametrize('kind,parts', [(0, 16), (1, 16), (0, 8), (1, 8)])
def test_boxes_of_a_few_cells_are_not_padded_out(kind, parts):
    """A system's memory on 24,576 boxes of one cell and 3072 of eight: at most five times the matrix entries and vectors a
    box cell needs (FP64: 10 d + d^2 factors, a forward result, an index), beside 40 MB of tables and allocation grain."""
    from paper_2009_02171_gb300 import fv
    g = fv.fv_build_grid(16, 16)
    fv.fv_free_system(fv.fv_assemble_system(g, kind, **PH, p=(1, 1, 1), overlap=0))  # code and tables are loaded
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    s = fv.fv_assemble_system(g, kind, **PH, p=(parts, parts, parts), overlap=0)
    used = before - torch.cuda.mem_get_info()[0]
    d = 7 if kind == 0 else 2
    assert used <= 5 * 6 * 16 ** 3 * ((11 * d + d * d) * 8 + 16) + 40e6, used
    fv.fv_free_system(s)
    fv.fv_free_grid(g)
