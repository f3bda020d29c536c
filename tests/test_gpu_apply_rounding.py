"""Rounding of the FP32 operator apply: its tables are FP64 values rounded once, so the error against the oracle's matrix on the
same FP32 vector stays below one and a half units of roundoff of the result's norm (an element sums about 15 products, most
of them of opposite signs, each with two roundings; they average over the vector)."""
import numpy as np
import pytest

torch = pytest.importorskip('torch')
pytestmark = pytest.mark.gpu

from oracle.discrete import Discretization, ppbe_matrix, vtbe_matrix  # noqa: E402
from oracle.grid import Grid  # noqa: E402

PH = dict(E=1e-3, Ra=100.0, Pr=1.0, Pm=5.0, dt=1e-4)


@pytest.mark.parametrize('kind,Ns,Nr', [(1, 33, 17), (1, 24, 12), (1, 40, 9), (0, 33, 17), (0, 24, 12)])
def test_fp32_apply_rounds_its_tables_once(kind, Ns, Nr):
    from paper_2009_02171_gb300 import fv
    d = Discretization(Grid(Ns, Nr))
    A = vtbe_matrix(d, **PH) if kind == 0 else ppbe_matrix(d, PH['E'], PH['dt'])
    g = fv.fv_build_grid(Ns, Nr)
    s = fv.fv_assemble_system(g, kind, **PH, precision=1, inner_maxit=2)
    x = torch.tensor(np.random.default_rng(4).standard_normal(A.shape[0]), device='cuda').float()
    y = fv.fv_apply_op_fp32(s, x, torch.empty_like(x)).double().cpu().numpy()
    ref = A @ x.double().cpu().numpy()
    assert np.linalg.norm(y - ref) <= 1.5 * 2.0 ** -24 * np.linalg.norm(ref)
    fv.fv_free_system(s)
    fv.fv_free_grid(g)
