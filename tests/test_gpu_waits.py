"""Bounded waits that run out are reported: the grid barrier of the Gram-Schmidt steps is given a limit of one try, which
its first arrivals always exceed (the kernels go on in range and end; no wait is left out)."""
import ctypes

import pytest

torch = pytest.importorskip('torch')
pytestmark = pytest.mark.gpu

from paper_2009_02171_gb300.inputs import random_vector  # noqa: E402

PH = dict(E=1e-3, Ra=100.0, Pr=1.0, Pm=5.0, dt=1e-4)
DEFAULT = 1 << 24


def _limit(fv, h, tries):
    f = fv.lib.fv_set_wait_limit
    f.argtypes, f.restype = [ctypes.c_void_p, ctypes.c_uint], ctypes.c_int
    assert f(h, tries) == 0


def _system(fv, g, prec, levels):
    s = fv.fv_assemble_system(g, fv.FV_PPBE, **PH, p=(2, 2, 1), overlap=1, levels=levels, precision=prec, inner_maxit=4,
                              coarse_maxit=4)
    x = torch.tensor(random_vector(fv.fv_system_size(s), 41), device='cuda')
    return s, fv.fv_apply_op(s, x, torch.empty_like(x))  # consistent for the Neumann block


@pytest.mark.parametrize('prec,levels,coarse', [
    (0, 1, False),  # the FP64 basis of the outer solve
    (0, 2, True),   # the FP64 basis of the coarse solve
    (1, 1, False),  # the FP32 basis of the inner solve (and the outer one)
    (1, 2, True)])  # the FP32 basis of the coarse solve inside the inner one: its words alone
def test_a_barrier_that_runs_out_fails_the_solve_and_no_later_one(prec, levels, coarse):
    from paper_2009_02171_gb300 import fv
    g = fv.fv_build_grid(16, 12)  # the coarse level's vectors span four blocks
    s, b = _system(fv, g, prec, levels)
    x = torch.zeros_like(b)
    h = fv.fv_coarse_system(s) if coarse else s
    _limit(fv, h, 1)
    with pytest.raises(fv.FvError, match='wait'):
        fv.fv_gmres_solve(s, b, x, rtol=1e-8)
    _limit(fv, h, DEFAULT)
    _limit(fv, s, DEFAULT)  # drops the captured inner solve, which holds the coarse limit
    assert fv.fv_gmres_solve(s, b, x.zero_(), rtol=1e-8).converged
    fresh, _ = _system(fv, g, prec, levels)
    y = torch.zeros_like(b)
    assert fv.fv_gmres_solve(fresh, b, y, rtol=1e-8).converged and torch.equal(x, y)
    for q in (s, fresh):
        fv.fv_free_system(q)
    fv.fv_free_grid(g)


@pytest.mark.parametrize('batch', [False, True])
def test_an_application_that_failed_is_reported_before_the_next_call_begins(batch):
    from paper_2009_02171_gb300 import fv
    g = fv.fv_build_grid(16, 12)
    s, b = _system(fv, g, 1, 1)
    _limit(fv, s, 1)
    z = fv.fv_precond_apply(s, b, torch.empty_like(b))  # returns before its kernels have finished
    torch.cuda.synchronize()
    _limit(fv, s, DEFAULT)
    x = torch.full_like(b, 0.5)
    solve = ((lambda: fv.fv_gmres_solve_batch(s, b[None], x[None], rtol=1e-8)[0]) if batch else
             (lambda: fv.fv_gmres_solve(s, b, x, rtol=1e-8)))
    with pytest.raises(fv.FvError, match='not begun, in an earlier call'):
        solve()
    assert (x == 0.5).all()
    assert solve().converged
    _limit(fv, s, 1)
    fv.fv_precond_apply(s, b, z)
    torch.cuda.synchronize()
    z.fill_(0.5)
    with pytest.raises(fv.FvError, match='not begun, in an earlier call'):
        fv.fv_precond_apply(s, b, z)
    assert (z == 0.5).all()
    fv.fv_free_system(s)
    fv.fv_free_grid(g)
