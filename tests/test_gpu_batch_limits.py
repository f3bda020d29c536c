"""A batched solve obeys its own iteration limit when it replays a restart cycle that a solve with another limit captured."""
import pytest

torch = pytest.importorskip('torch')
pytestmark = pytest.mark.gpu

from paper_2009_02171_gb300.inputs import random_vector  # noqa: E402

PH = dict(E=1e-3, Ra=100.0, Pr=1.0, Pm=5.0, dt=1e-4)


@pytest.mark.parametrize('limits', [(12, 2000, 12, 17), (2000, 12, 2000, 3)])
def test_replayed_cycles_obey_the_limit_of_the_call(limits):
    from paper_2009_02171_gb300 import fv
    g = fv.fv_build_grid(12, 12)
    s = fv.fv_assemble_system(g, fv.FV_PPBE, **PH, p=(2, 2, 2), overlap=1)
    n = fv.fv_system_size(s)
    B = torch.stack([torch.tensor(random_vector(n, 70 + r), device='cuda') for r in range(3)])
    for r in range(3):
        B[r] = fv.fv_apply_op(s, B[r].clone(), torch.empty_like(B[r]))  # consistent for the Neumann block
    X = torch.zeros_like(B)
    for limit in limits:  # FGMRES(5): one eager cycle, then captured and replayed ones
        X.zero_()
        st = fv.fv_gmres_solve_batch(s, B, X, restart=5, rtol=1e-8, max_it=limit, raise_on_noconv=False)
        for t in st:
            if limit == 2000:
                assert t.converged and 17 < t.iters < 2000
            else:
                assert not t.converged and t.iters == limit
    fv.fv_free_system(s)
    fv.fv_free_grid(g)
