"""Weight and bias gradients (csrc/nn.cu) where a chunk of 64 cells starts inside a row, touches many short rows, or reaches
past the last cell, against the FP64 oracle on the same BF16 weights (the bars of the network's gradient test)."""
import numpy as np
import pytest

from oracle import unet

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize('C,Ns,Nr,levels', [(16, 12, 4, 2), (16, 5, 3, 0), (32, 6, 2, 1), (16, 70, 1, 0)])
def test_gradients_at_chunk_edges(C, Ns, Nr, levels):
    import torch

    from paper_2009_02171_gb300 import fv
    from paper_2009_02171_gb300.inputs import multiscale_fields
    rng = np.random.default_rng(7)
    w = np.concatenate([np.concatenate([rng.standard_normal(27 * ci * co) * np.sqrt(2 / (27 * ci)), 0.1 * rng.standard_normal(co)])
                        for ci, co in unet.layer_shapes(C, levels).values()]).astype(np.float32)
    u = w.view(np.uint32).astype(np.uint64)
    u = (u + 0x7FFF + ((u >> 16) & 1)) >> 16  # nearest BF16, ties to even
    low = unet.unflatten((u << 16).astype(np.uint32).view(np.float32).astype(np.float64), C, levels)
    ref = {k: (low[k][0], b) for k, (_, b) in unet.unflatten(w.astype(np.float64), C, levels).items()}
    net = fv.fv_net_create(C, Ns, Nr, levels=levels, max_batch=2)
    fv.fv_net_set_params(net, w)
    r, e = multiscale_fields(Ns, Nr, 2, seed=5), multiscale_fields(Ns, Nr, 2, seed=6)
    dev = lambda a: torch.tensor(np.ascontiguousarray(a).ravel(), device='cuda')  # noqa: E731
    to = lambda v: v.reshape(-1, 2, 6, Nr, Ns, Ns).transpose(0, 2, 1, 3, 4, 5).reshape(-1, 2, Nr, Ns, Ns)  # noqa: E731
    loss, g = fv.fv_net_loss_grad(net, 2, dev(r), dev(e))
    L, gr = unet.loss_and_grads(ref, to(r), to(e), levels)
    g, want = g.astype(np.float64), unet.flatten(gr)
    assert abs(loss - L) < 1e-2 * L
    assert np.linalg.norm(g - want) < 5e-2 * np.linalg.norm(want)
    got = unet.unflatten(g, C, levels)
    for k in gr:
        for a, b in zip(got[k], gr[k]):
            cos = (a * b).sum() / max(np.linalg.norm(a) * np.linalg.norm(b), 1e-300)
            assert np.linalg.norm(a - b) < 0.2 * np.linalg.norm(b) and cos > 0.98, (k, cos)
    fv.fv_net_free(net)
