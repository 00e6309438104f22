"""BF16 products with more row tiles than the GPU has SMs (the persistent
kernel) and weight gradients with long k loops (six-stage ring), through
forward and backward of batches of 20,000 to 25,000 atoms.

Gradients against the FP32 path of the library, which other tests check against
the oracle, within the derived BF16 bound; predictions of a row-invariant
context against small batches, which the tile kernel computes, bit for bit."""
import numpy as np
import pytest
import torch

import synth
from gpu_common import write_both
from helpers import BF16_FWD_TOL, bf16_grad_bound, graph_set, rel_norm, residual_kappa

pytestmark = pytest.mark.gpu


def _step(g, st, gs, H, precision, recompute):
    G = gs.n_graphs
    ctx = g.Context(g.make_config(H, 1, G, gs.n_nodes, gs.n_edges, delta=st.delta(), precision=precision,
                                  recompute=recompute))
    ctx.set_params(synth.init_params(6, H, 1))
    b = ctx.collate(st, np.arange(G))
    pred = torch.empty(G, device="cuda")
    ctx.forward(b, pred, train=True)
    ctx.backward(b)
    ctx.check()
    return pred.cpu().numpy(), ctx.activations(b)[1], ctx.get_grads()


# widths: one partly filled column tile; two tiles, the last one partly filled;
# whole tiles (H = 256, whose dW_U splits k in two halves of 10,000 and more)
@pytest.mark.parametrize("recompute", [0, 1])
@pytest.mark.parametrize("G,lo,hi,H", [(1250, 18, 22, 24), (1250, 18, 22, 136), (641, 32, 32, 256)])
def test_many_rows(tmp_path, G, lo, hi, H, recompute):
    import paper_2207_11333_gb300 as g
    gs = graph_set(9, G, lo, hi)
    path, _ = write_both(gs, str(tmp_path))
    st = g.Store(path)
    assert gs.n_nodes > 152 * 128
    _, x16, g16 = _step(g, st, gs, H, g.PREC_BF16, recompute)
    p32, x32, g32 = _step(g, st, gs, H, g.PREC_FP32, recompute)
    assert rel_norm(x16, x32) < BF16_FWD_TOL  # (the predictions of random weights nearly cancel)
    assert rel_norm(g16, g32) < bf16_grad_bound(1, residual_kappa(p32, gs.y))


@pytest.mark.parametrize("H", [8, 72, 136, 256])
def test_rows_alone_and_in_a_large_batch(tmp_path, H):
    import paper_2207_11333_gb300 as g
    gs = graph_set(11, 1250, 18, 22)
    path, _ = write_both(gs, str(tmp_path))
    st = g.Store(path)

    def predictions(ids):
        ctx = g.Context(g.make_config(H, 2, len(ids), *map(int, st.batch_size(ids)), delta=st.delta(),
                                      precision=g.PREC_BF16, flags=g.FLAG_ROW_INVARIANT))
        ctx.set_params(synth.init_params(12, H, 2))
        pred = torch.empty(len(ids), device="cuda")
        ctx.forward(ctx.collate(st, ids), pred, train=False)
        ctx.check()
        return pred.cpu().numpy()

    whole = predictions(np.arange(1250))
    for ids in (np.arange(0, 5), np.arange(620, 640), np.arange(1249, 1250)):
        assert np.array_equal(whole[ids], predictions(ids))
