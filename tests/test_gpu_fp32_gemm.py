"""The FP32 GEMMs at the edges of their tiles, and the K-chunks of row-invariant products.

Edges: node counts around the tile heights (64, 96, 128 and 160 rows) and
widths that fill a 32-column warp, part of one and several tiles, against the
FP64 oracle with the tolerances of the parity tests (FP32 forward 1e-5,
gradients 1e-4, normwise).

Row invariance: a row-invariant context sums K in fixed chunks, in parallel
CTAs with a reduction for few rows and inside one CTA for many.  A molecule's
prediction has to be the same bit for bit either way (hidden 40: K = 640 in
the update, three chunks; more than 76 x 128 rows: one CTA each)."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_common import context, oracle_step, write_both
from helpers import FP32_FWD_TOL, FP32_GRAD_TOL, graph_set, rel_norm

pytestmark = pytest.mark.gpu


def _run(tmp_path, G, n, H, L):
    import paper_2207_11333_gb300 as g
    gs = graph_set(5, G, n, n)
    path, ost = write_both(gs, str(tmp_path))
    st = g.Store(path)
    ctx = context(H, L, G, gs.n_nodes, gs.n_edges, st.delta())
    params = synth.init_params(6, H, L)
    ctx.set_params(params)
    b = ctx.collate(st, np.arange(G))
    return ctx, b, oracle.collate(ost, np.arange(G), st.delta()), params


@pytest.mark.parametrize("G,n", [(1, 3), (3, 21), (1, 64), (5, 13), (5, 19), (1, 97), (1, 128), (43, 3), (7, 23)])
@pytest.mark.parametrize("H", [8, 40, 136])
def test_tile_edges(tmp_path, G, n, H):
    L = 1
    ctx, b, ob, params = _run(tmp_path, G, n, H, L)
    pred = torch.empty(G, device="cuda")
    ctx.forward(b, pred, train=True)
    ctx.backward(b)
    grads = ctx.get_grads()
    ctx.check()
    d = oracle.Dims(H=H, L=L)
    _, ograd, opred, _ = oracle_step(d, params, ob)
    assert rel_norm(pred.cpu().numpy(), opred) < FP32_FWD_TOL
    gv, ov = oracle.split_params(d, grads), oracle.split_params(d, ograd)
    for k in ov:
        assert rel_norm(gv[k], ov[k]) < FP32_GRAD_TOL, k


@pytest.mark.parametrize("H", [40, 104])
def test_row_invariant_chunks(tmp_path, H):
    import paper_2207_11333_gb300 as g
    gs = graph_set(7, 640, 17, 17)
    path, _ = write_both(gs, str(tmp_path))
    st = g.Store(path)
    assert gs.n_nodes > 76 * 128
    preds = []
    for G in (640, 1, 9):
        cfg = g.make_config(H, 1, G, 17 * G, int(gs.edge_ptr[G]), delta=st.delta(), flags=g.FLAG_ROW_INVARIANT)
        ctx = g.Context(cfg)
        ctx.set_params(synth.init_params(8, H, 1))
        pred = torch.empty(G, device="cuda")
        ctx.forward(ctx.collate(st, np.arange(G)), pred, train=False)
        ctx.check()
        preds.append(pred.cpu().numpy())
    assert np.array_equal(preds[0][:1], preds[1])
    assert np.array_equal(preds[0][:9], preds[2])
