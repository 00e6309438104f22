"""FP32 inference on the tensor cores (exact integer slices) against the FP64
oracle, beside the CUDA-core path (a training forward).

The slices keep 26 bits below a row's largest entry, two more than FP32, and
their sums are exact, so the error has to stay at or below the plain path's:
per layer at most 1.5 times it (both are a few roundings of FP32), and always
within the FP32 forward tolerance of the parity tests.  Row invariance, changed
parameters and non-finite weights are checked on the same contexts."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_common import context, write_both
from helpers import FP32_FWD_TOL, graph_set, rel_norm

pytestmark = pytest.mark.gpu


def _setup(tmp_path, G, lo, hi, H, L, flags=0):
    import paper_2207_11333_gb300 as g
    gs = graph_set(21, G, lo, hi)
    path, ost = write_both(gs, str(tmp_path))
    st = g.Store(path)
    ctx = g.Context(g.make_config(H, L, G, gs.n_nodes, gs.n_edges, delta=st.delta(), flags=flags))
    params = synth.init_params(22, H, L)
    ctx.set_params(params)
    return gs, ost, st, ctx, params


# widths: the smallest and the largest, whole and partly filled k tiles, column
# tiles of 64 to 112; more than 2,048 rows for the default contexts; the last
# batch runs an update's phases one after the other, the others in parallel
@pytest.mark.parametrize("G,lo,hi,H,L", [(110, 18, 22, 64, 2), (110, 18, 22, 72, 2), (130, 15, 20, 136, 2),
                                         (110, 18, 22, 200, 2), (110, 18, 22, 256, 1), (1100, 18, 22, 64, 1)])
def test_accuracy(tmp_path, G, lo, hi, H, L):
    gs, ost, st, ctx, params = _setup(tmp_path, G, lo, hi, H, L)
    assert gs.n_nodes >= 2048
    b = ctx.collate(st, np.arange(G))
    d = oracle.Dims(H=H, L=L)
    opred, oxs, _, _ = oracle.forward(d, params.astype(np.float64), oracle.collate(ost, np.arange(G), st.delta()),
                                      want_layers=True)
    pred = torch.empty(G, device="cuda")
    errors = []
    for train in (True, False):
        ctx.forward(b, pred, train=train)
        ctx.check()
        errors.append([rel_norm(x, o) for x, o in zip(ctx.activations(b)[1:], oxs[1:])])
        assert rel_norm(pred.cpu().numpy(), opred) < FP32_FWD_TOL
    for plain, slices in zip(*errors):
        assert slices < FP32_FWD_TOL and slices <= 1.5 * plain


def test_row_invariant_and_new_parameters(tmp_path):
    import paper_2207_11333_gb300 as g
    G = 700
    gs, ost, st, ctx, params = _setup(tmp_path, G, 18, 22, 104, 2, flags=g.FLAG_ROW_INVARIANT)
    pred = torch.empty(G, device="cuda")
    ctx.forward(ctx.collate(st, np.arange(G)), pred, train=False)
    whole = pred.cpu().numpy()
    for ids in (np.arange(3), np.arange(200, 330), np.arange(G - 1, G)):
        part = torch.empty(len(ids), device="cuda")
        ctx.forward(ctx.collate(st, ids), part, train=False)
        assert np.array_equal(part.cpu().numpy(), whole[ids])
    # the weights' slices follow every way the parameters change
    b = ctx.collate(st, np.arange(G))
    ctx.train_step(b, 1e-2)
    ctx.forward(b, pred, train=False)
    after = pred.cpu().numpy()
    assert not np.array_equal(after, whole)
    fresh = g.Context(g.make_config(104, 2, G, gs.n_nodes, gs.n_edges, delta=st.delta(), flags=g.FLAG_ROW_INVARIANT))
    fresh.set_params(ctx.get_params())
    fresh.forward(fresh.collate(st, np.arange(G)), pred, train=False)
    assert np.array_equal(pred.cpu().numpy(), after)
    ctx.forward(b, train=True)
    ctx.backward(b)
    ctx.step(1e-2)
    ctx.forward(b, pred, train=False)
    assert not np.array_equal(pred.cpu().numpy(), after)
    ctx.check()


def test_captured_forward_follows_parameters(tmp_path):
    """A capture made after an eager forward slices the weights anew in every replay."""
    G = 110
    gs, ost, st, _, params = _setup(tmp_path, G, 18, 22, 64, 2)
    import paper_2207_11333_gb300 as g
    with torch.cuda.stream(torch.cuda.Stream()):
        ctx = g.Context(g.make_config(64, 2, G, gs.n_nodes, gs.n_edges, delta=st.delta()))
        ctx.set_params(params)
        b = ctx.collate(st, np.arange(G))
        pred = torch.empty(G, device="cuda")
        ctx.forward(b, pred, train=False)
        graph = torch.cuda.CUDAGraph()
        graph.capture_begin()
        ctx.forward(b, pred, train=False)
        graph.capture_end()
        for p in (params, synth.init_params(23, 64, 2)):
            ctx.set_params(p)
            graph.replay()
            torch.cuda.synchronize()
            replayed = pred.cpu().numpy()
            ctx.forward(b, pred, train=False)
            ctx.check()
            np.testing.assert_array_equal(replayed, pred.cpu().numpy())


@pytest.mark.parametrize("bad", [float("inf"), float("-inf"), float("nan")])
def test_non_finite_values(tmp_path, bad):
    """An infinite or undefined weight gives the plain path's activations: the
    same infinities and zeros, the rest to FP32 accuracy.  (Weights near the
    largest float are not comparable: there the last bit of a message decides
    whether the variance of equal neighbours is 0 or overflows.)"""
    G, H = 110, 72
    gs, ost, st, ctx, params = _setup(tmp_path, G, 18, 22, H, 2)
    p = params.copy()
    p[7 * H + 5] = bad  # W_M of layer 0, row 0, column 5
    ctx.set_params(p)
    b = ctx.collate(st, np.arange(G))
    acts = []
    for train in (True, False):
        ctx.forward(b, train=train)
        ctx.check()
        acts.append(ctx.activations(b)[1])
    plain, slices = acts
    fine = np.isfinite(plain)
    assert np.array_equal(fine, np.isfinite(slices))
    assert np.array_equal(plain[~fine & ~np.isnan(plain)], slices[~fine & ~np.isnan(plain)])
    scale = np.abs(plain[fine]).max()
    assert np.abs(plain[fine] - slices[fine]).max() <= FP32_FWD_TOL * scale
