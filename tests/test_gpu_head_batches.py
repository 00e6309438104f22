"""The head's forward on more graphs than the GPU has SMs (several graphs per
block and pass) against the same graphs in small batches (one block each): the
sums are made in the same order, so with row-invariant layers below the
predictions agree bit for bit.  Widths: one and several float4 columns, more
columns than threads of a warp, one that is no multiple of 4 (always one block
per graph) and one whose W1 does not fit in shared memory."""
import numpy as np
import pytest
import torch

import synth
from gpu_common import write_both
from helpers import graph_set

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("H,Hh", [(8, 4), (40, 36), (24, 132), (40, 35), (200, 200), (64, 1024)])
def test_many_graphs_equal_few(tmp_path, H, Hh, precision):
    import paper_2207_11333_gb300 as g
    G = 1221  # two passes of 152 blocks of four graphs, and a remainder
    gs = graph_set(3, G, 1, 40)
    path, _ = write_both(gs, str(tmp_path))
    st = g.Store(path)

    def predictions(ids):
        cfg = g.make_config(H, 1, len(ids), *map(int, st.batch_size(ids)), delta=st.delta(), head_hidden=Hh,
                            precision=precision, flags=g.FLAG_ROW_INVARIANT)
        ctx = g.Context(cfg)
        ctx.set_params(synth.init_params(4, H, 1, Hh=Hh))
        pred = torch.full((len(ids),), float("nan"), device="cuda")
        ctx.forward(ctx.collate(st, ids), pred, train=False)
        ctx.check()
        return pred.cpu().numpy()

    whole = predictions(np.arange(G))
    assert np.isfinite(whole).all()
    for a, b in ((0, 120), (600, 720), (G - 9, G)):
        assert np.array_equal(whole[a:b], predictions(np.arange(a, b)))
