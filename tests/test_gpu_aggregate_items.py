"""Aggregation forward with several items per thread (batches large enough for it).

Every channel is reduced by itself, so a call over all channels (up to four items
per thread, stepping through rows whose width does not divide a block) has to give
the bits of a call over four of them (one item per thread).  Rows of degree 0, of
more edges than the registers keep, and a last block partly filled are included;
FP64 checks the values: a sum of at most seven messages of magnitude below 16
rounds by less than 7 x 7 x 16 x 2^-24 < 5e-5, the other aggregates by less."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

# float4 columns per row: 1, 3 (no divisor of 128), 50, 130 (more than a block);
# work items between 2 and 4 per thread and far above
SIZES = [(1_300_001, 4), (420_001, 12), (12_501, 200), (30_011, 200), (9_603, 520)]


@pytest.mark.parametrize("n,H", SIZES)
def test_items(n, H):
    import paper_2207_11333_gb300 as g
    rng = np.random.default_rng(n)
    deg = rng.integers(0, 8, n)
    deg[-1] = 7
    row = np.concatenate([[0], np.cumsum(deg)]).astype(np.int32)
    row_ptr = torch.from_numpy(row).cuda()
    col = torch.from_numpy(rng.integers(0, n, row[-1]).astype(np.int32)).cuda()
    PQ = torch.randn(n, 2 * H, device="cuda", generator=torch.Generator("cuda").manual_seed(n))
    agg = g.aggregate_fwd(PQ, row_ptr, col)
    c = (H // 4 // 2) * 4
    few = slice(0, min(n, 100_000))  # one item per thread: fewer rows as destinations, all as sources
    if n <= 100_000:
        part = torch.cat([PQ[:, c:c + 4], PQ[:, H + c:H + c + 4]], 1).contiguous()
        assert torch.equal(g.aggregate_fwd(part, row_ptr, col).view(n, 5, 4), agg.view(n, 5, H)[:, :, c:c + 4])
    a = agg.view(n, 5, H)[few].double().cpu().numpy()
    P, Q = PQ[:, :H].double().cpu().numpy(), PQ[:, H:].double().cpu().numpy()
    cols = col.cpu().numpy()
    for i in list(range(0, 300)) + list(range(a.shape[0] - 300, a.shape[0])):
        if deg[i] == 0:
            assert not a[i].any()
            continue
        m = P[i] + Q[cols[row[i]:row[i + 1]]]
        want = [m.sum(0), m.mean(0), m.min(0), m.max(0), np.sqrt(m.var(0) + 1e-5)]
        np.testing.assert_allclose(a[i], want, rtol=0, atol=5e-5)
    last = agg.view(n, 5, H)[-1].double().cpu().numpy()
    m = P[-1] + Q[cols[row[-2]:row[-1]]]
    np.testing.assert_allclose(last, [m.sum(0), m.mean(0), m.min(0), m.max(0), np.sqrt(m.var(0) + 1e-5)], rtol=0, atol=5e-5)
