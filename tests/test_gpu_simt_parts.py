"""FP32 path: the item tiles of a user tile are split into up to four parts (four for few users,
one from about 155,000 on a GPU of 152 SMs), each with two selectors per user.  Edges: users of a
partial tile, fewer item tiles than parts, a last tile of one item, k around the 32 of the warm
start, and every number of parts.  Integer entries: results must be identical to the oracle's."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rkm():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2504_13445_gb300 as m
    return m


@pytest.mark.parametrize("n,m,d,k", [(1, 64, 5, 64), (127, 127, 8, 1), (128, 128, 33, 16), (129, 129, 64, 32),
                                     (300, 385, 64, 33), (300, 513, 100, 64), (500, 1_025, 256, 10),
                                     (1_000, 2_000, 16, 64), (20_001, 640, 7, 20), (60_000, 300, 6, 5),
                                     (80_000, 300, 6, 33), (160_000, 257, 4, 2)])
def test_parts(rkm, n, m, d, k):
    rng = np.random.default_rng(n + m)
    U = rng.integers(-60, 61, size=(n, d)).astype(np.float32)
    P = rng.integers(-60, 61, size=(m, d)).astype(np.float32)
    P *= rng.integers(1, 9, size=(m, 1)).astype(np.float32)  # norms over three octaves: tiles stop early
    tau_o, tid_o, topk_o = oracle.kmips(U, P, k)
    want = oracle.scores_histogram(topk_o, m)
    Ud, Pd = torch.from_numpy(U).cuda(), torch.from_numpy(P).cuda()
    with rkm.Context("fp32") as ctx:
        tau, tid, _ = ctx.thresholds(Ud, Pd, k)
        np.testing.assert_array_equal(tau.cpu().numpy(), tau_o)
        np.testing.assert_array_equal(tid.cpu().numpy(), tid_o)
        np.testing.assert_array_equal(ctx.scores(Ud, Pd, tau, tid).cpu().numpy(), want)
        ids, sc = ctx.topn(Ud, Pd, k, min(m, 20))[:2]
        np.testing.assert_array_equal(sc.cpu().numpy(), np.sort(want)[::-1][:min(m, 20)])
        np.testing.assert_array_equal(want[ids.cpu().numpy()], sc.cpu().numpy())


@pytest.mark.parametrize("prec", ["fp32", "bf16", "fp8"])
@pytest.mark.parametrize("n,m,d,k,N", [(129, 300, 3, 10, 300), (500, 1_025, 8, 25, 400), (2_001, 3_000, 9, 5, 1_500)])
def test_top_n_ids_among_equal_scores(rkm, prec, n, m, d, k, N):
    """Most items share their score with others, and N cuts through such a group: ids decide."""
    rng = np.random.default_rng(n)
    U = rng.integers(-9, 10, size=(n, d)).astype(np.float32)
    P = rng.integers(-9, 10, size=(m, d)).astype(np.float32)
    _, _, topk_o = oracle.kmips(U, P, k)
    ids_o, top_o = oracle.topn(oracle.scores_histogram(topk_o, m), N)
    with rkm.Context(prec) as ctx:
        ids, top = ctx.topn(torch.from_numpy(U).cuda(), torch.from_numpy(P).cuda(), k, N)[:2]
    np.testing.assert_array_equal(ids.cpu().numpy(), ids_o)
    np.testing.assert_array_equal(top.cpu().numpy(), top_o)
