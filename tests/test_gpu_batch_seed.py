"""The shared seed launch of a batch: several seeded instances (2 to 16 seed tiles, one to four
K-blocks a tile, k around 16 and 32) beside one that the seed rule leaves out, and more user tiles than
SMs, so that a CTA goes from one instance's unit to another's.  A seed above tau_u would lose members of
S_k(u): every instance's top N equals the oracle's, also when the captured graph is replayed."""
import numpy as np
import pytest

import oracle
import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# (n, m, d, k, N)
SHAPES = [(7000, 12 * 256, 32, 5, 50), (700, 300, 64, 10, 20), (6001, 24 * 256 + 3, 128, 16, 50),
          (5000, 50 * 256, 200, 33, 50), (129, 97 * 256, 16, 10, 20), (4000, 25 * 256 - 1, 64, 1, 50)]


@pytest.fixture(scope="module")
def rkm():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2504_13445_gb300 as m
    return m


@pytest.fixture(scope="module")
def problems():
    out = []
    for j, (n, m, d, k, N) in enumerate(SHAPES):
        W = workloads.mf(n, m, d, k, N, seed=900 + j)
        _, _, topk = oracle.kmips(W.U, W.P, k, threads=8)
        out.append((torch.from_numpy(W.U).cuda(), torch.from_numpy(W.P).cuda(), k, N,
                    oracle.topn(oracle.scores_histogram(topk, m), N)))
    return out


@pytest.mark.parametrize("prec", ["bf16", "fp8"])
@pytest.mark.parametrize("order", [1, -1])
def test_several_seeded_instances(rkm, problems, prec, order):
    probs = problems[::order]
    with rkm.Context(prec) as ctx:
        outs = None
        for _ in range(3):
            outs = ctx.topn_batch([p[:4] for p in probs], outs)
            torch.cuda.synchronize()
            for (ids, sc), p in zip(outs, probs):
                np.testing.assert_array_equal(ids.cpu().numpy(), p[4][0])
                np.testing.assert_array_equal(sc.cpu().numpy(), p[4][1])
        assert ctx.stats()["retries"] == 0
