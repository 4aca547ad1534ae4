"""The Cauchy-Schwarz stop of the threshold pass at its tightest: with d = 1 every product reaches
||u|| ||p||.  Items are ordered by 16-bit norm buckets only, so among the several tiles of one
bucket a later tile may hold the largest norm; the stop must not end before it."""
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


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("k", [1, 3])
def test_largest_norm_in_a_later_tile_of_its_bucket(rkm, prec, k):
    U = np.array([[1.0], [0.75], [0.5]], np.float32)
    with rkm.Context(prec) as ctx:
        for m in range(60_000, 120_000, 3_000):
            rng = np.random.default_rng(m)
            P = rng.uniform(0.5, 1.0, size=(m, 1)).astype(np.float32)
            tau_o, tid_o, topk_o = oracle.kmips(U, P, k)
            tau, tid, topk = ctx.thresholds(torch.from_numpy(U).cuda(), torch.from_numpy(P).cuda(), k, want_topk=True)
            np.testing.assert_array_equal(topk.cpu().numpy(), topk_o)
            np.testing.assert_array_equal(tid.cpu().numpy(), tid_o)
            np.testing.assert_array_equal(tau.cpu().numpy(), tau_o)
