"""The top-N select and the bucket sort where they can go wrong: scores that decide at the first digit,
ties at the N-th place that only ids decide, N = 1 and the largest N; key counts around the one-block
sort's limit and the blocks' chunks, and keys that all fall into one bucket."""
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


@pytest.mark.parametrize("m", [1, 255, 1_025, 5_000])
@pytest.mark.parametrize("kind", ["zero", "equal", "spread", "two", "wide"])
def test_top_n_select(rkm, m, kind):
    rng = np.random.default_rng(m)
    score = {"zero": np.zeros(m), "equal": np.full(m, 3), "spread": rng.permutation(m) % 700,
             "two": np.where(np.arange(m) % 3 == 0, 257, 256), "wide": (rng.random(m) < 0.01) * 70_000}[kind].astype(int)
    lists = torch.from_numpy(np.repeat(np.arange(m), score).astype(np.int32)).cuda().reshape(-1, 1)
    with rkm.Context("bf16") as ctx:
        for N in sorted({1, min(7, m), min(m, 1_024), min(m, 4_096)}):
            ids, top = ctx.topn_from_topk(lists, m, 1, N)
            ids_o, top_o = oracle.topn(score, N)
            np.testing.assert_array_equal(ids.cpu().numpy(), ids_o)
            np.testing.assert_array_equal(top.cpu().numpy(), top_o)


@pytest.mark.parametrize("n", [1, 1_023, 16_384, 16_385, 40_000, 200_000])
@pytest.mark.parametrize("same", [False, True])
def test_bucket_sort(rkm, n, same):
    """Users in ratio order (ascending) and items by norm (descending): scores of a small catalogue and
    Eq. 2 bounds, which read the order and the prefix counts."""
    rng = np.random.default_rng(n)
    P = (rng.integers(-4096, 4097, size=(70, 4)) / 4096).astype(np.float32)
    U = (rng.integers(-4096, 4097, size=(1 if same else n, 4)) / 4096).astype(np.float32)
    U = np.repeat(U, n, axis=0) if same else U
    tau_o, tid_o, topk_o = oracle.kmips(U, P, 5)
    with rkm.Context("bf16") as ctx:
        Ud, Pd = torch.from_numpy(U).cuda(), torch.from_numpy(P).cuda()
        tau, tid, _ = ctx.thresholds(Ud, Pd, 5)
        np.testing.assert_array_equal(tau.cpu().numpy().view(np.uint64), tau_o.view(np.uint64))
        np.testing.assert_array_equal(tid.cpu().numpy(), tid_o)
        sc = ctx.scores(Ud, Pd, tau, tid).cpu().numpy()
        np.testing.assert_array_equal(sc, oracle.scores_histogram(topk_o, 70))
        assert np.all(ctx.item_bounds(Ud, Pd, tau).cpu().numpy() >= sc)
        if same and n > 2_000:
            return  # that many equal items are more candidates than a call's retries hold
        # the same rows as items: a catalogue of n, every norm in one bucket or in many
        tau2, tid2, _ = ctx.thresholds(Pd, Ud, 1)
        tau2_o, tid2_o, _ = oracle.kmips(P[:20], U, 1)
        np.testing.assert_array_equal(tau2.cpu().numpy()[:20].view(np.uint64), tau2_o.view(np.uint64))
        np.testing.assert_array_equal(tid2.cpu().numpy()[:20], tid2_o)
