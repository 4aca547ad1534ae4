"""The epilogues of the product kernels at their edges: chunks in which most values hit, candidate
lists that fill inside a chunk, band pairs that fill a warp's stage many times, item counts
around the 32-, 64- and 256-column steps, and user counts that give a counting CTA units of
several item tiles.  Scores against the oracle on every path."""
import numpy as np
import pytest

import oracle
import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rkm():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2504_13445_gb300 as m
    return m


def check(ctx, U, P, k):
    tau_o, tid_o, topk_o = oracle.kmips(U, P, k)
    Ud, Pd = torch.from_numpy(U).cuda(), torch.from_numpy(P).cuda()
    tau, tid, topk = ctx.thresholds(Ud, Pd, k, want_topk=True)
    np.testing.assert_array_equal(tau.cpu().numpy().view(np.uint64), tau_o.view(np.uint64))
    np.testing.assert_array_equal(tid.cpu().numpy(), tid_o)
    np.testing.assert_array_equal(topk.cpu().numpy(), topk_o)
    sc = ctx.scores(Ud, Pd, tau, tid).cpu().numpy()
    np.testing.assert_array_equal(sc, oracle.scores_histogram(topk_o, P.shape[0]))


@pytest.mark.parametrize("groups", [0, 2, 4])
@pytest.mark.parametrize("prec", ["bf16", "fp8", "fp32"])
@pytest.mark.parametrize("n,m,d,k", [(128, 31, 8, 31), (129, 33, 16, 33), (127, 64, 64, 64), (257, 65, 65, 1),
                                     (640, 255, 40, 40), (300, 257, 130, 64), (4_000, 2_049, 20, 25)])
def test_item_edges(rkm, prec, groups, n, m, d, k):
    W = workloads.mf(n, m, d, min(k, m), 1, seed=n + m)
    with rkm.Context(prec, epilogue_groups=groups) as ctx:
        check(ctx, W.U, W.P, min(k, m))


@pytest.mark.parametrize("prec", ["bf16", "fp8", "fp32"])
def test_every_value_in_the_band(rkm, prec):
    """Items equal to within the guard band: every pair is a hit, the candidate lists overflow and
    grow inside a chunk, and every pair goes through the band stage."""
    rng = np.random.default_rng(8)
    base = rng.integers(2048, 4097, size=(1, 48)) / 4096.0
    P = np.repeat(base, 1_100, axis=0)
    P[np.arange(1_100), rng.integers(0, 48, 1_100)] -= rng.integers(0, 2, 1_100) / 4096.0
    U = rng.integers(1024, 4097, size=(200, 48)) / 4096.0
    with rkm.Context(prec, cand_capacity=32, band_capacity=1_000) as ctx:
        check(ctx, U.astype(np.float32), P.astype(np.float32), 20)


@pytest.mark.parametrize("prec", ["bf16", "fp8"])
def test_units_over_several_tiles(rkm, prec):
    """Counting units of one CTA that skip item tiles, stay in one, and lie in the next: few and many
    user tiles per item tile."""
    for n, m in ((100, 20_000), (5_000, 3_000), (30_000, 700)):
        W = workloads.mf(n, m, 12, 10, 1, seed=n)
        with rkm.Context(prec) as ctx:
            check(ctx, W.U, W.P, 10)
