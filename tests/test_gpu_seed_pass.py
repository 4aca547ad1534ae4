"""The seed pass of the tensor-core threshold kernel (lower bounds of tau_u from maxima of 16 item
columns): the thresholds equal the oracle's where its rule begins and ends, for every number of
seed tiles, K-blocks per tile and parity of the user tiles that a CTA takes."""
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


# (n, m, d, k): item tiles around 12 (the fewest the rule takes), 24, 48 and 96; k around 16 and 32
CASES = [(300, 11 * 256, 24, 16, 0), (300, 12 * 256, 24, 16, 1), (300, 12 * 256, 24, 17, 0),
         (129, 24 * 256 + 3, 64, 31, 1), (129, 24 * 256, 128, 32, 1), (1, 48 * 256, 40, 64, 1),
         (700, 50 * 256, 200, 33, 1), (20_000, 97 * 256, 16, 10, 1), (20_000, 24 * 256, 256, 1, 1)]


@pytest.mark.parametrize("prec", ["bf16", "fp8"])
@pytest.mark.parametrize("n,m,d,k,seeded", CASES)
def test_seed_pass(rkm, prec, n, m, d, k, seeded):
    W = workloads.mf(n, m, d, k, 5, seed=n + m + d + k)
    sample = np.unique(np.linspace(0, n - 1, 400).astype(int))
    tau_o, tid_o, topk_o = oracle.kmips(W.U[sample], W.P, k, threads=8)
    U, P = torch.from_numpy(W.U).cuda(), torch.from_numpy(W.P).cuda()
    with rkm.Context(prec) as ctx:
        tau, tid, topk = (x.cpu().numpy() for x in ctx.thresholds(U, P, k, want_topk=True))
        if prec == "bf16":
            assert ctx.stats()["threshold_launches"] == 1 + seeded
    np.testing.assert_array_equal(tau[sample].view(np.uint64), tau_o.view(np.uint64))
    np.testing.assert_array_equal(tid[sample], tid_o)
    np.testing.assert_array_equal(topk[sample], topk_o)


@pytest.mark.parametrize("prec", ["bf16", "fp8"])
def test_seed_pass_negative_zero_and_equal_scores(rkm, prec):
    rng = np.random.default_rng(4)
    P = (rng.integers(1, 64, size=(13 * 256, 8)) / 64).astype(np.float32)
    P[1000:2600] = P[7]  # equal rows across several seed groups
    U = -(rng.integers(1, 64, size=(300, 8)) / 64).astype(np.float32)  # every score negative
    U[::5] = 0.0
    U[1::5] *= -1.0
    with rkm.Context(prec) as ctx:
        for k in (1, 9, 16):
            tau_o, tid_o, topk_o = oracle.kmips(U, P, k)
            tau, tid, topk = ctx.thresholds(torch.from_numpy(U).cuda(), torch.from_numpy(P).cuda(), k, want_topk=True)
            np.testing.assert_array_equal(tau.cpu().numpy().view(np.uint64), tau_o.view(np.uint64))
            np.testing.assert_array_equal(tid.cpu().numpy(), tid_o)
            np.testing.assert_array_equal(topk.cpu().numpy(), topk_o)
