"""Exact rescoring of candidates (K3) and of band pairs (K6) at the edges of its forms: rows that
are not whole 16-byte pieces or start off 16-byte boundaries, depths around the 8- and 32-column
groups, lists longer than one chunk, scores that FP32 cannot tell apart, integer sums beyond 32
bits.  Inputs are multiples of 2^-20 (off the 2^-12 grid, but every product and sum is exact in
FP64) or lie on the grid, so the oracle's values are exact and results must be identical."""
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


def dev(x, pad):
    """On the device with a row stride of d + pad; pad = -1: contiguous."""
    t = torch.from_numpy(np.ascontiguousarray(x)).cuda()
    if pad < 0:
        return t
    wide = torch.full((x.shape[0], x.shape[1] + pad), float("nan"), dtype=torch.float32, device="cuda")
    wide[:, :x.shape[1]] = t
    return wide[:, :x.shape[1]]


def check(ctx, U, P, k, pad=-1):
    tau_o, tid_o, topk_o = oracle.kmips(U, P, k)
    Ud, Pd = dev(U, pad), dev(P, pad)
    tau, tid, topk = ctx.thresholds(Ud, Pd, k, want_topk=True)
    tau2, tid2, _ = ctx.thresholds(Ud, Pd, k)
    for t, i in ((tau, tid), (tau2, tid2)):
        np.testing.assert_array_equal(t.cpu().numpy().view(np.uint64), tau_o.view(np.uint64))
        np.testing.assert_array_equal(i.cpu().numpy(), tid_o)
    np.testing.assert_array_equal(topk.cpu().numpy(), topk_o)
    sc = ctx.scores(Ud, Pd, tau, tid).cpu().numpy()
    np.testing.assert_array_equal(sc, oracle.scores_histogram(topk_o, P.shape[0]))
    ctx.resident_set(Ud, tau, tid)
    Q = P[: min(70, len(P))]
    np.testing.assert_array_equal(ctx.query_new_items(dev(Q, pad)).cpu().numpy(), oracle.query_new_items(U, tau_o, Q))


def fine(rng, n, d):
    """Entries in [-1, 1], multiples of 2^-20: off the grid, inner products exact in FP64."""
    return (rng.integers(-(1 << 20), (1 << 20) + 1, size=(n, d)) / float(1 << 20)).astype(np.float32)


@pytest.mark.parametrize("prec", ["bf16", "fp8", "fp32"])
@pytest.mark.parametrize("d,k,pad", [(1, 1, -1), (3, 5, 0), (8, 64, 1), (31, 2, 3), (32, 33, 4), (33, 10, -1),
                                     (100, 50, 2), (128, 7, -1), (200, 20, 4), (255, 11, -1), (256, 64, 0)])
def test_off_grid_depths_and_strides(rkm, prec, d, k, pad):
    rng = np.random.default_rng(d * 100 + k)
    U, P = fine(rng, 150, d), fine(rng, 700, d)
    with rkm.Context(prec) as ctx:
        check(ctx, U, P, k, pad)
        assert ctx.stats()["exact_integer_path"] == 0


@pytest.mark.parametrize("prec", ["bf16", "fp8"])
def test_off_grid_scores_fp32_cannot_tell_apart(rkm, prec):
    """Families of items that differ by 2^-20 in one entry, and exact duplicates: FP32 sums of a
    family are closer than their error bound, so FP64 values and ids decide."""
    rng = np.random.default_rng(3)
    base = fine(rng, 40, 100) * np.float32(0.5)
    P = np.repeat(base, 12, axis=0)
    at = rng.integers(0, 100, size=len(P))
    P[np.arange(len(P)), at] += (rng.integers(-1, 2, size=len(P)) / float(1 << 20)).astype(np.float32)
    U = fine(rng, 200, 100)
    with rkm.Context(prec) as ctx:
        for k in (1, 6, 30, 64):
            check(ctx, U, P, k)


@pytest.mark.parametrize("grid", [True, False])
@pytest.mark.parametrize("prec", ["bf16", "fp8"])
def test_lists_longer_than_a_chunk(rkm, prec, grid):
    """Hundreds of candidates per user: items of one direction whose scores lie within the guard
    band of each other (many of them equal), more than any threshold on the bounds separates."""
    rng = np.random.default_rng(11)
    dirn = rng.integers(1024, 4097, size=(1, 64)) / 4096.0
    step = 4096.0 if grid else float(1 << 20)
    P = np.rint(np.repeat(dirn, 900, axis=0) * step) / step
    P[np.arange(900), rng.integers(0, 64, 900)] -= rng.integers(0, 3, size=900) / step
    U = np.abs(fine(rng, 60, 64)) if not grid else rng.integers(1, 4097, size=(60, 64)) / 4096.0
    with rkm.Context(prec) as ctx:
        for k in (1, 25, 64):
            check(ctx, U.astype(np.float32), P.astype(np.float32), k)


@pytest.mark.parametrize("prec", ["bf16", "fp8"])
def test_integer_sums_beyond_32_bits(rkm, prec):
    """d = 256 rows of +-1 (grid code 4096): |sum| reaches 2^32."""
    rng = np.random.default_rng(5)
    U, P = np.ones((140, 256), np.float32), np.ones((300, 256), np.float32)
    U[70:] = -1.0
    P[rng.integers(0, 300, 200), rng.integers(0, 256, 200)] = 0.5
    P[250:] *= -1.0
    with rkm.Context(prec) as ctx:
        check(ctx, U, P, 20)
        assert ctx.stats()["exact_integer_path"] == 1


@pytest.mark.parametrize("scale", [2.0 ** 55, 2.0 ** -60])
def test_off_grid_magnitudes(rkm, scale):
    rng = np.random.default_rng(6)
    U, P = fine(rng, 130, 40), fine(rng, 400, 40)
    with rkm.Context("bf16") as ctx:
        check(ctx, (U * np.float32(scale)).astype(np.float32), (P * np.float32(scale)).astype(np.float32), 10)


@pytest.mark.parametrize("n", [1, 31, 33, 9_729, 40_001])
def test_users_per_warp(rkm, n):
    """Numbers of users around the steps of the users-per-warp rule."""
    W = workloads.mf(n, 600, 24, 5, 5, seed=n)
    off = (W.U * np.float32(1.0 + 2.0 ** -14)).astype(np.float32)  # 12-bit codes no longer hold it
    with rkm.Context("bf16") as ctx:
        for U in (W.U, off):
            tau_o, tid_o, _ = oracle.kmips(U, W.P, 5)
            tau, tid, _ = ctx.thresholds(dev(U, -1), dev(W.P, -1), 5)
            np.testing.assert_array_equal(tid.cpu().numpy(), tid_o)
            np.testing.assert_allclose(tau.cpu().numpy(), tau_o, rtol=1e-12, atol=1e-300)


@pytest.mark.parametrize("prec", ["bf16", "fp8", "fp32"])
def test_later_tiles_of_far_larger_subnormal_norms(rkm, prec):
    """All norms below 2^-133 share one bucket, so the first item tile can hold norms of 2^-149 only
    and a later one 32,764 times that.  The FP32 error bound must cover the later ones: the scores
    of a user lie so close that FP32 sums put them in another order than FP64 ones."""
    rng = np.random.default_rng(8)
    unit = np.float32(2.0 ** -149)
    P = np.zeros((2900, 64), np.float32)
    P[np.arange(2500), rng.integers(0, 64, 2500)] = unit
    codes = np.full((400, 64), 4095.0)
    for row in codes:
        row[rng.permutation(64)[:32]] += 1.0
    P[2500:] = (codes * 2.0 ** -149).astype(np.float32)
    # Entries 2^49 (1 + r 2^-19), r < 2^17: off the grid, sums exact in FP64.
    U = ((2.0 ** 19 + rng.integers(0, 1 << 17, size=(150, 64))) * 2.0 ** 30).astype(np.float32)
    with rkm.Context(prec) as ctx:
        for k in (1, 20):
            check(ctx, U, P, k)
            assert ctx.stats()["exact_integer_path"] == 0
            tau_o, _, _ = oracle.kmips(U, P, k)
            np.testing.assert_array_equal(ctx.query_new_items(dev(P, -1)).cpu().numpy(),
                                          oracle.query_new_items(U, tau_o, P))


@pytest.mark.parametrize("scale", [1.0, 2.0 ** 60])
@pytest.mark.parametrize("k", [1, 25])
def test_norms_and_sums_beyond_fp32(rkm, scale, k):
    """Users off the grid whose squared norms overflow FP32: no FP32 bound holds, so FP64 ranks all
    candidates and decides all pairs.  With items of 2^60 the FP32 sums overflow as well.  Entries are
    positive, so that the products overflow to infinity and not to NaN."""
    rng = np.random.default_rng(9)
    U, P = np.abs(fine(rng, 130, 40)) * np.float32(2.0 ** 70), np.abs(fine(rng, 400, 40)) * np.float32(scale)
    P[200:210] = P[190:200]  # equal scores: ids decide
    with rkm.Context("bf16") as ctx:
        check(ctx, U.astype(np.float32), P.astype(np.float32), k)
        assert ctx.stats()["exact_integer_path"] == 0
        tau_o, _, topk_o = oracle.kmips(U, P, k)
        ids, top = ctx.topn(dev(U, -1), dev(P, -1), k, 50)[:2]
        ids_o, top_o = oracle.topn(oracle.scores_histogram(topk_o, 400), 50)
        np.testing.assert_array_equal(ids.cpu().numpy(), ids_o)
        np.testing.assert_array_equal(top.cpu().numpy(), top_o)
