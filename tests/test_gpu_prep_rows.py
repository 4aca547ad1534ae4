"""Row preparation (K1): norms, grid codes and the BF16 operand of a row in one pass, eight columns
a lane.  Edges: rows that start off 16-byte boundaries, the last column group, users of a partial
tile, exponents whose scaling is not one normal float, retries (which pack over the operand rows)
and slices (whose users start inside them).  Entries are exact in FP64 sums, so results must be
identical to the oracle's."""
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


def ints(rng, n, d, scale=0):
    """Integers up to 2^10 times 2^scale: on the grid, squares and inner products exact."""
    return np.ldexp(rng.integers(-1024, 1025, size=(n, d)).astype(np.float32), scale).astype(np.float32)


def dev(x, lead, pad):
    """Rows of x at an offset of lead floats, row stride d + pad, NaN around them."""
    n, d = x.shape
    flat = torch.full((lead + n * (d + pad) + 8,), float("nan"), dtype=torch.float32, device="cuda")
    v = flat[lead:lead + n * (d + pad)].view(n, d + pad)[:, :d]
    v.copy_(torch.from_numpy(x))
    return v


def check(ctx, U, P, k, N, lead=0, pad=0):
    tau_o, tid_o, topk_o = oracle.kmips(U, P, k)
    Ud, Pd = dev(U, lead, pad), dev(P, lead, pad)
    for _ in range(2):
        tau, tid, _ = ctx.thresholds(Ud, Pd, k)
        np.testing.assert_array_equal(tau.cpu().numpy(), tau_o)
        np.testing.assert_array_equal(tid.cpu().numpy(), tid_o)
    want = oracle.scores_histogram(topk_o, P.shape[0])
    ids, sc = ctx.topn(Ud, Pd, k, N)[:2]
    np.testing.assert_array_equal(sc.cpu().numpy(), np.sort(want)[::-1][:N])
    np.testing.assert_array_equal(want[ids.cpu().numpy()], sc.cpu().numpy())


@pytest.mark.parametrize("prec", ["bf16", "fp8", "fp32"])
@pytest.mark.parametrize("n,d,lead,pad", [(1, 1, 1, 0), (127, 7, 0, 1), (128, 8, 0, 0), (129, 9, 4, 3), (300, 63, 3, 1),
                                          (300, 64, 4, 4), (257, 65, 0, 3), (200, 129, 2, 3), (130, 200, 4, 0),
                                          (130, 255, 0, 1), (130, 256, 1, 0)])
def test_alignment_and_edges(rkm, prec, n, d, lead, pad):
    rng = np.random.default_rng(n + d)
    with rkm.Context(prec) as ctx:
        check(ctx, ints(rng, n, d), ints(rng, 600, d), 5, 20, lead, pad)


@pytest.mark.parametrize("prec", ["bf16", "fp32"])
@pytest.mark.parametrize("scale", [-130, -100, 40])
def test_exponents(rkm, prec, scale):
    """Users at each end of FP32's exponents (below 2^-114 the scaling is no normal float)."""
    rng = np.random.default_rng(scale & 255)
    U, P = ints(rng, 140, 40, scale), ints(rng, 500, 40)
    with rkm.Context(prec) as ctx:
        check(ctx, U, P, 3, 10)


def test_retry(rkm):
    """Lists of 32 slots overflow under 3,000 equal items until they have grown to 2,048."""
    rng = np.random.default_rng(5)
    U, P = ints(rng, 300, 100), np.repeat(ints(rng, 1, 100), 3000, axis=0)
    with rkm.Context("bf16", cand_capacity=32) as ctx:
        check(ctx, U, P, 10, 20)


def test_slices(rkm):
    """Lists of 2^22 slots leave room for a few hundred users at a time in the list budget (48 GB)."""
    rng = np.random.default_rng(6)
    with rkm.Context("bf16", cand_capacity=1 << 22) as ctx:
        check(ctx, ints(rng, 1000, 100), ints(rng, 700, 100), 10, 20)
