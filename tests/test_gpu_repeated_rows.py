"""The repeated-row sum's split of a pattern's terms: items of 1024, the high
digits' values over a block's warps, tables of the low digits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gbs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1908_10070_gb300 as g

    return g


# one value of the high digits and few, tables of one mode, of up to 256 low
# combinations exactly (3^3 * 9 = 243, 4^4 = 256), a last item of a few terms
REPS = [(30,), (24,), (17, 13), (12, 12), (6, 6, 6, 6), (8, 2, 2, 8), (3, 3, 3, 3, 3, 3, 3, 3), (2, 2, 2, 8, 4, 4),
        (1, 1, 1, 1, 1, 1, 14), (5, 5, 5, 5), (4, 4, 4, 4, 4, 4)]


def call(gbs, K, pats):
    idx, n, offs = gbs.pack_patterns(pats)
    b = len(pats)
    h, err = np.zeros(2 * b), np.zeros(b)
    gbs.prob_batch(K, idx, n, offs, gbs.FP64, haf_out=h, err_out=err)
    return h[0::2] + 1j * h[1::2], err


def test_splits_of_the_terms(gbs):
    """Against the oracle's exactly rounded sum of the same terms. Their errors
    add like the terms' moduli: err_est is n 2^-53 times those over |Haf|, and a
    term is a power of a sum of d products, with about n roundings: twice that
    estimate. The same bits alone and beside the others."""
    import oracle
    import workloads as W

    m = 10
    U, r = W.haar_unitary(m, 77), np.full(m, 0.9)
    K = gbs.build_kernel(U, r)
    B = oracle.build_B(U, r)
    rng = np.random.default_rng(5)
    pats = [np.sort(np.repeat(rng.choice(m, size=len(c), replace=False), c)).astype(np.int32) for c in REPS]
    h, err = call(gbs, K, pats)
    for x, a, e in zip(pats, h, err):
        modes, reps = np.unique(x, return_counts=True)
        ref = oracle.haf_repeated(B[np.ix_(modes, modes)], reps)
        assert abs(a - ref) <= 2 * e * abs(a) + 1e-15 * abs(ref), (reps, a, ref, e)
        h1, e1 = call(gbs, K, [x])
        assert h1[0] == a and e1[0] == e
