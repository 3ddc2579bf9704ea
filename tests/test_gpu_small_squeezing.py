"""Marginals and chain samples do not depend on the squeezing (identical on all modes)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SMALL = (1e-3, 1e-5, 1e-14, 1e-17, 1e-20, 1e-28, 1e-60, 1e-150, 1e-300)


@pytest.fixture(scope="module")
def gbs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1908_10070_gb300 as g

    return g


@pytest.mark.parametrize("n,k", [(4, 3), (12, 6), (16, 12), (20, 14), (20, 18), (20, 20)])
def test_marginals_are_the_same_at_any_squeezing(gbs, n, k):
    """Prefixes with tables in shared memory, in device memory, and taken set by
    set. q is a sum of positive terms of about n roundings each, and B's own
    rounding enters k times: 1e-12 as for the other marginal tests."""
    import workloads as W

    U = W.haar_unitary(24, 3)
    x = np.random.default_rng(k).integers(0, 24, size=(2, k)).astype(np.int32)
    ref = gbs.marginal_batch(gbs.build_kernel(U, np.full(24, 0.7)), x, n)
    for r in SMALL:
        q = gbs.marginal_batch(gbs.build_kernel(U, np.full(24, r)), x, n)
        assert np.all(np.abs(q - ref) <= 1e-12 * ref), (r, q, ref)


@pytest.mark.parametrize("n", [2, 8, 12, 20])
def test_chain_samples_are_the_same_at_any_squeezing(gbs, n):
    import workloads as W

    U = W.haar_unitary(24, 3)
    u = np.random.default_rng(n).random((6, n))
    ref = gbs.sample_chain_batch(gbs.build_kernel(U, np.full(24, 0.7)), n, u)
    for r in SMALL:
        assert np.array_equal(gbs.sample_chain_batch(gbs.build_kernel(U, np.full(24, r)), n, u), ref), r
