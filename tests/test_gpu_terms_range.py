"""Matrices whose estimate leaves the fixed-point range while its terms are formed."""
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


def haf(gbs, mats, noalloc=False):
    flat, n, offs = gbs.pack_matrices(mats)
    out = torch.zeros(2 * len(mats), dtype=torch.float64, device="cuda")
    kap = torch.zeros(len(mats), dtype=torch.float64, device="cuda")
    f = gbs.hafnian_batch_noalloc if noalloc else gbs.hafnian_batch
    f(torch.from_numpy(flat).cuda(), n, offs, gbs.FP64, haf_out=out, kappa_out=kap)
    torch.cuda.synchronize()
    o = out.cpu().numpy()
    return o[0::2] + 1j * o[1::2], kap.cpu().numpy()


def hidden_powers(n, rng, eps=0.01):
    """D M D + noise, M of rank one and equal in two halves of the pairs, D = i on
    the second half: products over a pair of one half and its twin cancel, so
    the whole matrix's powers, from which the range is fixed, are 2 to 8 times
    smaller beside that range than those of subsets of one half."""
    h = n // 2
    q = h // 2
    twin = np.array([t % q if t < 2 * q else t for t in range(h)])
    v = np.exp(2j * np.pi * rng.random(n))[np.concatenate([twin, twin + h])]
    d = np.ones(n, complex)
    d[q:2 * q] = d[h + q:h + 2 * q] = 1j
    w = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    return np.outer(d * v, d * v) + eps * (w + w.T) / 2


@pytest.mark.parametrize("n,count", [(16, 200), (20, 3), (24, 5)])
def test_range_left_by_some_blocks_of_a_matrix(gbs, n, count):
    """Some of the blocks that share a matrix find it out of range: the FP64
    kernel's kappa, the same bits twice, and the matrices beside it untouched.
    The two kappas differ by the Hafnian's error in the subset sum, n 2^-53
    kappa relative, and by the moduli's, near 1e-15: 1e-12 leaves a factor of
    1000."""
    rng = np.random.default_rng(n)
    plain = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    mats = [hidden_powers(n, rng) for _ in range(count)] + [(plain + plain.T) / 2]
    h1, k1 = haf(gbs, mats)
    h2, k2 = haf(gbs, mats)
    assert np.array_equal(h1, h2) and np.array_equal(k1, k2)
    assert haf(gbs, mats[-1:])[1][0] == k1[-1]
    some = list(range(min(8, count))) + [count]
    _, k0 = haf(gbs, [mats[i] for i in some], noalloc=True)
    for ka, kb in zip(k1[some], k0):
        assert abs(ka - kb) <= (1e-12 + 2 * n * 2.0**-53 * kb) * kb, (ka, kb)
