"""sum |f|_1 of the error estimate where it is formed in FP64: the small orders,
and matrices that the fixed-point kernels cannot do.

kappa times the modulus of the Hafnian that comes with it is that sum, whatever
the Hafnian's own error. It adds moduli, so nothing cancels, and its relative
error is that of the terms: sums of products of at most h = n/2 entries, with
n roundings or so on the way to each, which grow like a square root when they
are independent. n 2^-52 leaves more than 4 over that for two quotients."""
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


def rand_sym(n, rng):
    A = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    return (A + A.T) / 2


def haf(gbs, mats, noalloc=False):
    flat, n, offs = gbs.pack_matrices(mats)
    out = torch.zeros(2 * len(mats), dtype=torch.float64, device="cuda")
    kap = torch.zeros(len(mats), dtype=torch.float64, device="cuda")
    f = gbs.hafnian_batch_noalloc if noalloc else gbs.hafnian_batch
    f(torch.from_numpy(flat).cuda(), n, offs, gbs.FP64, haf_out=out, kappa_out=kap)
    torch.cuda.synchronize()
    o = out.cpu().numpy()
    return o[0::2] + 1j * o[1::2], kap.cpu().numpy()


def moduli(A):
    """sum_S |f(X A_S)|_1 from the power traces, in long double (64 bits or more)."""
    n = len(A)
    h = n // 2
    pos = [p // 2 + (h if p % 2 else 0) for p in range(n)]
    A = A[np.ix_(pos, pos)].astype(np.clongdouble)
    A[np.arange(n), np.arange(n)] = 0
    total = np.longdouble(0)
    for S in range(1, 1 << h):
        rows = [2 * p + q for p in range(h) if S >> p & 1 for q in (0, 1)]
        M = A[np.ix_([r ^ 1 for r in rows], rows)]
        power, tr, c = M, [None], [np.clongdouble(1)]
        for k in range(1, h + 1):
            tr.append(np.trace(power))
            c.append(sum(tr[i] * c[k - i] for i in range(1, k + 1)) / (2 * k))
            power = (power[:, :, None] * M[None, :, :]).sum(1)
        total += abs(c[h].real) + abs(c[h].imag)
    return total


@pytest.mark.parametrize("n,count", [(2, 1), (2, 300), (4, 1), (4, 70), (6, 33), (8, 17), (10, 1), (10, 9)])
def test_small_orders_keep_double_precision(gbs, n, count):
    """Blocks of one and of many matrices, the last one partly filled."""
    rng = np.random.default_rng(100 * n + count)
    mats = [rand_sym(n, rng) for _ in range(count)]
    h, kappa = haf(gbs, mats)
    for b in sorted({0, 1 % count, count // 2, count - 1}):
        K = moduli(mats[b])
        assert abs(kappa[b] * abs(h[b]) - K) <= n * 2.0**-52 * K, (b, kappa[b] * abs(h[b]), K)


def unequal_rows(n, rng):
    """Rows 2^30 apart in size: fixed point has no room for them."""
    d = np.ldexp(1.0, 15 * (1 - 2 * (rng.permutation(n) % 2)))
    A = rand_sym(n, rng)
    return A * d[:, None] * d[None, :], A


@pytest.mark.parametrize("n,count", [(4, 2), (12, 3), (14, 3), (16, 5), (18, 1), (18, 6), (20, 2), (24, 2)])
def test_matrices_without_a_fixed_point_range(gbs, n, count):
    """Scaled rows scale the Hafnian by exact powers of two, a zero row makes it
    0; sum |f| is the FP64 subset kernel's (both by the bound above), beside
    matrices that stay in fixed point."""
    rng = np.random.default_rng(n + count)
    pairs = [unequal_rows(n, rng) for _ in range(count)]
    zero = rand_sym(n, rng)
    zero[1, :] = zero[:, 1] = 0
    plain = rand_sym(n, rng)
    mats = [p[0] for p in pairs] + [zero, plain, rand_sym(4, rng)]
    h, kappa = haf(gbs, mats)
    assert np.array_equal(h[:count], haf(gbs, [p[1] for p in pairs])[0])  # prod of the scales is 1
    assert h[count] == 0 and kappa[count] == np.inf
    assert kappa[count + 1] == haf(gbs, [plain])[1][0]
    h0, k0 = haf(gbs, [p[0] for p in pairs], noalloc=True)
    for b in range(count):
        K, K0 = kappa[b] * abs(h[b]), k0[b] * abs(h0[b])
        assert abs(K - K0) <= 2 * n * 2.0**-52 * K0, (b, K, K0)


def test_served_requests_without_a_fixed_point_range_count_once(gbs):
    """Blocks of modes 9 orders of magnitude apart: the batched call's results,
    the same bits, and as many subset terms counted as the subset sum has."""
    import scipy.linalg
    import workloads as W

    U = scipy.linalg.block_diag(*[W.haar_unitary(12, s) for s in (1, 2, 3)])
    K = gbs.build_kernel(U, np.repeat([0.8, 1e-4, 1e-9], 12))
    rng = np.random.default_rng(12)
    pats = [np.sort(np.concatenate([12 * i + rng.choice(12, size=c, replace=False) for i, c in enumerate(cs)])).astype(np.int32)
            for cs in [(6, 4, 4), (8, 6, 2), (2, 2, 2), (2, 0, 0), (10, 10, 4), (4, 0, 6), (0, 8, 0), (12, 2, 10)] * 3]
    srv = gbs.Server(K, max_slots=16)
    try:
        tickets, got = [srv.submit(x) for x in pats], []
        for t in tickets:
            while (q := srv.poll(t)) is None:
                pass
            got.append(q)
        stats = srv.stats()
    finally:
        srv.destroy()
    assert stats["completed"] == len(pats)
    assert stats["subsets"] == sum(2 ** (len(x) // 2) - 1 for x in pats)
    idx, n, offs = gbs.pack_patterns(pats)
    b = len(pats)
    p, h, err = np.zeros(b), np.zeros(2 * b), np.zeros(b)
    gbs.prob_batch(K, idx, n, offs, gbs.FP64, p_out=p, haf_out=h, err_out=err)
    assert [q[0] for q in got] == list(p) and [q[2] for q in got] == list(err)


@pytest.mark.parametrize("graphs", [1, -1])
def test_server_wall_time_covers_device_time(gbs, graphs):
    """A step's wall time runs from the start of its launch to its detected
    completion, so it is no shorter than its time on the device."""
    import workloads as W

    K = gbs.build_kernel(W.haar_unitary(60, 5), np.full(60, 0.8))
    rng = np.random.default_rng(4)
    srv = gbs.Server(K, use_graphs=graphs)
    try:
        for n in (4, 12, 16, 20, 24) * 4:
            t = srv.submit(np.sort(rng.choice(60, size=n, replace=False)).astype(np.int32))
            while srv.poll(t) is None:
                pass
        stats = srv.stats()
    finally:
        srv.destroy()
    assert stats["step_wall_s"] >= stats["step_device_s"] > 0, stats
