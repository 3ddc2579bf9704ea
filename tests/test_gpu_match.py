"""The FP64 batched route: Hafnians by partial matchings and the subset sum's
terms (for kappa) in fixed point, at the sizes where they change over.

Tolerances. A Hafnian by matchings is a sum of products of h = n/2 entries with
at most n roundings on the way to each; on random matrices their effect grows
like the square root of that: 1e-13 leaves a factor of 50 at n = 30. kappa is
compared with the FP64 subset kernel's (gbs_hafnian_batch_noalloc, the same
pairing for n <= 24): its Hafnian's error, kappa 2^-53 n relative, dominates:
1e-10 as everywhere in these tests."""
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


def rand_sym(n, rng, scale=0.3):
    A = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    return scale * (A + A.T) / 2


def haf(gbs, mats, kappa=False, noalloc=False):
    flat, n, offs = gbs.pack_matrices(mats)
    A = torch.from_numpy(flat).cuda()
    out = torch.zeros(2 * len(mats), dtype=torch.float64, device="cuda")
    kap = torch.zeros(len(mats), dtype=torch.float64, device="cuda") if kappa else None
    (gbs.hafnian_batch_noalloc if noalloc else gbs.hafnian_batch)(A, n, offs, gbs.FP64, haf_out=out, kappa_out=kap)
    torch.cuda.synchronize()
    o = out.cpu().numpy()
    return o[0::2] + 1j * o[1::2], kap.cpu().numpy() if kappa else None


@pytest.mark.parametrize("n,count", [(2, 1), (2, 700), (4, 33), (6, 5), (10, 650), (16, 3), (16, 620), (18, 1), (18, 310),
                                     (20, 1), (20, 3), (22, 2), (26, 1)])
def test_matchings_match_oracle(gbs, n, count):
    """Tiles of one and of several matrices (the last one partly filled), the
    largest order in shared memory, the smallest ones in device memory."""
    import oracle

    rng = np.random.default_rng(n * 1000 + count)
    mats = [rand_sym(n, rng) for _ in range(count)]
    got, _ = haf(gbs, mats)
    for b in sorted({0, count // 2, count - 1}):
        ref = oracle.haf_subset(mats[b])
        assert abs(got[b] - ref) <= 1e-13 * abs(ref), (b, got[b], ref)


def test_matchings_ragged_batch_and_estimate_do_not_change_bits(gbs):
    """Every order 0..30 at once, each as it is alone, and with or without kappa."""
    rng = np.random.default_rng(7)
    mats = [rand_sym(n, rng) for n in range(0, 31)]
    got, _ = haf(gbs, mats)
    with_k, kap = haf(gbs, mats, kappa=True)
    assert np.array_equal(got, with_k)
    assert got[0] == 1 and np.all(got[1::2] == 0) and np.all(kap[2::2] >= 1)
    for n in (4, 18, 20, 28):
        assert haf(gbs, [mats[n]])[0][0] == got[n]


def scaled_rows(A, power):
    d = np.ldexp(1.0, power * (1 - 2 * (np.arange(len(A)) % 2)))
    return A * d[:, None] * d[None, :]


def special(kind, n, rng):
    A = rand_sym(n, rng)
    if kind == "zero_row":
        A[0, :] = A[:, 0] = 0
    elif kind == "rows_2^15":
        A = scaled_rows(A, 15)
    elif kind == "rows_2^4":
        A = scaled_rows(A, 4)
    elif kind == "huge":
        A = A * 1e30
    elif kind == "tiny":
        A = A * 1e-30
    elif kind == "subnormal":
        A = A * 1e-310
    elif kind == "ones":
        A = np.ones((n, n), complex)
    elif kind == "permutation":
        A = np.zeros((n, n), complex)
        p = rng.permutation(n)
        for i in range(0, n, 2):
            A[p[i], p[i + 1]] = A[p[i + 1], p[i]] = 1
    elif kind == "nan":
        A[0, 1] = A[1, 0] = np.nan
    elif kind == "inf":
        A[0, 1] = A[1, 0] = np.inf
    return A


@pytest.mark.parametrize("kind", ["random", "zero_row", "rows_2^15", "rows_2^4", "huge", "tiny", "subnormal", "ones",
                                  "permutation", "nan", "inf"])
def test_terms_match_fp64_kernel(gbs, kind):
    """kappa in fixed point against the FP64 subset kernel's, on matrices that
    fit the fixed-point range and on ones that must be given back to it."""
    rng = np.random.default_rng(3)
    orders = (2, 4, 6, 8, 10, 14, 16, 18, 20, 24)
    mats = [special(kind, n, rng) for n in orders] + [rand_sym(16, rng)]
    h1, k1 = haf(gbs, mats, kappa=True)
    h0, k0 = haf(gbs, mats, kappa=True, noalloc=True)
    for a, b, ka, kb, n in zip(h1, h0, k1, k0, list(orders) + [16]):
        if not np.isfinite(b):
            assert not np.isfinite(a), (n, a, b)
            continue
        if abs(b) == 0 or not np.isfinite(kb) or abs(a) == 0:
            # a zero Hafnian: the subset sum leaves rounding or zero there
            assert abs(a) <= 1e-10 * max(1.0, abs(b)) or kb > 1e10, (n, a, b)
            continue
        if kb < 1e6:
            assert abs(a - b) <= 1e-10 * abs(b) and abs(ka - kb) <= 1e-10 * kb, (n, a, b, ka, kb)


@pytest.mark.parametrize("m,n,k", [(9, 14, 11), (9, 14, 12), (7, 14, 13), (6, 16, 14), (6, 16, 15), (5, 20, 17), (5, 20, 18),
                                   (5, 20, 19)])
def test_marginals_sum_across_prefix_lengths(gbs, m, n, k):
    """sum_l q(x_1..x_k, l) = q(x_1..x_k): the tables in shared memory (up to 12
    photons), in device memory, and the sets taken one by one near k = n, with
    repeated modes. q is a sum of positive terms of about n roundings each:
    1e-12 leaves a factor of 100."""
    import workloads as W

    K = gbs.build_kernel(W.haar_unitary(m, 17 * m + n), np.full(m, 0.7))
    x = np.random.default_rng(n * k).integers(0, m, size=(3, k)).astype(np.int32)
    whole = gbs.marginal_batch(K, x, n)
    ext = np.repeat(x, m, axis=0)
    ext = np.hstack([ext, np.tile(np.arange(m, dtype=np.int32), 3)[:, None]])
    parts = gbs.marginal_batch(K, ext, n).reshape(3, m).sum(1)
    assert np.all(whole > 0) and np.all(np.abs(parts - whole) <= 1e-12 * whole), (whole, parts)


@pytest.mark.parametrize("kind,slots", [("haar", 256), ("haar", 3), ("blocks", 64), ("zero_modes", 64)])
def test_server_whole_requests_match_batch(gbs, kind, slots):
    """Requests that go as a whole (orders 2..30, several steps of them, few
    slots), on a device of equal modes, on one whose blocks of modes differ by
    9 orders of magnitude and on one with unsqueezed modes: the batched call's
    results within the two estimates, estimates equal to 1e-9 (sums of up to
    2^12 positive terms, 1e-15 each), the same bits alone and in the crowd, and
    as many terms counted as the subset sum has."""
    import scipy.linalg
    import workloads as W

    rng = np.random.default_rng(11)
    if kind == "haar":
        K = gbs.build_kernel(W.haar_unitary(60, 5), np.full(60, 0.8))
        pats = [rng.choice(60, size=n, replace=False) for n in list(range(2, 31)) * 3 + [30, 30, 30, 28]]
    else:
        U = scipy.linalg.block_diag(*[W.haar_unitary(12, s) for s in (1, 2, 3)])
        r = np.repeat([0.8, 1e-4, 1e-9] if kind == "blocks" else [0.8, 0.0, 0.5], 12)
        K = gbs.build_kernel(U, r)
        pats = [np.concatenate([12 * i + rng.choice(12, size=c, replace=False) for i, c in enumerate(cs)])
                for cs in [(6, 4, 4), (8, 6, 2), (2, 2, 2), (10, 10, 8), (4, 0, 6), (0, 8, 0), (12, 0, 0), (12, 8, 10)]]
    pats = [np.sort(x).astype(np.int32) for x in pats]
    srv = gbs.Server(K, max_slots=slots)

    def serve(xs):
        tickets, res = [srv.submit(x) for x in xs], []
        for t in tickets:
            while (q := srv.poll(t)) is None:
                pass
            res.append(q)
        return res

    try:
        got = serve(pats)
        terms = srv.stats()["subsets"]
        alone = [serve([x])[0] for x in pats[::5]]
    finally:
        srv.destroy()
    assert got[::5] == alone
    assert terms >= sum(2 ** (len(x) // 2) - 1 for x in pats if len(x) % 2 == 0)
    idx, n, offs = gbs.pack_patterns(pats)
    b = len(pats)
    p, h, err = np.zeros(b), np.zeros(2 * b), np.zeros(b)
    gbs.prob_batch(K, idx, n, offs, gbs.FP64, p_out=p, haf_out=h, err_out=err)
    for i, (pg, hg, eg) in enumerate(got):
        ref = complex(h[2 * i], h[2 * i + 1])
        # each estimate is relative to its own Hafnian, and infinite for one of 0
        tol = 1e-13 * abs(ref) + eg * abs(hg) + (err[i] * abs(ref) if ref else 0)
        assert hg == ref or abs(hg - ref) <= tol, (i, n[i], hg, ref, eg, err[i])
        if eg + err[i] > 1e-3:
            continue
        assert abs(pg - p[i]) <= 2.1 * (1e-13 + eg + err[i]) * p[i], (i, n[i], pg, p[i])
        # (a large order's estimate is that of the ordering chosen for it, by either call)
        assert eg == err[i] or n[i] >= 26 or abs(eg - err[i]) <= (1e-9 + eg + err[i]) * err[i], (i, n[i], eg, err[i])
