"""What a user of the library runs: its public entry points over the sizes they are called at.

Every case is a dict with a "kind":

  prob      gbs.prob_batch: `count` patterns over `m` modes with n_lo..n_hi
            photons (every `n_step`-th number), squeezing r_lo..r_hi per mode.
            `spread` is how the photons fall ("free": no mode twice, "cap3": at
            most 3 in a mode, "any": with replacement), `outs` the outputs that
            are asked for, `host` whether lists and outputs are host arrays.
  haf       gbs.hafnian_batch: `count` random symmetric matrices of orders
            n_lo..n_hi, the Hafnians alone.
  marginal  gbs.marginal_batch: the marginals of every mode after one prefix.
  chain     gbs.sample_chain_batch: `count` samples of n photons.
  brute     gbs.sample_bruteforce: `count` draws over all configurations.
  serve     a gbs.Server that answers `count` requests handed in at once.
"""
import math

import numpy as np
import torch

import paper_1908_10070_gb300 as gbs

PREC = {"fp64": gbs.FP64, "mixed": gbs.MIXED}


def _prob(name, **kw):
    c = dict(name=name, kind="prob", m=64, n_lo=16, n_hi=16, n_step=2, count=1, r_lo=0.88, r_hi=0.88,
             spread="free", prec="fp64", outs="p,haf,err", host=False)
    c.update(kw)
    return c


def listed():
    return [
        # one probability at a time, lists and results on the host: the call of
        # the README, and what a per-pattern client sends; latency is all
        _prob("one_pattern_n16", r_lo=0.6, r_hi=1.0, host=True),
        # every small pattern of an 8-mode device (checks of p(s) sums): many
        # tiny orders, the vacuum and odd photon numbers among them
        _prob("tiny_ragged_m8", m=8, n_lo=0, n_hi=8, n_step=1, count=107, r_lo=0.5, r_hi=0.5, spread="cap3",
              outs="p,logp", host=True),
        # the library's headline workload: probabilities of 16-photon patterns
        # with all outputs, everything on the device
        _prob("batch_n16_fp64", count=4096, r_lo=0.6, r_hi=1.0, outs="p,logp,haf,err"),
        # the same in the mixed precision that a caller may choose
        _prob("batch_n16_mixed", count=4096, r_lo=0.6, r_hi=1.0, prec="mixed", outs="p,logp,haf,err"),
        # likelihoods of measured patterns: ragged photon numbers, collisions,
        # probabilities and their logarithms without the error estimate
        _prob("ragged_m144_fp64", m=144, n_lo=8, n_hi=24, count=2048, spread="cap3", outs="p,logp"),
        # the largest orders: a 900-mode interferometer, 28 and 30 photons (the
        # probabilities are near 1e-200: their logarithms are what is used)
        _prob("large_m900_fp64", m=900, n_lo=28, n_hi=30, count=80, r_lo=1.0, r_hi=1.0, outs="logp,haf,err"),
        # photons bunched into few modes (a small interferometer, strong pump)
        _prob("bunched_n24_m8", m=8, n_lo=24, n_hi=24, count=512, r_lo=1.0, r_hi=1.0, spread="any", host=True),
        # Hafnians of explicit matrices (graph problems, other Gaussian states):
        # every order up to 22, odd ones among them
        dict(name="haf_ragged_fp64", kind="haf", n_lo=1, n_hi=22, count=301),
        # conditional weights of one step of the chain rule: all modes after a
        # prefix of 8 photons
        dict(name="marginal_n16_k9", kind="marginal", m=256, n=16, k=9),
        # position-basis samples in the m = n^2 setting, many at once
        dict(name="chain_n16_m256", kind="chain", m=256, n=16, count=64),
        # the paper's brute-force check: every 4-photon configuration of 16 modes
        dict(name="brute_n4_m16", kind="brute", m=16, n=4, count=400000, prec="fp64"),
        # a burst of single-pattern requests of mixed sizes through the server
        dict(name="serve_burst_m256", kind="serve", m=256, n_lo=12, n_hi=26, count=384, prec="fp64"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _subset_cost(n):
    """Size of the subset sum of one matrix, for drawing batches of bounded cost."""
    return 2.0 ** (n // 2) * max(n, 4) ** 3


def draw(rng):
    kind = rng.choice(["prob"] * 6 + ["haf", "marginal", "chain", "brute", "serve"])
    if kind in ("prob", "haf"):
        # 2.5e10: below large_m900_fp64
        n_hi = rng.choice([4, 8, 11, 14, 16, 18, 20, 22, 24, 26, 28, 30])
        n_lo = n_hi if rng.random() < 0.4 else rng.randint(max(0, n_hi - 12), n_hi)
        count = max(1, min(_log(rng, 1, 5000), int(2.5e10 / _subset_cost(n_hi))))
        if count < 8:
            n_lo = n_hi
        step = rng.choice([1, 2])
        if n_lo % 2 and (n_lo == n_hi or step == 2):
            n_lo -= 1  # not odd photon numbers alone: their probabilities are all 0
        if kind == "haf":
            return dict(kind="haf", n_lo=n_lo, n_hi=min(n_hi, 26), count=min(count, 1500))
        spread = rng.choice(["free", "free", "cap3", "any"])
        m = _log(rng, max(8, n_hi), 600) if spread != "any" else rng.randint(6, 40)
        r = rng.uniform(0.3, 1.1)
        c = _prob("", m=m, n_lo=n_lo, n_hi=n_hi, n_step=step, count=count, r_lo=round(0.7 * r, 3),
                  r_hi=round(r, 3), spread=spread, prec=rng.choice(["fp64"] * 4 + ["mixed"]),
                  outs=rng.choice(["p,haf,err", "p,logp", "p", "p,logp,haf,err", "haf"]), host=rng.random() < 0.4)
        del c["name"]
        return c
    if kind == "marginal":
        n = 2 * rng.randint(2, 9)
        return dict(kind="marginal", m=rng.randint(20, 400), n=n, k=rng.randint(2, min(n, 13)))
    if kind == "chain":
        n = 2 * rng.randint(2, 8)
        return dict(kind="chain", m=rng.randint(n, 300), n=n, count=_log(rng, 1, 100))
    if kind == "brute":
        n, m = rng.choice([(2, 60), (4, 20), (6, 12), (8, 8)])
        return dict(kind="brute", m=rng.randint(m // 2, m), n=n, count=_log(rng, 10, 400000), prec="fp64")
    n_hi = rng.randint(8, 26)
    return dict(kind="serve", m=_log(rng, 32, 400), n_lo=rng.randint(2, n_hi - 1), n_hi=n_hi, count=_log(rng, 8, 384),
                prec=rng.choice(["fp64", "fp64", "mixed"]))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _haar(m, rng):
    """Haar-random unitary: QR of a Ginibre matrix with the phases of R's diagonal moved to Q."""
    z = torch.from_numpy(rng.standard_normal((m, m)) + 1j * rng.standard_normal((m, m))).cuda()
    q, r = torch.linalg.qr(z)
    d = torch.diagonal(r)
    return (q * (d / d.abs())[None, :]).contiguous()


def _patterns(case, rng):
    m, free = case["m"], case["spread"] == "free"
    numbers = [n for n in range(case["n_lo"], case["n_hi"] + 1, case["n_step"]) if not free or n <= m]
    if case["spread"] == "cap3":
        numbers = [n for n in numbers if n <= 2 * m]
    pats = []
    for _ in range(case["count"]):
        n = int(numbers[rng.integers(len(numbers))])
        if free:
            x = rng.choice(m, size=n, replace=False)
        else:
            x = rng.integers(0, m, size=n)
            while case["spread"] == "cap3" and n and np.bincount(x).max() > 3:
                x = rng.integers(0, m, size=n)
        pats.append(np.sort(x).astype(np.int32))
    return pats


def _inputs(case, seed):
    """The case's numbers, from the seed alone."""
    rng = np.random.default_rng([seed, 1908])
    kind, d = case["kind"], {}
    if kind == "haf":
        mats = []
        for _ in range(case["count"]):
            n = int(rng.integers(case["n_lo"], case["n_hi"] + 1))
            z = (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))) / math.sqrt(2.0)
            mats.append((z + z.T) / math.sqrt(2.0))
        d["mats"] = mats
        return d
    d["U"] = _haar(case["m"], rng)
    lo, hi = (case["r_lo"], case["r_hi"]) if kind == "prob" else (0.88, 0.88)
    d["r"] = np.full(case["m"], lo) if lo == hi else rng.uniform(lo, hi, size=case["m"])
    if kind == "prob":
        d["pats"] = _patterns(case, rng)
    elif kind == "marginal":
        prefix = np.sort(rng.choice(case["m"], size=case["k"] - 1, replace=False))
        x = np.tile(np.append(prefix, 0), (case["m"], 1)).astype(np.int32)
        x[:, -1] = np.arange(case["m"])
        d["x"] = x
    elif kind == "chain":
        d["u"] = rng.random((case["count"], case["n"]))
    elif kind == "brute":
        d["u"] = rng.random(case["count"])
    elif kind == "serve":
        d["pats"] = []
        for _ in range(case["count"]):
            n = min(int(rng.integers(case["n_lo"], case["n_hi"] + 1)), case["m"])
            d["pats"].append(np.sort(rng.choice(case["m"], size=n, replace=False)).astype(np.int32))
    return d


OUTS = (("p", 1), ("logp", 1), ("haf", 2), ("err", 1))


def prepare(case, seed):
    d, kind = _inputs(case, seed), case["kind"]
    s = {"case": case}
    if kind == "haf":
        flat, s["n"], s["offs"] = gbs.pack_matrices(d["mats"])
        s["A"] = torch.from_numpy(flat).cuda()
        s["haf"] = torch.zeros(2 * case["count"], dtype=torch.float64, device="cuda")
        return s
    s["K"] = gbs.build_kernel(torch.view_as_real(d["U"]).contiguous(), torch.from_numpy(d["r"]).cuda())
    torch.cuda.synchronize()
    if kind == "prob":
        s["idx"], s["n"], s["offs"] = gbs.pack_patterns(d["pats"])
        if not case["host"]:
            s["idx"] = torch.from_numpy(s["idx"]).cuda()
        s["out"] = {}
        for o, width in OUTS:
            if o in case["outs"].split(","):
                k = width * case["count"]
                s["out"][o] = np.zeros(k) if case["host"] else torch.zeros(k, dtype=torch.float64, device="cuda")
    elif kind == "serve":
        s["pats"] = d["pats"]
        s["server"] = gbs.Server(s["K"], max_n=26)
    elif kind == "marginal":
        s["x"] = d["x"]
    else:
        s["u"] = d["u"]
    return s


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "prob":
        o = s["out"]
        gbs.prob_batch(s["K"], s["idx"], s["n"], s["offs"], PREC[case["prec"]], p_out=o.get("p"),
                       logp_out=o.get("logp"), haf_out=o.get("haf"), err_out=o.get("err"))
        return dict(o)
    if kind == "haf":
        gbs.hafnian_batch(s["A"], s["n"], s["offs"], gbs.FP64, haf_out=s["haf"])
        return {"haf": s["haf"]}
    if kind == "marginal":
        return {"q": gbs.marginal_batch(s["K"], s["x"], case["n"])}
    if kind == "chain":
        return {"x": gbs.sample_chain_batch(s["K"], case["n"], s["u"])}
    if kind == "brute":
        x, total = gbs.sample_bruteforce(s["K"], case["n"], s["u"], PREC[case["prec"]])
        return {"x": x, "total": total}
    # serve: hand every request in, then collect whatever is done until all are
    srv, prec, count = s["server"], PREC[case["prec"]], len(s["pats"])
    at = {srv.submit(x, prec): i for i, x in enumerate(s["pats"])}
    p, haf, err, got = np.empty(count), np.empty(count, np.complex128), np.empty(count), 0
    while got < count:
        t, pp, hh, ee, rc = srv.wait_any(timeout_s=1.0)
        if len(rc) and rc.min() < 0:
            raise RuntimeError("a request failed with %d" % rc.min())
        k = [at[int(v)] for v in t]
        p[k], haf[k], err[k] = pp, hh, ee
        got += len(k)
    return {"p": p, "haf": haf, "err": err}


# ---------------------------------------------------------------------------
# the least work
# ---------------------------------------------------------------------------
def _matching_macs(n):
    """Complex multiply-adds of a Hafnian by summing over the matchings of a
    growing prefix: a partial sum for each set of j later positions that the
    first i positions are matched with, each formed from j earlier ones."""
    if n < 2 or n % 2:
        return 0
    return sum(j * math.comb(n - i, j) for i in range(1, n + 1) for j in range(i % 2, min(i, n - i) + 1, 2))


def _subset_flops(n):
    """The 2^(n/2)-subset sum, one characteristic polynomial (8 N^3 flops) a
    subset: what an error estimate needs, which sums the moduli of its terms."""
    h = n // 2
    return 0 if n < 2 or n % 2 else sum(math.comb(h, s) * 8 * (2 * s) ** 3 for s in range(1, h + 1))


def work(case):
    kind = case["kind"]
    if kind in ("prob", "haf", "serve"):
        numbers = range(case["n_lo"], case["n_hi"] + 1, case.get("n_step", 1))
        estimate = kind == "serve" or "err" in case.get("outs", "").split(",")
        one = _subset_flops if estimate else (lambda n: 8 * _matching_macs(n))
        mean = 1.0 / len(numbers)
        flops = case["count"] * mean * sum(one(n) for n in numbers)
        read = sum(16 * n * n if kind == "haf" else 4 * n for n in numbers) * mean * case["count"]
        if kind != "haf":
            read += 16 * case["m"] ** 2
        width = dict(OUTS)
        outs = ("haf",) if kind == "haf" else ("p", "haf", "err") if kind == "serve" else case["outs"].split(",")
        return {"bytes": read + 8 * case["count"] * sum(width[o] for o in outs), "flops": flops}
    m, n = case["m"], case["n"]
    if kind == "brute":
        c = math.comb(m + n - 1, n)
        return {"bytes": 16 * m * m + case["count"] * (8 + 4 * n), "flops": c * 8 * max(1, _matching_macs(n))}

    def products(k):
        """Products Haf(W_s) Haf(W_rest) of the marginal sum over a prefix of
        k: the even subsets s of the even sets that have a term in range."""
        lo, t = max(0, 2 * k - n), 0
        for c in range(0, k + 1, 2):
            ok = [a for a in range(0, c + 1, 2) if a >= lo and any(
                b >= lo and max(0, 3 * k - a - b - n) <= k - c <= k - max(a, b) for b in range(0, c + 1, 2))]
            t += math.comb(k, c) * sum(math.comb(c, a) for a in ok if a <= c - a or c - a not in ok)
        return t

    if kind == "marginal":
        return {"bytes": 16 * m * m + m * (4 * case["k"] + 8), "flops": m * 8 * products(case["k"])}
    return {"bytes": 16 * m * m + case["count"] * n * 12,
            "flops": case["count"] * m * 8 * sum(products(k) for k in range(1, n + 1))}


# ---------------------------------------------------------------------------
# the same in plain 64-bit torch
# ---------------------------------------------------------------------------
_MASKS = {}


def _masks(r, j):
    """The j-subsets of r positions as bit masks, in increasing order."""
    if j < 0 or j > r:
        return np.zeros(0, np.int64)
    if j == 0:
        return np.zeros(1, np.int64)
    if (r, j) not in _MASKS:
        _MASKS[r, j] = np.concatenate([_masks(r - 1, j), _masks(r - 1, j - 1) | (1 << (r - 1))])
    return _MASKS[r, j]


def _hafnians(A):
    """Haf of a batch of symmetric matrices (b, n, n): sums over the matchings
    of a growing prefix, kept for every set of later positions they use up."""
    b, n = A.shape[0], A.shape[1]
    if n % 2:
        return torch.zeros(b, dtype=A.dtype, device=A.device)
    level = {0: torch.ones(b, 1, dtype=A.dtype, device=A.device)}
    for i in range(n):  # position i is matched now; sets lie in the R positions after it
        R, new = n - i - 1, {}
        for j in range((i + 1) % 2, min(i + 1, R) + 1, 2):
            sets = _masks(R, j)
            v = torch.zeros(b, len(sets), dtype=A.dtype, device=A.device)
            if j + 1 in level:  # i itself was used up before
                v += level[j + 1][:, torch.from_numpy(np.searchsorted(_masks(R + 1, j + 1), sets * 2 + 1)).to(A.device)]
            rest = sets.copy()
            for _ in range(j):  # i is matched with the set's lowest remaining position
                low = rest & -rest
                at = np.round(np.log2(low)).astype(np.int64) + i + 1
                src = np.searchsorted(_masks(R + 1, j - 1), (sets ^ low) * 2)
                v += A[:, i, torch.from_numpy(at).to(A.device)] * level[j - 1][:, torch.from_numpy(src).to(A.device)]
                rest ^= low
            new[j] = v
        level = new
    return level[0][:, 0]


def _kappa(A):
    """sum_S |f(X A_S)|_1 over the subsets of the pairs (t, t + n/2), zero diagonal."""
    b, n = A.shape[0], A.shape[1]
    h = n // 2
    order = [p // 2 + (h if p % 2 else 0) for p in range(n)]
    A = A[:, order][:, :, order] * (1 - torch.eye(n, dtype=A.dtype, device=A.device))
    total = torch.zeros(b, dtype=torch.float64, device=A.device)
    for mask in range(1, 1 << h):
        rows = [2 * p + q for p in range(h) if mask >> p & 1 for q in (0, 1)]
        swapped = [v ^ 1 for v in rows]
        M = A[:, swapped][:, :, rows]
        power, c = M, [torch.ones(b, dtype=A.dtype, device=A.device)]
        tr = []
        for k in range(1, h + 1):  # exp(sum_k tr_k x^k / (2 k)) up to x^h
            tr.append(torch.diagonal(power, dim1=1, dim2=2).sum(1))
            c.append(sum(tr[i - 1] * c[k - i] for i in range(1, k + 1)) / (2 * k))
            power = power @ M if k < h else power
        total += c[h].real.abs() + c[h].imag.abs()
    return total


def _marginals(W, x, n):
    """q_n of the rows of x by the theorem's sum over position sets rho and
    their subsets, for distinct modes in a row and for repeated ones."""
    (b, k), m = x.shape, W.shape[0]
    V = W[x[:, :, None], x[:, None, :]].cpu().numpy()
    H = {0: np.ones(b, np.complex128)}
    for t in range(1, 1 << k):
        if bin(t).count("1") % 2 == 0:
            i, rest = (t & -t).bit_length() - 1, t & (t - 1)
            H[t] = sum(V[:, i, j] * H[rest ^ (1 << j)] for j in range(k) if rest >> j & 1)

    def lg(a, c):
        return math.lgamma(a + 1) - math.lgamma(c + 1) - math.lgamma(a - c + 1)

    lo, q = max(0, 2 * k - n), np.zeros(b)
    for rho in H:
        c = bin(rho).count("1")
        mu, sizes = k - c, range(0, c + 1, 2)

        def fits(a, d):
            return min(a, d) >= lo and max(0, 3 * k - a - d - n) <= mu <= k - max(a, d)

        need = [a for a in sizes if any(fits(a, d) for d in sizes)]
        if not need:
            continue
        G, s = {a: np.zeros(b, np.complex128) for a in need}, rho
        while True:
            a = bin(s).count("1")
            if a in G and a % 2 == 0:
                G[a] += H[s] * H[rho ^ s]
            if s == 0:
                break
            s = (s - 1) & rho
        form = np.zeros(b)
        for a in need:
            for d in need:
                if fits(a, d):
                    f = math.exp(math.lgamma(n - k + 1) + lg(0.5 * (n - k + mu + m) - 1, k - 0.5 * (a + d) + 0.5 * m - 1)
                                 - math.lgamma(n + 1) - lg(0.5 * (m + n) - 1, 0.5 * n))
                    form += f * (G[a] * np.conj(G[d])).real
        w = np.ones(b)  # prod_v alpha_v! C(m_v, alpha_v), alpha_v the copies of v outside rho
        for i in range(k):
            same = x == x[:, i:i + 1]
            first = ~same[:, :i].any(1)
            out = np.array([not rho >> p & 1 for p in range(k)])
            mult, alpha = same.sum(1), (same & out[None, :]).sum(1)
            w *= np.where(first, [math.factorial(e) * math.comb(v, e) for v, e in zip(mult, alpha)], 1.0)
        q += w * form
    return q


def _exact_patterns(d, case, want):
    """p, log p, Haf and the error estimate (for orders up to 16, whose pairing
    is the library's documented default) of a case's patterns."""
    count, pats = len(d["pats"]), d["pats"]
    t = torch.tanh(torch.from_numpy(d["r"]).cuda())
    B = (d["U"] * t[None, :]) @ d["U"].T
    norm = float(np.log(np.cosh(d["r"])).sum())
    haf, kap = np.zeros(count, np.complex128), np.zeros(count)
    ns = np.array([len(x) for x in pats])
    # bunched lists take another sum, whose estimate is its own
    kappa = "err" in want and ns.max() <= 16 and all(len(set(x.tolist())) == len(x) for x in pats)
    for n in sorted(set(ns.tolist())):
        at = np.nonzero(ns == n)[0]
        step = max(1, (1 << 27) // max(1, 2 ** n if n < 20 else int(1.62 ** n)))
        for lo in range(0, len(at), step):
            sel = at[lo:lo + step]
            x = torch.from_numpy(np.array([pats[i] for i in sel], dtype=np.int64).reshape(len(sel), n)).cuda()
            A = B[x[:, :, None], x[:, None, :]]
            haf[sel] = _hafnians(A).cpu().numpy() if n else 1.0
            if kappa and n and n % 2 == 0:
                kap[sel] = _kappa(A).cpu().numpy()
    fact = np.array([math.prod(math.factorial(int(v)) for v in np.bincount(x)) if len(x) else 1 for x in pats], float)
    with np.errstate(divide="ignore", invalid="ignore"):
        q = np.abs(haf) ** 2 / fact
        u = 2.0 ** -53 * ns if case["prec"] == "fp64" else 2.0 ** -24 * np.minimum(ns, 4)
        even = kappa and bool((ns > 0).all() and (ns % 2 == 0).all())
        return {"p": q * math.exp(-norm), "logp": np.log(q) - norm, "haf": haf, "err": u * kap / np.abs(haf) if even else None}


def exact(case, seed):
    kind, d = case["kind"], _inputs(case, seed)
    if kind in ("prob", "serve"):
        want = case["outs"].split(",") if kind == "prob" else ["p", "haf", "err"]
        e = _exact_patterns(d, case, want)
        out = {o: e[o] for o in want}
        if kind == "prob" and "haf" in out:
            out["haf"] = out["haf"].view(np.float64)
        return out
    if kind == "haf":
        out = np.zeros(case["count"], np.complex128)
        for n in sorted(set(M.shape[0] for M in d["mats"])):
            at = [i for i, M in enumerate(d["mats"]) if M.shape[0] == n]
            out[at] = _hafnians(torch.from_numpy(np.array([d["mats"][i] for i in at])).cuda()).cpu().numpy() if n else 1.0
        return {"haf": out.view(np.float64)}
    if kind == "marginal":
        return {"q": _marginals(d["U"] @ d["U"].T, d["x"], case["n"])}
    if kind == "brute":
        # the total is P_n, the coefficient of z^n of prod sech r (1 - tanh^2 r z^2)^(-1/2)
        n, m, r = case["n"], case["m"], d["r"][0]
        if n % 2:
            return {"x": None, "total": 0.0}
        log_p = math.lgamma(m / 2 + n / 2) - math.lgamma(m / 2) - math.lgamma(n / 2 + 1)
        return {"x": None, "total": math.exp(log_p + n * math.log(math.tanh(r)) - m * math.log(math.cosh(r)))}
    return None
