"""Calls on different streams do not wait for each other."""
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


def test_a_call_does_not_wait_for_another_streams(gbs):
    """While one stream is held up (by a second of spinning, with a call of its
    own behind that), calls on another one that use a side stream finish: by
    their results, with the first stream still busy."""
    rng = np.random.default_rng(8)
    held, free = torch.cuda.Stream(), torch.cuda.Stream()
    calls = []
    for orders in ((16, 20, 22), (16, 20, 24)):  # two shapes: a kept plan's upload is not shared
        mats = [rand_sym(n, rng) for n in orders]
        flat, n, offs = gbs.pack_matrices(mats)
        out = torch.zeros(2 * len(mats), dtype=torch.float64, device="cuda")
        kap = torch.zeros(len(mats), dtype=torch.float64, device="cuda")
        A = torch.from_numpy(flat).cuda()
        gbs.hafnian_batch(A, n, offs, gbs.FP64, haf_out=out, kappa_out=kap)  # plans, scratch
        torch.cuda.synchronize()
        calls.append((A, n, offs, torch.zeros_like(out), torch.zeros_like(kap), out, kap))

    def call(c, st):
        gbs.hafnian_batch(c[0], c[1], c[2], gbs.FP64, stream=st, haf_out=c[3], kappa_out=c[4])

    with torch.cuda.stream(held):
        torch.cuda._sleep(int(2e9))
    call(calls[0], held)
    for _ in range(3):
        call(calls[1], free)
    free.synchronize()
    assert not held.query()
    assert torch.equal(calls[1][3].cpu(), calls[1][5].cpu())
    held.synchronize()
    for c in calls:
        assert torch.equal(c[3], c[5]) and torch.equal(c[4], c[6])
