"""Calls under a caller's spin limit: however small it is, a call ends with its
results or with the timeout status, and the library works on afterwards."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TIMEOUT = 6


@pytest.fixture(scope="module")
def iso():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1702_04739_gb300 import isoclust
    isoclust.load()
    yield isoclust
    isoclust.set_omega_gram(-1)


def _points(n, d, k):
    rng = np.random.default_rng(n + d)
    return (rng.uniform(-10, 10, size=(k, d))[np.arange(n) % k] + rng.normal(size=(n, d))).astype(np.float32)


# one centre for all tiles (no barrier but the flags' between a block's two first preparations), and several
@pytest.mark.parametrize("n,d,k", [(1500, 64, 1), (1500, 64, 6), (1100, 200, 2), (900, 30, 1)])
def test_any_limit_ends(iso, n, d, k):
    Xd = torch.from_numpy(_points(n, d, k)).cuda()
    iso.set_omega_gram(1)
    ref = iso.cluster_detail(Xd, 3, 2.0)
    sref = iso.cluster_batched(Xd, [0, 400, n], [2, 2], 2.0, detail=True)
    ended = set()
    for e in range(0, 26):
        o = iso.opts(spin_limit=1 << e)
        for call, want in ((lambda: iso.cluster_detail(Xd, 3, 2.0, o), ref),
                           (lambda: iso.cluster_batched(Xd, [0, 400, n], [2, 2], 2.0, o, detail=True), sref)):
            try:
                got = call()
                ended.add("ok")
                assert torch.equal(got["omega"], want["omega"]) and torch.equal(got["labels"], want["labels"])
            except iso.IsoclustError as err:
                ended.add(err.code)
    assert "ok" in ended and ended <= {"ok", TIMEOUT}, ended
    after = iso.cluster_detail(Xd, 3, 2.0)
    assert torch.equal(after["omega"], ref["omega"]) and torch.equal(after["parent"], ref["parent"])
    iso.set_omega_gram(-1)


# the direct sums of long rows (two clusters far from one another) take some 10^7 cycles a block
@pytest.mark.parametrize("n,d,sigma", [(3279, 1558, 40.0), (2000, 512, 23.0)])
def test_limit_above_the_waits_for_hardware(iso, n, d, sigma):
    Xd = torch.from_numpy(_points(n, d, 2)).cuda()
    iso.set_omega_gram(1)
    want = iso.cluster_detail(Xd, 2, sigma)
    got = iso.cluster_detail(Xd, 2, sigma, iso.opts(spin_limit=1000000))
    iso.set_omega_gram(-1)
    assert torch.equal(got["omega"], want["omega"])
