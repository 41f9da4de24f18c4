"""omega of a set's long rows keeps its accuracy whatever the set's size: the
Gram on the tensor cores from 64 dimensions on, with errors that do not grow
with the row length as those of plain sums of squares do."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def iso():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1702_04739_gb300 import isoclust
    isoclust.load()
    isoclust.set_omega_gram(-1)
    return isoclust


def _blobs(n, d):
    rng = np.random.default_rng(n + d)
    return (rng.uniform(-10, 10, size=(5, d))[np.arange(n) % 5] + rng.normal(size=(n, d))).astype(np.float32)


@pytest.mark.parametrize("n,d", [(2, 64), (130, 64), (1000, 65), (2000, 130), (800, 620), (500, 1558), (512, 1100)])
def test_small_sets(iso, oracle_lib, n, d):
    X = _blobs(n, d)
    om = iso.cluster_detail(torch.from_numpy(X).cuda(), 1, 1.0)["omega"].cpu().numpy()
    assert iso.last_profile()["omega_symmetric"] == 3
    ref, _ = oracle_lib.weights(X, 1.0)
    # d2 to 2^-46 of itself at any length, y = d / sigma to half of that relatively, a term to y
    # times it; 4: the exponential and the sums
    y = np.sqrt(oracle_lib.nn_rows(X, np.arange(n))[1])
    assert (np.abs(om - ref) <= 2.0 ** -47 * (y + 4.0) * ref).all()


@pytest.mark.parametrize("n,d,expect", [(130, 63, 2), (2000, 63, 2), (130, 64, 3)])
def test_rule(iso, n, d, expect):
    iso.cluster_detail(torch.from_numpy(_blobs(n, d)).cuda(), 1, 1.0)
    assert iso.last_profile()["omega_symmetric"] == expect


@pytest.mark.parametrize("n,d", [(64, 33), (64, 61), (64, 64), (50, 256), (64, 620), (33, 1300), (64, 1558)])
def test_direct_sums_do_not_lean(iso, n, d):
    """Pairs that cancel (clusters far from their tile's centre) take sums of squared differences.
    Their roundings may not lean one way: the errors of omega's rows average out to less than 2^-50
    of the exponent's half (d2 to y) and of the exponential and the sums (4 such units)."""
    rng = np.random.default_rng(n + d)
    X = (rng.uniform(-10, 10, size=(4, d))[np.arange(n) % 4] + rng.normal(size=(n, d))).astype(np.float32)
    iso.set_omega_gram(1)
    om = iso.cluster_detail(torch.from_numpy(X).cuda(), 1, 1.0)["omega"].cpu().numpy()
    iso.set_omega_gram(-1)
    assert iso.last_profile()["omega_gram_direct_pairs"] >= n * (n // 4 - 1)
    L = X.astype(np.longdouble)
    y = np.stack([np.sqrt(np.square(L - row).sum(1)) for row in L])
    np.fill_diagonal(y, np.inf)
    ref = np.exp(-y).sum(1)
    err = ((om - ref) / ref).astype(np.float64)
    assert abs(err.mean()) <= 2.0 ** -50 * (float(y.min(1).mean()) / 2 + 4.0), err.mean()
