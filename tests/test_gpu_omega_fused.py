"""eq. omega with the Gram on the tensor cores at the edges of its kernel: row
lengths about a chunk (32), the resident rows' limit (64) and an accumulator
set's (192), sets of ragged sizes, rows far from all others, clusters that
share a centre and ones that do not; against the FP64 oracle, and the rule
that picks it against the CUDA-core sums."""
import math

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
    yield isoclust
    isoclust.set_omega_gram(-1)


def _bound(orc, X, sigma):
    # d2 to 2^-46 (sqrt(d / 64) more for longer rows), so y = d / sigma to half of that
    # relatively, every term to y times it; 4: the exponential and the sums
    nn, nd2 = orc.nn_rows(X, np.arange(X.shape[0]))
    return 2.0 ** -45 * max(1.0, math.sqrt(X.shape[1] / 64.0)) * (np.sqrt(nd2) / sigma + 4.0)


def _points(d, n, seed):
    rng = np.random.default_rng(seed)
    cen = rng.uniform(-10, 10, size=(4, d))
    X = cen[np.arange(n) % 4] + rng.normal(size=(n, d))
    X[:: 97] = rng.uniform(-60, 60, size=(len(X[:: 97]), d))     # far rows
    return X.astype(np.float32)


@pytest.mark.parametrize("d", [3, 31, 32, 33, 64, 65, 191, 192, 193, 400])
def test_row_lengths(iso, oracle_lib, d):
    n, sigma = 1000 + d % 7, math.sqrt(d) / 3.0
    X = _points(d, n, d)
    iso.set_omega_gram(1)
    om = iso.cluster_detail(torch.from_numpy(X).cuda(), 3, sigma)["omega"].cpu().numpy()
    assert iso.last_profile()["omega_symmetric"] == 3
    iso.set_omega_gram(-1)
    ref, _ = oracle_lib.weights(X, sigma)
    assert (np.abs(om - ref) / ref <= _bound(oracle_lib, X, sigma)).all()


@pytest.mark.parametrize("d,sizes", [(8, [2, 64, 65, 3, 128, 129, 500]), (33, [700, 63, 2, 192]), (70, [260, 5, 64])])
def test_sets(iso, oracle_lib, d, sizes):
    sigma = math.sqrt(d) / 3.0
    X = _points(d, sum(sizes), 7)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    Xd = torch.from_numpy(X).cuda()
    iso.set_omega_gram(1)
    om = iso.cluster_batched(Xd, off, [1] * len(sizes), sigma, detail=True)["omega"].cpu().numpy()
    assert iso.last_profile()["omega_symmetric"] == 3
    iso.set_omega_gram(-1)
    for a, b in zip(off[:-1], off[1:]):
        ref, _ = oracle_lib.weights(X[a:b], sigma)
        assert (np.abs(om[a:b] - ref) / ref <= _bound(oracle_lib, X[a:b], sigma)).all(), (a, b)


@pytest.mark.parametrize("n,d,expect", [(4096, 37, 2), (4096, 38, 3), (12000, 11, 2), (12000, 12, 3)])
def test_rule(iso, n, d, expect):
    # 4,096 rows: 64 tiles, 2,080 tile pairs, 65,536 / 2,080 = 31.5 above 6; below 12 dimensions never
    assert 64 * 65 // 2 * (37 - 6) < 65536 <= 64 * 65 // 2 * (38 - 6)
    iso.set_omega_gram(-1)
    iso.cluster_detail(torch.from_numpy(_points(d, n, 3)).cuda(), 3, 2.0)
    assert iso.last_profile()["omega_symmetric"] == expect
