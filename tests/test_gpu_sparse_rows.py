"""Rows with few non-zeros: the spanning tree and omega from the rows' lists
against the oracle (the tree bit for bit) and against the dense kernels, with
empty rows, duplicates, one full row, a dimension all rows hold, and the
density rule."""
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
    isoclust.set_sweep_variant(-1)
    isoclust.set_omega_gram(-1)


def _rows(n, d, kind):
    rng = np.random.default_rng(n + d)
    X = np.zeros((n, d), np.float32)
    nnz = max(2, d // 100)
    for i in range(n):
        pool = rng.integers(0, d, size=4 * nnz) if i % 5 else np.arange(4 * nnz)
        c = rng.choice(pool, nnz)
        X[i, c] = np.exp(rng.normal(size=nnz))
    if kind == "odd":
        X[n // 2] = 0.0                                        # empty
        X[-1] = 0.0                                            # and its duplicate
        X[1] = X[0]
        X[min(3, n - 1)] = rng.normal(size=d) * 0.1            # a full row
        X[:: 7] *= -1.0
    elif kind == "shared":
        X[:, 5] = 40.0                                         # products that cancel in every distance
    return X


SHAPES = [(2, 512), (33, 600), (127, 512), (129, 1000), (700, 4096), (6200, 513)]


@pytest.mark.parametrize("n,d", SHAPES)
@pytest.mark.parametrize("kind", ["plain", "odd", "shared"])
def test_tree(iso, oracle_lib, n, d, kind):
    X = _rows(n, d, kind)
    eu, ev, ed, _, _ = oracle_lib.mst_prim(X)
    Xd = torch.from_numpy(X).cuda()
    for v in (-1, 0):                                          # 0: the dense sweep
        iso.set_sweep_variant(v)
        gu, gv, gd = iso.cluster_mst(Xd)
        assert (gu.cpu().numpy() == eu).all() and (gv.cpu().numpy() == ev).all()
        assert (gd.cpu().numpy() == ed).all()
        if v < 0 and n > 6144:
            assert iso.last_profile()["mst_tiles_full"] == 0   # not the sweep
    iso.set_sweep_variant(-1)


@pytest.mark.parametrize("share,sparse", [(16, True), (15, False)])
def test_density_rule(iso, share, sparse):
    n, d = 6200, 512
    X = np.zeros((n, d), np.float32)
    X[:, : d // 16 + (0 if sparse else 1)] = np.random.default_rng(1).normal(size=(n, d // 16 + (0 if sparse else 1)))
    iso.cluster_mst(torch.from_numpy(X).cuda())
    assert (iso.last_profile()["mst_tiles_full"] == 0) == sparse


def _bound(orc, X, sigma):
    # d2 to 2^-46 (of its parts where they do not cancel to under a quarter of them), so y = d /
    # sigma to half of that relatively, every term to y times it; 4: the exponential and the sums
    nn, nd2 = orc.nn_rows(X, np.arange(X.shape[0]))
    return 2.0 ** -45 * max(1.0, math.sqrt(X.shape[1] / 64.0)) * (np.sqrt(nd2) / sigma + 4.0)


@pytest.mark.parametrize("n,d", SHAPES[:-1] + [(2500, 512)])
@pytest.mark.parametrize("kind", ["plain", "odd", "shared"])
def test_omega(iso, oracle_lib, n, d, kind):
    X = _rows(n, d, kind)
    Xd = torch.from_numpy(X).cuda()
    for sigma in (1.0, 0.3):
        ref, _ = oracle_lib.weights(X, sigma)
        iso.set_omega_gram(1)
        om = iso.cluster_detail(Xd, 1, sigma)["omega"].cpu().numpy()
        assert iso.last_profile()["omega_symmetric"] == 3
        iso.set_omega_gram(-1)
        assert (np.abs(om - ref) <= _bound(oracle_lib, X, sigma) * ref).all()
