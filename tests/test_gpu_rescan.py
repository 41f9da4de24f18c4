"""Rows whose candidates the tensor-core sweep cannot close (far from the mean
and close together, so that its bound is wider than their spread, or exact
ties): the rescan by tiles, the keys of long rows, and what the tiles leave
over.  The tree is the oracle's, bit for bit."""
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
    isoclust.set_sweep_variant(0)                # small sets too take the tensor-core sweep
    yield isoclust
    isoclust.set_sweep_variant(-1)


def _same_tree(iso, orc, X):
    eu, ev, ed, _, _ = orc.mst_prim(X)
    gu, gv, gd = iso.cluster_mst(torch.from_numpy(np.ascontiguousarray(X)).cuda())
    assert (gu.cpu().numpy() == eu).all() and (gv.cpu().numpy() == ev).all()
    assert (gd.cpu().numpy() == ed).all()
    return iso.last_profile()["rescanned_rows"]


@pytest.mark.parametrize("n,d", [(129, 64), (257, 255), (300, 256), (641, 257), (1100, 1558)])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_far_clusters(iso, oracle_lib, n, d, dtype):
    rng = np.random.default_rng(n + d)
    cen = rng.normal(size=(4, d)) * 3000.0
    X = (cen[np.arange(n) % 4] + rng.normal(size=(n, d))).astype(dtype)
    queued = _same_tree(iso, oracle_lib, X)
    assert queued > 0 or d < 256


@pytest.mark.parametrize("n,d", [(200, 2), (300, 300)])
def test_ties(iso, oracle_lib, n, d):
    rng = np.random.default_rng(n)
    X = (rng.integers(0, 2, size=(n, d)) if d < 64 else np.eye(n, d)).astype(np.float32)    # every distance tied
    assert _same_tree(iso, oracle_lib, X) > 0
