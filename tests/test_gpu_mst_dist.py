"""The spanning tree on stored distances (small sets) against the oracle's, bit
for bit, at the edges of its tiles and of the rule that picks it, with exact
ties, duplicates, offsets and large magnitudes; and against the tensor-core
sweep, which a forced variant keeps."""
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


def _points(kind, n, d, dtype):
    rng = np.random.default_rng(n + 3 * d)
    X = rng.normal(size=(n, d)) + 6.0 * rng.integers(0, 3, size=(n, 1))
    if kind == "grid":
        X = rng.integers(-1, 2, size=(n, d))
    elif kind == "offset":
        X = X + 3e5
    elif kind == "huge":
        X = X * (1e18 if dtype == np.float32 else 1e100)
    elif kind == "same":
        X = np.ones((n, d))
    return np.ascontiguousarray(X.astype(dtype))


def _check(iso, orc, X):
    eu, ev, ed, _, _ = orc.mst_prim(X)
    gu, gv, gd = iso.cluster_mst(torch.from_numpy(X).cuda())
    assert (gu.cpu().numpy() == eu).all() and (gv.cpu().numpy() == ev).all()
    assert (gd.cpu().numpy() == ed).all()


@pytest.mark.parametrize("n,d", [(2, 1), (3, 2), (63, 31), (64, 32), (65, 33), (129, 63), (130, 64), (257, 65), (1025, 8),
                                 (300, 255), (301, 300), (1000, 2)])
@pytest.mark.parametrize("kind", ["plain", "grid", "offset", "huge", "same"])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_tree(iso, oracle_lib, n, d, kind, dtype):
    if kind == "same" and n > 300:
        pytest.skip("every pair tied: the oracle's own time")
    _check(iso, oracle_lib, _points(kind, n, d, dtype))


@pytest.mark.parametrize("n", [6144, 6145])
def test_rule(iso, oracle_lib, n):
    X = _points("plain", n, 5, np.float32)
    _check(iso, oracle_lib, X)
    assert (iso.last_sweep_variant() == -1) == (n <= 6144)
    iso.set_sweep_variant(0)
    _check(iso, oracle_lib, X)
    assert iso.last_sweep_variant() == 0
    iso.set_sweep_variant(-1)
