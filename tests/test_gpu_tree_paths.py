"""Each way to the spanning tree on the data it finds hardest, and the path the
profile names for it: the tensor-core sweep on small sets (forced; they take
stored distances by default) with FP32 and FP64 points, ties, duplicates and
points that the FP64 input's FP32 copy cannot tell apart, down to the rescans of
short rows; rows as lists in their own right.  Trees bit for bit the oracle's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture()
def iso():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1702_04739_gb300 import isoclust
    isoclust.load()
    isoclust.set_sweep_variant(-1)
    yield isoclust
    isoclust.set_sweep_variant(-1)


def _points(kind, n, d, dtype):
    rng = np.random.default_rng(n + 5 * d)
    X = rng.normal(size=(n, d)) + 6.0 * rng.integers(0, 3, size=(n, 1))
    if kind == "offset":
        X = X + (1e9 if dtype == np.float64 else 3e4)
    elif kind == "grid":
        X = rng.integers(-1, 2, size=(n, d))
    elif kind == "one-hot":
        X = np.zeros((n, d))
        X[np.arange(n), np.arange(n) % d] = 1.0
    elif kind == "duplicates":
        X[n // 2:] = X[: n - n // 2]
    elif kind == "close":
        X[1::2] = X[: 2 * (n // 2): 2] + 1e-12 * rng.normal(size=(n // 2, d))
    return np.ascontiguousarray(X.astype(dtype))


def _check(iso, orc, X, path):
    eu, ev, ed, _, _ = orc.mst_prim(X)
    gu, gv, gd = iso.cluster_mst(torch.from_numpy(X).cuda())
    assert (gu.cpu().numpy() == eu).all() and (gv.cpu().numpy() == ev).all()
    assert (gd.cpu().numpy() == ed).all()
    prof = iso.last_profile()
    assert prof["tree_path"] == path
    return prof["rescanned_rows"]


@pytest.mark.parametrize("kind", ["plain", "offset", "grid", "one-hot", "duplicates", "close"])
@pytest.mark.parametrize("n,d", [(2, 1), (127, 3), (129, 33), (700, 8), (700, 50), (1500, 70)])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("variant", [0, 3])
def test_sweep(iso, oracle_lib, kind, n, d, dtype, variant):
    iso.set_sweep_variant(variant)
    queued = _check(iso, oracle_lib, _points(kind, n, d, dtype), "tc_sweep")
    assert iso.last_sweep_variant() == variant
    if kind == "one-hot" and n >= 127:                 # exact ties: every row's margin holds more than its keys
        assert queued > 0


@pytest.mark.parametrize("kind", ["plain", "one-hot"])
@pytest.mark.parametrize("n,d,dtype,path", [(700, 50, np.float32, "stored"), (700, 50, np.float64, "stored"),
                                            (1500, 70, np.float64, "tc_sweep"), (6145, 3, np.float32, "tc_sweep")])
def test_default(iso, oracle_lib, kind, n, d, dtype, path):
    _check(iso, oracle_lib, _points(kind, n, d, dtype), path)


def test_fp64_sweep(iso, oracle_lib):
    X = _points("plain", 300, 7, np.float64)
    _check(iso, oracle_lib, X * 1e-155, "sweep")       # past the copy's range
    iso.cluster_mst(torch.from_numpy(X).cuda(), iso.opts(precision=iso.PREC_FP64))
    assert iso.last_profile()["tree_path"] == "sweep"


@pytest.mark.parametrize("n,nnz,paths", [(700, 32, ("lists", "gram_lists")), (700, 33, ("stored", "gram_tc")),
                                         (2, 5, ("lists", "gram_lists"))])
def test_lists(iso, oracle_lib, n, nnz, paths):
    rng = np.random.default_rng(nnz)
    X = np.zeros((n, 512), np.float32)
    for i in range(n):
        X[i, rng.choice(512, nnz, replace=False)] = rng.normal(size=nnz)
    _check(iso, oracle_lib, X, paths[0])
    iso.cluster_detail(torch.from_numpy(X).cuda(), 1, 5.0)
    prof = iso.last_profile()
    assert (prof["tree_path"], prof["omega_path"]) == paths


def test_omega_paths(iso):
    X = torch.from_numpy(_points("plain", 500, 20, np.float32)).cuda()
    iso.cluster_detail(X, 2, 1.0)
    assert iso.last_profile()["omega_path"] == "sums"
    iso.cluster_detail(X, 2, 1.0, iso.opts(omega_mode=iso.OMEGA_TREE))
    assert iso.last_profile()["omega_path"] == "none"
    iso.cluster_mst(X)
    assert iso.last_profile()["omega_path"] == "none"
    iso.cluster_batched(X, [0, 200, 500], [2, 2], 1.0)
    assert (iso.last_profile()["tree_path"], iso.last_profile()["omega_path"]) == ("tc_sweep", "sums")
