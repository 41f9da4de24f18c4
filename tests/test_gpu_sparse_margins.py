"""The spanning tree from rows as lists: the margin of a row's candidates
follows from its own entries and norms, so that neither one full or long row nor
rows far from the origin make candidates of every column; and rows with more candidates than a block
keys together (exact ties) give the oracle's tree all the same."""
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
    return isoclust


def _unit_rows(n, d, nnz, rng):
    X = np.zeros((n, d), np.float32)
    for i in range(n):
        X[i, rng.choice(d, nnz, replace=False)] = np.exp(rng.normal(size=nnz))
    return X / np.linalg.norm(X, axis=1, keepdims=True)


def _same_tree(iso, orc, X):
    eu, ev, ed, _, _ = orc.mst_prim(X)
    gu, gv, gd = iso.cluster_mst(torch.from_numpy(np.ascontiguousarray(X)).cuda())
    assert (gu.cpu().numpy() == eu).all() and (gv.cpu().numpy() == ev).all()
    assert (gd.cpu().numpy() == ed).all()
    return iso.last_profile()["rescanned_rows"]


@pytest.mark.parametrize("row", ["ones", "random", "long"])
def test_one_full_row(iso, oracle_lib, row):
    n, d = 900, 4096
    rng = np.random.default_rng(4)
    X = _unit_rows(n, d, 41, rng)
    X[77] = {"ones": np.ones(d), "random": rng.normal(size=d) / 64.0, "long": 300.0 * X[77]}[row]
    assert _same_tree(iso, oracle_lib, X) == 0          # no row with more than 128 candidates


@pytest.mark.parametrize("value", [30.0, 1000.0, -3e6])
@pytest.mark.parametrize("rows", ["all", "half", "one block"])
def test_far_from_the_origin(iso, oracle_lib, value, rows):
    n, d = 900, 1024
    X = _unit_rows(n, d, 20, np.random.default_rng(5))
    X[{"all": slice(None), "half": slice(None, None, 2), "one block": slice(100, 300)}[rows], 5] = value
    X[201] = X[200]
    # products that cancel make no candidates of every column; of two groups that far apart the one
    # round that joins them finds the distances between them tied in FP32
    assert _same_tree(iso, oracle_lib, X) <= (0 if rows == "all" else n)


@pytest.mark.parametrize("kind", ["one-hot", "equal", "identical"])
@pytest.mark.parametrize("n", [700, 2500])
def test_ties(iso, oracle_lib, kind, n):
    d = 512
    rng = np.random.default_rng(n)
    if kind == "one-hot":                               # every pair tied, or the same point
        X = np.zeros((n, d), np.float32)
        X[np.arange(n), rng.integers(0, d, size=n)] = 1.0
    elif kind == "equal":                               # binary rows of two entries: few different distances
        X = np.zeros((n, d), np.float32)
        for i in range(n):
            X[i, rng.choice(40, 2, replace=False)] = 0.5
    else:                                               # a block of identical rows among others
        X = _unit_rows(n, d, 20, rng)
        X[50:350] = X[3]
    assert _same_tree(iso, oracle_lib, X) > 0
