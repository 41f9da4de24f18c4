"""FP64 input: the tensor-core sweep on an FP32 copy with keys from the points
themselves (the tree bit for bit the oracle's, also where the copy cannot tell
points apart: offsets far larger than the spread, exact ties, duplicates) and
the symmetric FP64 omega at the edges of its tiles.  omega's bound per row: d2
carries up to (d + 2) / 2 roundings on either side, so the exponent y = d /
sigma moves by y (d / 2 + 4) 2^-52 between the two, and so does the term's
relative value; a row's sum is dominated by terms whose y is near that of its
nearest neighbour (2 more allowed for), and the sums add 8 roundings."""
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


def _points(kind, n, d, rng):
    X = rng.normal(size=(n, d)) + 6.0 * rng.integers(0, 3, size=(n, 1))
    if kind == "offset":
        X = X + 1e9                                   # the copy is of the centred points
    elif kind == "tiny":
        X = X * 1e-120                                # scaled into FP32's range
    elif kind == "huge":
        X = X * 1e120
    elif kind == "extreme":
        X = X * 1e-155                                # outside the sweep's range: the FP64 sweep
    elif kind == "grid":
        X = rng.integers(-3, 4, size=(n, d)).astype(np.float64)
    elif kind == "close":
        X[1::2] = X[: 2 * (n // 2) : 2] + 1e-12 * rng.normal(size=(n // 2, d))    # far below FP32's spacing
    return np.ascontiguousarray(X)


@pytest.mark.parametrize("kind", ["plain", "offset", "tiny", "huge", "extreme", "grid", "close"])
@pytest.mark.parametrize("n,d", [(2, 1), (127, 3), (129, 33), (700, 8), (1500, 70)])
def test_f64_tree_bit_exact(iso, oracle_lib, kind, n, d):
    X = _points(kind, n, d, np.random.default_rng(n + 7 * d))
    eu, ev, ed, _, _ = oracle_lib.mst_prim(X)
    gu, gv, gd = iso.cluster_mst(torch.from_numpy(X).cuda())
    assert (gu.cpu().numpy() == eu).all() and (gv.cpu().numpy() == ev).all()
    assert (gd.cpu().numpy() == ed).all()


@pytest.mark.parametrize("n,d", [(2, 1), (16, 2), (17, 33), (31, 5), (1023, 4), (1024, 3), (1025, 3), (1057, 65)])
@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_f64_weights(iso, oracle_lib, n, d, dtype):
    X = _points("plain", n, d, np.random.default_rng(n + d)).astype(dtype)
    o = dict(alpha=0.3, include_self=bool(n & 1))
    nn = np.sqrt(oracle_lib.nn_rows(X, np.arange(n))[1])
    for sigma in (0.02, 1.7):                         # terms down to the subnormal range, and ordinary ones
        tol = 2.0 ** -52 * ((d / 2 + 4) * (nn / sigma + 2) + 8)
        om, p = oracle_lib.weights(X, sigma, **o)
        gom, gp = iso.vertex_weights(torch.from_numpy(X).cuda(), sigma, iso.opts(precision=iso.PREC_FP64, **o))
        # a sum of subnormal terms is exact to their spacing only
        assert (np.abs(gom.cpu().numpy() - om) <= tol * om + n * 5e-324).all()
        assert np.allclose(gp.cpu().numpy(), p, rtol=1e-13, atol=0)
    om1, _ = oracle_lib.weights(X, 1.7)
    gom1, _ = iso.vertex_weights(torch.from_numpy(X).cuda(), 1.7, iso.opts(precision=iso.PREC_FP64), want_p=False)
    assert (np.abs(gom1.cpu().numpy() - om1) <= tol * om1).all()
