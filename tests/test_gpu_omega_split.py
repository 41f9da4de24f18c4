"""omega with potentials over column splits (fewer blocks than the chip holds)
at the edges of the splits' rule, against the FP64 oracle."""
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
    return isoclust


@pytest.mark.parametrize("n,d", [(2, 3), (448, 11), (449, 11), (512, 2), (1025, 40), (4900, 7)])
def test_potentials(iso, oracle_lib, n, d):
    rng = np.random.default_rng(n)
    X = (rng.normal(size=(n, d)) + 5.0 * rng.integers(0, 3, size=(n, 1))).astype(np.float32)
    sigma, alpha = 1.5, 0.01
    o = iso.cluster_detail(torch.from_numpy(X).cuda(), 1, sigma, iso.opts(alpha=alpha))
    om, p = oracle_lib.weights(X, sigma, alpha)
    nn, nd2 = oracle_lib.nn_rows(X, np.arange(n))
    # d2 to 2^-46, a term to y times 2^-47, 4 for the exponential and the sums; a potential's terms
    # to 2^-46, one more rounding of the double-word sum per term
    bound = 2.0 ** -45 * max(1.0, math.sqrt(d / 64.0)) * (np.sqrt(nd2) / sigma + 4.0)
    assert (np.abs(o["omega"].cpu().numpy() - om) <= bound * om).all()
    assert (np.abs(o["p"].cpu().numpy() - p) <= (n + 8) * 2.0 ** -46 * p).all()
