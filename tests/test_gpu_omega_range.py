"""Distances past FP32's range: a call whose squared distances overflow the
double-word FP32 sums is refused as non-finite by every form of omega's
kernel (the sums of squares, the Gram on the tensor cores, independent sets),
and one that stays within the range is answered within omega's bound."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NONFINITE, INTERNAL = 3, 8


@pytest.fixture(scope="module")
def iso():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1702_04739_gb300 import isoclust
    isoclust.load()
    yield isoclust
    isoclust.set_omega_gram(-1)


def _points(n, d, scale):
    return (scale * np.random.default_rng(n + d).normal(size=(n, d))).astype(np.float32)


@pytest.mark.parametrize("n,d", [(300, 16), (1000, 64), (700, 200)])
@pytest.mark.parametrize("scale", [4e18, 1e20])
@pytest.mark.parametrize("mode", [0, 1, -1])
def test_overflow_is_refused(iso, n, d, scale, mode):
    X = _points(n, d, scale)
    assert np.square(X[:64, None].astype(np.float64) - X[None, :64]).sum(-1).max() > 3.5e38
    Xd = torch.from_numpy(X).cuda()
    iso.set_omega_gram(mode)
    with pytest.raises(iso.IsoclustError) as e:
        iso.cluster_detail(Xd, 3, scale)
    assert e.value.code == NONFINITE, str(e.value)
    with pytest.raises(iso.IsoclustError) as e:                # (sets: their sweep may give up before omega)
        iso.cluster_batched(Xd, [0, n // 3, n], [2, 2], scale, detail=True)
    assert e.value.code in (NONFINITE, INTERNAL), str(e.value)


@pytest.mark.parametrize("n,d", [(300, 16), (1000, 64), (700, 200)])
@pytest.mark.parametrize("mode", [0, 1])
def test_large_within_range(iso, oracle_lib, n, d, mode):
    scale = 1e17
    X = _points(n, d, scale)
    X[1] = X[0]                                                # coincident: a term of 1
    iso.set_omega_gram(mode)
    om = iso.cluster_detail(torch.from_numpy(X).cuda(), 3, scale)["omega"].cpu().numpy()
    ref, _ = oracle_lib.weights(X, scale)
    # d2 to 2^-46 (sqrt(d / 64) more for longer rows), y = d / sigma to half of that relatively,
    # every term to y times it; 4: the exponential and the sums
    nn = np.sqrt(oracle_lib.nn_rows(X, np.arange(n))[1])
    assert (np.abs(om - ref) <= 2.0 ** -45 * max(1.0, math.sqrt(d / 64.0)) * (nn / scale + 4.0) * ref).all()
