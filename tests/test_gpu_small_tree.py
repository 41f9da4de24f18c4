"""The search of a tree of up to 12,288 vertices (a block per threshold, the
tree in shared memory) at the ends of its range and against the larger trees'
passes, and the pointer jumping of up to 16,384 elements by one block: the
oracle's i_k, labels and residual, with and without potentials."""
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


@pytest.mark.parametrize("n", [2, 3, 511, 512, 513, 4898, 8193, 8194, 12287, 12288, 12289, 16384, 16385])
@pytest.mark.parametrize("shape", ["random", "star", "deep", "binary"])
def test_bit_exact(iso, oracle_lib, n, shape):
    from paper_1702_04739_gb300 import workloads
    rng = np.random.default_rng(n)
    parent, phi, om, p = workloads.random_rooted_tree(seed=n, n=n, shape=shape)
    for k, q, f in ((1, None, phi), (min(n, 37), p, phi), (min(n, 5), None, np.where(rng.random(n) < 0.5, 1.0, phi))):
        ref = oracle_lib.tree_stage(parent, f, om, q, k)
        lab, res, ik = iso.tree_isoperimetric(*[torch.from_numpy(np.ascontiguousarray(a)).cuda() if a is not None else None
                                                for a in (parent, f, om, q)], k)
        assert float(ik.cpu()[0]) == ref["i_k"]
        assert (lab.cpu().numpy() == ref["labels"]).all() and (res.cpu().numpy() == ref["residual"]).all()
