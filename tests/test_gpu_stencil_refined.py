"""Stencils on node sets that are not evenly spread: the same selection, bit for bit, as a brute-force
search in FP64 (by distance^2, then index)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2504_13379_gb300 as nf
    nf.lib()
    return nf


def f64(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64), device="cuda")


def _brute(X, C, k):
    out = np.empty((len(C), k), dtype=np.int32)
    for i, c in enumerate(C):
        d = (X[:, 0] - c[0]) ** 2 + (X[:, 1] - c[1]) ** 2
        if X.shape[1] == 3:
            d = d + (X[:, 2] - c[2]) ** 2
        out[i] = np.argsort(d, kind="stable")[:k]
    return out


def _refined(kind, dim, n, rng):
    if kind == "cluster":  # four fifths of the nodes in a ball of 1 % of the domain
        X = rng.uniform(-1, 1, (n, dim))
        m = 4 * n // 5
        X[:m] = 0.3 + 0.01 * rng.uniform(-1, 1, (m, dim))
    elif kind == "graded":  # density falling by orders of magnitude away from a point
        d = rng.normal(size=(n, dim))
        X = d / np.linalg.norm(d, axis=1, keepdims=True) * rng.uniform(0, 1, (n, 1)) ** 4
    else:  # "coincident": many nodes at the very same places
        X = rng.uniform(-1, 1, (n, dim))[rng.integers(0, 6, n)]
        X[: n // 8] = rng.uniform(-1, 1, (n // 8, dim))
    return X


@pytest.mark.parametrize("k", [1, 24, 64])
@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("kind", ["cluster", "graded", "coincident"])
def test_refined_sets(nf, kind, dim, k):
    rng = np.random.default_rng(dim * 100 + k)
    X = _refined(kind, dim, 5000, rng)
    C = np.concatenate([X[rng.integers(0, len(X), 150)], rng.uniform(-1, 1, (40, dim)), X[:10] * 1.0001])
    got = nf.nf_build_stencils_at(f64(X), f64(C), k).cpu().numpy()
    np.testing.assert_array_equal(got, _brute(X, C, k))
