"""Stencils at every scale of the coordinates: the same selection, bit for bit, as a brute-force search
in FP64 (by distance^2, then index)."""
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


@pytest.mark.parametrize("power", [-160, -75, -67, -63, -55, 55, 63, 67, 127, 131, 160])
@pytest.mark.parametrize("dim", [2, 3])
def test_any_scale_of_the_coordinates(nf, dim, power):
    """Scaling by a power of two is exact, so it changes no selection."""
    rng = np.random.default_rng(dim)
    X = rng.uniform(0, 1, (3000, dim))
    C = rng.uniform(0, 1, (400, dim))
    want = nf.nf_build_stencils_at(f64(X), f64(C), 24).cpu().numpy()
    np.testing.assert_array_equal(want[:50], _brute(X, C[:50], 24))
    got = nf.nf_build_stencils_at(f64(X * 2.0 ** power), f64(C * 2.0 ** power), 24).cpu().numpy()
    np.testing.assert_array_equal(got, want)
