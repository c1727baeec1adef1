"""Dense paths with several trajectories per stream of the matrix, and the symmetric paths with a
block pair cut over a cluster of CTAs: every pass width (1, 2, 3, 4, 8 and mixtures), ragged node
counts and 1 to 21 block pairs, against the FP64 oracle within the library's 1e-5 bar per
trajectory; trajectories do not depend on what shares their pass beyond FP32 rounding."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

REL_L2 = 1e-5


@pytest.fixture(scope="module")
def nf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2504_13379_gb300 as nf
    nf.lib()
    return nf


def f64(a):
    return np.asarray(a, dtype=np.float32).astype(np.float64)


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float32), device="cuda")


@pytest.mark.parametrize("n", [64, 1024, 1025, 3000, 6100])
@pytest.mark.parametrize("path", ["DENSE_FP32", "DENSE_BF16X2", "DENSE_SYM_FP32", "DENSE_SYM_BF16X2"])
def test_pass_widths_match_oracle(nf, path, n):
    rng = np.random.default_rng(n)
    X = rng.uniform(-1, 1, size=(n, 3)).astype(np.float32)
    q = (rng.uniform(0.5, 1.5, n) / n).astype(np.float32)
    kern = (1.0, 0.3, 0.5, 0.6)
    Bmax = 19
    u = rng.normal(0.3, 0.4, size=(Bmax, n)).astype(np.float32)
    beta = rng.uniform(10, 40, Bmax).astype(np.float32)
    theta = rng.uniform(0.1, 0.3, Bmax).astype(np.float32)
    want = oracle.nonlocal_sum(f64(X), f64(q), f64(u), tuple(f64(kern)), f64(beta), f64(theta))
    op = nf.Operator(dev(X), dev(q), kern, getattr(nf, path))
    for B in (1, 2, 3, 4, 5, 8, 11, 19):
        got = nf.nf_nonlocal_apply(op, dev(u[:B]), dev(beta[:B]), dev(theta[:B])).cpu().numpy()
        err = np.linalg.norm(got - want[:B], axis=1) / np.linalg.norm(want[:B], axis=1)
        assert err.max() < REL_L2, (path, n, B, err.max())
        again = nf.nf_nonlocal_apply(op, dev(u[:B]), dev(beta[:B]), dev(theta[:B])).cpu().numpy()
        np.testing.assert_array_equal(got, again)
