"""Matrix-free sums of several trajectories: every group width (4, 8, 12, 16 and remainders behind
full groups of 16), kernel form and distance, on sets whose tiles are skipped, shortened and
full, against the FP64 oracle within the library's 1e-5 bar per trajectory."""
import math

import numpy as np
import pytest
import torch

import nodesets
import oracle

pytestmark = pytest.mark.gpu

REL_L2 = 1e-5
L = float(np.float32(2.0 * math.pi))
KERNELS = {"ratio4": (1.0, 0.1, 0.5, 0.2), "ratio3": (0.7, 0.06, 0.4, 0.06 * math.sqrt(3.0)),
           "ratio2": (1.0, 0.05, 2.0, 0.05 * math.sqrt(2.0)), "general": (1.2, 0.08, 0.6, 0.25),
           "one": (1.0, 0.06, 0.0, 0.2), "wide": (1.0, 0.6, 0.5, 1.2)}


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


@pytest.mark.parametrize("n", [500, 1025, 3300])
@pytest.mark.parametrize("periodic", [False, True])
@pytest.mark.parametrize("name", sorted(KERNELS))
def test_group_widths_match_oracle(nf, name, periodic, n):
    rng = np.random.default_rng(n)
    if periodic:
        X = np.concatenate([rng.uniform(0, L, (n, 2)), 0.1 * rng.normal(size=(n, 1))], 1)
    else:
        X = nodesets.torus_point(rng.uniform(0, 2 * math.pi, n), rng.uniform(0, 2 * math.pi, n), 1.0, 0.4)
    X = X.astype(np.float32)
    q = (rng.uniform(0.5, 1.5, n) / n).astype(np.float32)
    kern = KERNELS[name] + (L if periodic else 0.0,)
    Bmax = 37
    u = rng.normal(0.3, 0.4, size=(Bmax, n)).astype(np.float32)
    beta = rng.uniform(10, 40, Bmax).astype(np.float32)
    theta = rng.uniform(0.1, 0.3, Bmax).astype(np.float32)
    want = oracle.nonlocal_sum(f64(X), f64(q), f64(u), tuple(f64(kern[:4])), f64(beta), f64(theta), period=kern[4])
    op = nf.Operator(dev(X), dev(q), kern, nf.MATRIX_FREE)
    for B in (4, 5, 8, 11, 13, 16, 18, 37):
        got = nf.nf_nonlocal_apply(op, dev(u[:B]), dev(beta[:B]), dev(theta[:B])).cpu().numpy()
        err = np.linalg.norm(got - want[:B], axis=1) / np.linalg.norm(want[:B], axis=1)
        assert err.max() < REL_L2, (name, periodic, n, B, err.max())
    op.mf_schedule(nf.MF_PACKED)
    for B in (1, 2, 3):
        got = nf.nf_nonlocal_apply(op, dev(u[:B]), dev(beta[:B]), dev(theta[:B])).cpu().numpy()
        assert max(np.linalg.norm(got - want[:B], axis=1) / np.linalg.norm(want[:B], axis=1)) < REL_L2


def test_non_finite_values_spread(nf):
    rng = np.random.default_rng(8)
    X = nodesets.torus_point(rng.uniform(0, 2 * math.pi, 3000), rng.uniform(0, 2 * math.pi, 3000), 1.0, 0.4)
    op = nf.Operator(dev(X), dev(np.ones(3000)), (1.0, 0.05, 0.5, 0.1), nf.MATRIX_FREE)
    u = rng.normal(0.3, 0.4, size=(6, 3000)).astype(np.float32)
    u[2, 5] = np.nan
    I = nf.nf_nonlocal_apply(op, dev(u), 10.0, 0.2)
    assert torch.isnan(I[2]).all() and torch.isfinite(I[[0, 1, 3, 4, 5]]).all()
