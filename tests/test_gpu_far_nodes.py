"""Tile classes where a wrong one shows at once, on every kernel that takes them: nodes that only far
nodes reach have sums made of nothing else.  The firing rates are non-zero in one cluster only; the far nodes
are compared one by one, on the 256- and 128-node blocks of the small sets, on the packed kernel
and with four and five trajectories (the multi-trajectory kernel).

Bar as for the large blocks: coordinates of up to 128 exponent units carry rounding errors of
2^-18, so exponents of up to 12 units are off by at most 4e-4, and the narrow Gaussian of ratio 4
by four times that: 1e-3 of each sum.  A missing or misclassed tile is an error of order 1."""
import math

import numpy as np
import pytest
import torch

import nodesets

pytestmark = pytest.mark.gpu

L = float(np.float32(2.0 * math.pi))
KERNELS = {"ratio4": (1.0, 0.05, 0.5, 0.1), "ratio3": (0.7, 0.06, 0.4, 0.06 * math.sqrt(3.0)),
           "ratio2": (1.0, 0.05, 2.0, 0.05 * math.sqrt(2.0)), "steep_ratio4": (1.0e4, 0.05, 0.5, 0.1),
           "no_narrow": (0.0, 0.05, 0.5, 0.1), "general": (1.2, 0.04, 0.6, 0.13),
           "general_reversed": (1.2, 0.13, 0.6, 0.04), "one": (1.0, 0.06, 0.0, 0.2)}


@pytest.fixture(scope="module")
def nf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2504_13379_gb300 as nf
    nf.lib()
    return nf


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float32), device="cuda")


@pytest.mark.parametrize("n", [1025, 3072, 3073, 5000])
@pytest.mark.parametrize("shape", ["torus", "square", "periodic"])
@pytest.mark.parametrize("name", sorted(KERNELS))
def test_far_nodes_one_by_one(nf, name, shape, n):
    kern, per = KERNELS[name], (L if shape == "periodic" else 0.0)
    rng = np.random.default_rng(3)
    if shape == "torus":
        X = nodesets.torus_point(rng.uniform(0, 2 * math.pi, n), rng.uniform(0, 2 * math.pi, n), 1.0, 0.4)
    else:
        X = np.concatenate([rng.uniform(0, L, (n, 2)), np.zeros((n, 1))], 1)
    X = X.astype(np.float32)
    near = ((X.astype(np.float64) - X[0]) ** 2).sum(1) < 0.15
    u = np.where(near, rng.uniform(0.0, 0.5, (5, n)), -1e3)
    x, q, v = dev(X), dev(rng.uniform(0.5, 1.5, n)), dev(u)
    A1, s1, A2, s2 = (float(np.float32(a)) for a in kern)
    live = torch.as_tensor(near, device="cuda")
    d = x.double()[:, None] - x.double()[None, live]
    if per:
        d = torch.cat([d[..., :2] - per * torch.round(d[..., :2] / per), d[..., 2:]], -1)
    r2 = (d * d).sum(-1)
    g = q.double()[live] * torch.sigmoid(10.0 * (v.double()[:, live] - float(np.float32(0.2))))
    want = g @ (A1 * torch.exp(-r2 / s1 ** 2) - A2 * torch.exp(-r2 / s2 ** 2)).T
    # far nodes: the narrow Gaussian below 2^-36 of its peak, the wide one above 2^-100
    e = r2.min(1).values * math.log2(math.e)
    wide = max(s1 if A1 else 0.0, s2 if A2 else 0.0)
    far = (e > 36.0 * min(s1, s2) ** 2) & (e < 100.0 * wide ** 2)
    op = nf.Operator(x, q, kern + (per,), nf.MATRIX_FREE)
    for sched in (nf.MF_AUTO, nf.MF_SYMMETRIC, nf.MF_PACKED):
        op.mf_schedule(sched)
        for B in (1, 2, 4, 5):
            got = nf.nf_nonlocal_apply(op, v[:B].contiguous(), 10.0, 0.2).double()
            err = (got - want[:B]).abs()
            assert bool((err.norm(dim=1) <= 1e-5 * want[:B].norm(dim=1)).all()), (sched, B)
            assert bool((err[:, far] <= 1e-3 * want[:B][:, far].abs()).all()), (sched, B)
