"""Accuracy of the sums of small sets and of several trajectories by themselves, against FP64 (the
library's bar of 1e-5 would not see them degrade).

Bar.  The exponent a = r^2 / s^2 (in powers of 2) of a pair is formed from the caller's FP32
coordinates by a difference, a square, the sum of squares and a scale factor, each rounded to
2^-24: relative error at most 4 * 2^-24.  Over the pairs that make up a sum a averages below 2, so
the sum is off by at most 4 * 2^-24 * 2 * ln 2 = 3.3e-7 of itself.  Coordinates rounded to the
kernel's units first have an error of 2^-24 of their own size instead, which is larger the
narrower the kernel: a Gaussian of width 0.05 on the torus of 2,003 nodes was off by 6.5e-7."""
import math

import numpy as np
import pytest
import torch

import nodesets

pytestmark = pytest.mark.gpu

BAR = 3.3e-7
KERNELS = {"ratio4": (1.0, 0.1, 0.5, 0.2), "narrow": (1.0, 0.05, 0.5, 0.1), "general": (1.2, 0.08, 0.6, 0.25),
           "one": (1.0, 0.1, 0.0, 0.2)}


@pytest.fixture(scope="module")
def nf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2504_13379_gb300 as nf
    nf.lib()
    return nf


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float32), device="cuda")


def _nodes(shape, n):
    if shape == "torus":
        return nodesets.torus_lattice(n + n % 2, seed=0).nodes[:n]
    if shape == "square":
        return np.concatenate([np.random.default_rng(n).uniform(0, 1, (n, 2)), np.zeros((n, 1))], 1)
    i = np.arange(n) + 0.5
    z, phi = 1.0 - 2.0 * i / n, math.pi * (1.0 + math.sqrt(5.0)) * i
    s = np.sqrt(1.0 - z * z)
    return np.stack([s * np.cos(phi), 0.8 * s * np.sin(phi), 0.6 * z], 1)


@pytest.mark.parametrize("n", [500, 2003, 5000])
@pytest.mark.parametrize("shape", ["torus", "square", "ellipsoid"])
@pytest.mark.parametrize("name", sorted(KERNELS))
def test_sums_against_fp64(nf, name, shape, n):
    kern, rng = KERNELS[name], np.random.default_rng(n)
    x, q, u = dev(_nodes(shape, n)), dev(rng.uniform(0.5, 1.5, n) / n), dev(rng.normal(0.3, 0.4, (12, n)))
    A1, s1, A2, s2 = (float(np.float32(v)) for v in kern)
    X = x.double()
    r2 = ((X[:, None] - X[None]) ** 2).sum(-1)
    g = q.double() * torch.sigmoid(20.0 * (u.double() - float(np.float32(0.2))))
    want = g @ (A1 * torch.exp(-r2 / s1 ** 2) - A2 * torch.exp(-r2 / s2 ** 2))
    op = nf.Operator(x, q, kern, nf.MATRIX_FREE)
    for B in (1, 2, 3, 4, 5, 8, 12):
        got = nf.nf_nonlocal_apply(op, u[:B].contiguous(), 20.0, 0.2).double()
        err = (got - want[:B]).norm(dim=1) / want[:B].norm(dim=1)
        assert float(err.max()) <= BAR, (B, float(err.max()))
