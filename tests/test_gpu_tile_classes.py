"""Tile classes of the symmetric pair kernels: tiles whose pairs add exactly nothing are skipped and
tiles whose narrow Gaussian is below the wide one's last bit take one exponential.  Nodes that
only far nodes reach show a class taken too early at once (their sums are made of nothing else),
so the firing rates are non-zero in one cluster only, and the far nodes are compared by themselves.

Bars: 1e-5 relative L2 over all nodes, as for every sum of the library.  Far nodes: coordinates of
up to 128 exponent units carry FP32 rounding errors of 2^-18, at distances up to 12 units the
exponent is then off by up to 2 * 12 * 4 * 2^-18 = 4e-4 (3 coordinates, two nodes) and, for the
narrow Gaussian of ratio 4, its power by four times that: 1e-3 of each term and of the sum.  A
missing or misclassed term is an error of order 1 there."""
import math

import numpy as np
import pytest
import torch

import nodesets

pytestmark = pytest.mark.gpu

L = float(np.float32(2.0 * math.pi))
KERNELS = {
    "ratio4": (1.0, 0.05, 0.5, 0.1),
    "ratio4_wide": (1.0, 0.1, 0.5, 0.2),
    "ratio3": (0.7, 0.06, 0.4, 0.06 * math.sqrt(3.0)),
    "ratio2": (1.0, 0.05, 2.0, 0.05 * math.sqrt(2.0)),
    "steep_ratio4": (1.0e4, 0.05, 0.5, 0.1),
    "no_narrow": (0.0, 0.05, 0.5, 0.1),
    "general": (1.2, 0.04, 0.6, 0.13),
    "general_reversed": (1.2, 0.13, 0.6, 0.04),
    "one": (1.0, 0.06, 0.0, 0.2),
}


@pytest.fixture(scope="module")
def nf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2504_13379_gb300 as nf
    nf.lib()
    return nf


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float32), device="cuda")


def _case(shape, n, seed):
    """Nodes, weights and a state whose firing rates vanish outside one cluster."""
    rng = np.random.default_rng(seed)
    if shape == "torus":
        X = nodesets.torus_point(rng.uniform(0, 2 * math.pi, n), rng.uniform(0, 2 * math.pi, n), 1.0, 0.4)
    else:
        X = np.concatenate([rng.uniform(0, L, (n, 2)), np.zeros((n, 1))], 1)
    X = X.astype(np.float32)
    q = rng.uniform(0.5, 1.5, n).astype(np.float32)
    d = X.astype(np.float64) - X[0]
    u = np.where((d ** 2).sum(1) < 0.15, rng.uniform(0.0, 0.5, n), -1e3).astype(np.float32)
    return X, q, u


def _reference(X, q, u, kern, beta, theta, per):
    X, q, u = (np.asarray(a, dtype=np.float64) for a in (X, q, u))
    A1, s1, A2, s2 = (float(np.float32(v)) for v in kern)
    with np.errstate(over="ignore"):
        g = q / (1.0 + np.exp(-beta * (u - float(np.float32(theta)))))
    live = g > 0
    D = X[:, None, :] - X[None, live, :]
    if per:
        D[..., :2] -= per * np.rint(D[..., :2] / per)
    r2 = (D ** 2).sum(-1)
    I = (A1 * np.exp(-r2 / s1 ** 2) - A2 * np.exp(-r2 / s2 ** 2)) @ g[live]
    # far nodes: the narrow Gaussian below 2^-36 of its peak, the wide one above 2^-100
    u2 = r2.min(1) * math.log2(math.e)
    wide = max(s1 if A1 else 0.0, s2 if A2 else 0.0)
    return I, (u2 > 36.0 * min(s1, s2) ** 2) & (u2 < 100.0 * wide ** 2)


@pytest.mark.parametrize("n", [1000, 1025, 3071, 5000])
@pytest.mark.parametrize("shape", ["torus", "square", "periodic"])
@pytest.mark.parametrize("name", sorted(KERNELS))
def test_sums_node_by_node(nf, name, shape, n):
    kern, per = KERNELS[name], (L if shape == "periodic" else 0.0)
    X, q, u = _case(shape, n, 3)
    want, far = _reference(X, q, u, kern, 10.0, 0.2, per)
    op = nf.Operator(dev(X), dev(q), kern + (per,), nf.MATRIX_FREE)
    for sched in (nf.MF_SYMMETRIC_1024, nf.MF_SYMMETRIC_512):
        op.mf_schedule(sched)
        err = np.abs(nf.nf_nonlocal_apply(op, dev(u), 10.0, 0.2).double().cpu().numpy() - want)
        assert np.linalg.norm(err) <= 1e-5 * np.linalg.norm(want)
        assert np.all(err[far] <= 1e-3 * np.abs(want[far])), np.max(err[far] / np.abs(want[far]))


def test_non_finite_values_spread(nf):
    """A NaN state reaches every node, however narrow the kernel, as in the plain sum."""
    X, q, u = _case("torus", 3000, 4)
    for kern in (KERNELS["ratio4"], KERNELS["one"], KERNELS["general"]):
        op = nf.Operator(dev(X), dev(q), kern, nf.MATRIX_FREE).mf_schedule(nf.MF_SYMMETRIC_1024)
        v = u.copy()
        v[17] = np.nan
        assert torch.isnan(nf.nf_nonlocal_apply(op, dev(v), 10.0, 0.2)).all()


@pytest.mark.parametrize("name", ["ratio4", "ratio2", "general", "one"])
@pytest.mark.parametrize("n", [1025, 5000])
def test_gradients_against_fp64(nf, name, n):
    """One RK4 step: the adjoint's sums over classed tiles against dense FP64 autograd."""
    kern = KERNELS[name]
    X, q, _ = _case("torus", n, 5)
    rng = np.random.default_rng(6)
    u0 = rng.normal(0.1, 0.3, n).astype(np.float32)
    lam = rng.normal(0.0, 1.0, n).astype(np.float32)
    q = (q / n).astype(np.float32)
    dt, beta, theta = 0.1, 5.0, float(np.float32(0.2))
    op = nf.Operator(dev(X), dev(q), kern, nf.MATRIX_FREE)
    u = dev(u0)[None].contiguous()
    ck = torch.empty((2, 1, n), device="cuda")
    nf.nf_rk4_advance(op, u, 0.0, dt, 1, beta, theta, ckpt=ck, C_every=1)
    gu, gk = nf.nf_adjoint(op, ck, 1, 0.0, dt, 1, beta, theta, dev(lam)[None].contiguous())
    x, qd = dev(X).double(), dev(q).double()
    kp = torch.tensor([float(np.float32(v)) for v in kern], dtype=torch.float64, device="cuda", requires_grad=True)
    v0 = dev(u0).double().requires_grad_(True)
    r2 = ((x[:, None] - x[None]) ** 2).sum(-1)
    W = kp[0] * torch.exp(-r2 / kp[1] ** 2) - kp[2] * torch.exp(-r2 / kp[3] ** 2)
    f = lambda U: -U + W @ (qd * torch.sigmoid(beta * (U - theta)))
    k1 = f(v0)
    k2 = f(v0 + 0.5 * dt * k1)
    k3 = f(v0 + 0.5 * dt * k2)
    k4 = f(v0 + dt * k3)
    uT = v0 + dt / 6.0 * (k1 + 2 * k2 + 2 * k3 + k4)
    wu, wk = torch.autograd.grad((uT * dev(lam).double()).sum(), (v0, kp))
    assert (gu.double()[0] - wu).norm() <= 1e-5 * wu.norm()
    assert (gk.double()[0] - wk).norm() <= 1e-4 * wk.norm()
