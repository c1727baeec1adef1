"""The adjoint differentiates around the very states of the forward run: stage inputs recomputed from a
checkpoint take the forward's kernels, so the gradients do not depend on the checkpoints' spacing
to the last bit."""
import numpy as np
import pytest
import torch

import nodesets

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2504_13379_gb300 as nf
    nf.lib()
    return nf


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float32), device="cuda")


def _case(nf, n, B, kern):
    ns = nodesets.torus_lattice(n, seed=n)
    rng = np.random.default_rng(n + B)
    op = nf.Operator(dev(ns.nodes), dev(np.full(ns.n, ns.area / ns.n)), kern, nf.MATRIX_FREE)
    return op, dev(rng.normal(0.2, 0.4, (B, ns.n))), dev(rng.normal(0.0, 1.0, (B, ns.n)))


@pytest.mark.parametrize("n,B,kern", [(700, 1, (1.0, 0.1, 0.5, 0.2)), (1500, 3, (1.0, 0.1, 0.5, 0.2)),
                                      (3072, 2, (1.2, 0.08, 0.6, 0.25)), (3200, 1, (1.0, 0.1, 0.5, 0.2)),
                                      (1500, 5, (1.0, 0.1, 0.5, 0.2))])
def test_gradients_do_not_depend_on_the_checkpoints(nf, n, B, kern):
    op, u0, lam = _case(nf, n, B, kern)
    steps, dt, grads = 12, 0.05, []
    for C in (1, 4, 12):
        u = u0.clone()
        ck = torch.empty((steps // C + 1, B, op.n), device="cuda")
        nf.nf_rk4_advance(op, u, 0.0, dt, steps, 20.0, 0.2, ckpt=ck, C_every=C)
        grads.append(nf.nf_adjoint(op, ck, C, 0.0, dt, steps, 20.0, 0.2, lam))
    for gu, gk in grads[1:]:
        assert torch.equal(gu, grads[0][0]) and torch.equal(gk, grads[0][1])
    op.check()
