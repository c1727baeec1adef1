"""A step that leaves a non-finite state is reported by nf_operator_check after the adjoint's
recomputation as after the forward run, wherever in a checkpoint segment it stands."""
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


@pytest.mark.parametrize("n", [700, 3200])
@pytest.mark.parametrize("steps,C", [(1, 1), (2, 1), (4, 2)])
def test_non_finite_steps_are_reported(nf, n, steps, C):
    ns = nodesets.torus_lattice(n, seed=n)
    op = nf.Operator(dev(ns.nodes), dev(np.full(n, ns.area / n)), (1.0, 0.1, 0.5, 0.2), nf.MATRIX_FREE)
    lam = torch.ones(1, n, device="cuda")
    ck = torch.zeros((steps // C + 1, 1, n), device="cuda")
    ck[:, 0, 3] = float("nan")
    nf.nf_adjoint(op, ck, C, 0.0, 0.05, steps, 20.0, 0.2, lam)
    with pytest.raises(nf.NFError) as ei:
        op.check()
    assert ei.value.name == "NF_ERR_NONFINITE"
