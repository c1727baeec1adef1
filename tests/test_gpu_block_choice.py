"""The node block of the symmetric kernel is timed per operator and kept for operators like it.  An
operator of the same size and form with another kernel is not like it: its own choice costs no
more than the better of the two blocks, whatever operator came first."""
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


def test_another_kernel_makes_its_own_choice(nf):
    n = 29000
    g = torch.Generator(device="cuda")
    g.manual_seed(0)
    x = 2.0 * torch.rand(n, 3, generator=g, device="cuda") - 1.0
    q, u = torch.full((n,), 1.0 / n, device="cuda"), torch.rand(1, n, generator=g, device="cuda")
    be, th, out = torch.full((1,), 20.0, device="cuda"), torch.full((1,), 0.2, device="cuda"), torch.empty_like(u)
    e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]

    def best(op):
        ms = []
        for _ in range(12):
            e[0].record()
            nf.nf_nonlocal_apply(op, u, be, th, out=out)
            e[1].record()
            torch.cuda.synchronize()
            ms.append(e[0].elapsed_time(e[1]))
        return min(ms)

    narrow, wide = (1.2, 0.02, 0.6, 0.07), (1.2, 0.08, 0.6, 0.25)
    for kern in (narrow, wide, narrow):
        op = nf.Operator(x, q, kern, nf.MATRIX_FREE)
        own = best(op)
        fixed = [best(nf.Operator(x, q, kern, nf.MATRIX_FREE).mf_schedule(s))
                 for s in (nf.MF_SYMMETRIC_512, nf.MF_SYMMETRIC_1024)]
        assert own < 1.15 * min(fixed), (kern, own, fixed, op.launch_shape())
