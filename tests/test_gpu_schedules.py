"""Back on the automatic schedule an operator runs the launch shape it was created with, whatever
schedules were asked for in between."""
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


@pytest.mark.parametrize("n", [700, 3072, 3073, 4000, 13000])
def test_automatic_schedule_is_restored(nf, n):
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    x, q, u = (torch.rand(*s, generator=g, device="cuda") for s in ((n, 3), (n,), (2, n)))
    op = nf.Operator(x, q / n, (1.0, 0.1, 0.5, 0.2), nf.MATRIX_FREE)
    shape, want = op.launch_shape(), nf.nf_nonlocal_apply(op, u, 20.0, 0.2)
    for sched in (nf.MF_SYMMETRIC_1024, nf.MF_SYMMETRIC_512, nf.MF_SYMMETRIC, nf.MF_PACKED):
        op.mf_schedule(sched)
        nf.nf_nonlocal_apply(op, u, 20.0, 0.2)
        op.mf_schedule(nf.MF_AUTO)
        assert op.launch_shape() == shape
        assert torch.equal(nf.nf_nonlocal_apply(op, u, 20.0, 0.2), want)
