"""The first sum of an operator, made on a stream of its own while the default stream is busy: its work
arrays are cleared on the stream that uses them, so that padded columns are zero before the first
kernel reads them and no late clearing meets a later call.  Bit-identical to a repeated call."""
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


@pytest.mark.parametrize("path,n,B", [("MATRIX_FREE", 1100, 1), ("MATRIX_FREE", 3500, 5), ("DENSE_FP32", 1100, 2)])
def test_first_call_beside_a_busy_default_stream(nf, path, n, B):
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    x = torch.rand(n, 3, generator=g, device="cuda")
    q = torch.rand(n, generator=g, device="cuda") / n
    u = torch.rand(B, n, generator=g, device="cuda")
    be, th = torch.full((B,), 20.0, device="cuda"), torch.full((B,), 0.2, device="cuda")
    op = nf.Operator(x, q, (1.0, 0.1, 0.5, 0.2), getattr(nf, path))
    out = torch.empty_like(u)
    nan = [torch.full((1 << s,), float("nan"), device="cuda") for s in range(10, 22) for _ in range(4)]
    del nan  # so that new device memory does not start as zeros
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    torch.cuda._sleep(int(2e8))  # about a tenth of a second on the default stream
    with torch.cuda.stream(s):
        nf.nf_nonlocal_apply(op, u, be, th, out=out)
        first = out.clone()
    torch.cuda.synchronize()
    assert torch.equal(first, nf.nf_nonlocal_apply(op, u, be, th))
    op.check()
