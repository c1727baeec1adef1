"""A caller's CUDA graph of nf_nonlocal_apply stays valid while the operator serves other calls of the
same width: RK4 steps add the stage states beside the sums' work arrays without moving those, and the
graph holds its own copies of scalar parameters.  Bit-identical to a direct call: the sums run the
same kernels in the same order."""
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


@pytest.mark.parametrize("path,n,B", [("MATRIX_FREE", 700, 1), ("MATRIX_FREE", 3072, 2), ("MATRIX_FREE", 3073, 1),
                                      ("MATRIX_FREE", 2100, 5), ("DENSE_BF16X2", 1500, 3), ("DENSE_SYM_FP32", 1500, 1)])
def test_captured_apply_survives_other_calls(nf, path, n, B):
    g = torch.Generator(device="cuda")
    g.manual_seed(n + B)
    x = torch.rand(n, 3, generator=g, device="cuda")
    q = torch.rand(n, generator=g, device="cuda") / n
    u = torch.rand(B, n, generator=g, device="cuda")
    op = nf.Operator(x, q, (1.0, 0.1, 0.5, 0.2), getattr(nf, path))
    out = torch.empty_like(u)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        nf.nf_nonlocal_apply(op, u, 20.0, 0.2, out=out)  # allocates what the capture cannot
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        nf.nf_nonlocal_apply(op, u, 20.0, 0.2, out=out)
    v = u.clone()
    nf.nf_rk4_advance(op, v, 0.0, 0.05, 2, 20.0, 0.2)
    with torch.cuda.stream(s):
        for k in range(20):  # more scalars than an operator keeps
            nf.nf_nonlocal_apply(op, u, 1.0 + k, 0.3)
    torch.cuda.synchronize()
    junk = [torch.full((B,), -7.0, device="cuda") for _ in range(64)]
    u.copy_(torch.rand(B, n, generator=g, device="cuda"))
    out.zero_()
    torch.cuda.synchronize()
    graph.replay()
    torch.cuda.synchronize()
    got = out.clone()
    assert torch.equal(got, nf.nf_nonlocal_apply(op, u, 20.0, 0.2))
    assert float(got.abs().max()) > 0.0 and len(junk) == 64
    op.check()
