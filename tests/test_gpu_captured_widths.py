"""A caller's CUDA graph of nf_nonlocal_apply stays valid while the operator serves calls of other
widths: the work arrays that the capture names are kept when a call needs larger ones, also where
fewer trajectories need more (two buffers of firing rates up to 3,072 nodes, one partial slot per
node block above).  Bit-identical to a direct call: the same kernels in the same order."""
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


@pytest.mark.parametrize("path,n,B,others", [("MATRIX_FREE", 2100, 5, (3,)), ("MATRIX_FREE", 2100, 4, (12,)),
                                             ("MATRIX_FREE", 4000, 4, (3, 9)), ("MATRIX_FREE", 14000, 4, (3,)),
                                             ("DENSE_SYM_FP32", 1500, 1, (2, 7)), ("DENSE_FP32", 4000, 40, (32, 50))])
def test_captured_apply_survives_other_widths(nf, path, n, B, others):
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
    held = []
    for b in others:
        v = torch.rand(b, n, generator=g, device="cuda")
        nf.nf_nonlocal_apply(op, v, 20.0, 0.2)
        nf.nf_rk4_advance(op, v, 0.0, 0.05, 2, 20.0, 0.2)
        held += [torch.full((1 << 18,), -7.0, device="cuda") for _ in range(16)]
    u.copy_(torch.rand(B, n, generator=g, device="cuda"))
    torch.cuda.synchronize()
    for _ in range(2):
        out.zero_()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        got = out.clone()
        assert torch.equal(got, nf.nf_nonlocal_apply(op, u, 20.0, 0.2))
        assert float(got.abs().max()) > 0.0
    assert all(bool((t == -7.0).all()) for t in held)
    op.check()
