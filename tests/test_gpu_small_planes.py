"""FP32 planes of small node sets with many trajectories: passes over the plane up to a count, one GEMM
from there on.  Both sides of the line against FP64 within the library's 1e-5 bar, and the line by
time: a smaller plane takes no longer than the next larger one, which always uses the GEMM."""
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


KERN = (1.0, 0.3, 0.5, 0.6)


def _case(nf, n, B):
    g = torch.Generator(device="cuda")
    g.manual_seed(n + B)
    x = 2.0 * torch.rand(n, 3, generator=g, device="cuda") - 1.0
    q = (0.5 + torch.rand(n, generator=g, device="cuda")) / n
    u = 0.3 + 0.4 * torch.randn(B, n, generator=g, device="cuda")
    return nf.Operator(x, q, KERN, nf.DENSE_FP32), x, q, u


@pytest.mark.parametrize("n", [700, 1024, 1025, 2048])
@pytest.mark.parametrize("B", [168, 169, 256])
def test_both_sides_match_fp64(nf, n, B):
    op, x, q, u = _case(nf, n, B)
    got = nf.nf_nonlocal_apply(op, u, 20.0, 0.2).double()
    r2 = torch.cdist(x.double(), x.double(), compute_mode="donot_use_mm_for_euclid_dist") ** 2
    A1, s1, A2, s2 = (float(np.float32(v)) for v in KERN)
    W = A1 * torch.exp(-r2 / s1 ** 2) - A2 * torch.exp(-r2 / s2 ** 2)
    want = (q.double() * torch.sigmoid(20.0 * (u.double() - float(np.float32(0.2))))) @ W
    assert float(((got - want).norm(dim=1) / want.norm(dim=1)).max()) < 1e-5


def test_many_trajectories_on_a_small_plane(nf):
    def best(n, B):
        op, _, _, u = _case(nf, n, B)
        be, th, out = torch.full((B,), 20.0, device="cuda"), torch.full((B,), 0.2, device="cuda"), torch.empty_like(u)
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        ms = []
        for _ in range(12):
            e[0].record()
            for _ in range(4):
                nf.nf_nonlocal_apply(op, u, be, th, out=out)
            e[1].record()
            torch.cuda.synchronize()
            ms.append(e[0].elapsed_time(e[1]))
        return min(ms)

    for n in (1000, 2000):
        assert best(n, 512) < 1.2 * best(2500, 512)
