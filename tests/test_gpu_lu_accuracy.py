"""Accuracy of the mixed path's blocked LU with tensor-core updates (the default
from M = 48 up): on one slice's chain its G is no further from the complex128
path's, root mean square over all walkers and entries, than that of the
CUDA-core LU, which sums everything in FP32 FMA."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,rs,theta,dtau,W", [(57, 14, 1.0, 0.125, 0.05, 96), (123, 14, 2.0, 0.25, 0.05, 64),
                                                 (257, 66, 1.0, 0.0625, 0.025, 24)])
def test_tensor_core_lu_is_as_accurate_as_the_cuda_core_lu(M, N, rs, theta, dtau, W):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2012_12228_gb300 as ftq
    out = []
    for precision, kind in ((ftq.FTQ_FP64, 0), (ftq.FTQ_MIXED, 1), (ftq.FTQ_MIXED, 2)):
        p = ftq.Propagator(N, M, rs, theta, dtau, walkers=W, precision=precision)
        if kind:
            p.set_green_kernel(kind)
        g = torch.Generator(device="cuda")
        g.manual_seed(97 + M)
        p.propagate(torch.randn((1, W, p.n_alpha), generator=g, device="cuda", dtype=torch.float64))
        assert p.status() == 0
        out.append(p.green().clone())
        p.close()
    tc, simt = ((g - out[0]).abs().square().mean().sqrt().item() for g in out[1:])
    print(f"M={M}: rms error of G {tc:.3e} (tensor cores), {simt:.3e} (CUDA cores)")
    assert tc <= simt
