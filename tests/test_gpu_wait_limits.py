"""Bounded waits that run out in the tensor-core kernels whose CTAs walk several
work items: cut to zero polls, a launch latches FTQ_ETIMEOUT, ends its own
copies and MMAs with the normal bound and frees its tensor memory, and after a
reset the same context reproduces a clean run bit for bit.

The bases are the smallest that launch each kernel, the walkers enough for more
items than SMs."""
import pytest

from synthetic_inputs import gaussian_fields

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FTQ_ETIMEOUT = -4


@pytest.fixture(scope="module")
def ftq():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2012_12228_gb300 as m
    return m


def _context(ftq, precision, M, N, W, green_kernel):
    p = ftq.Propagator(N, M, 1.0, 0.25, 0.05, walkers=W, precision=precision)
    if precision == ftq.FTQ_MIXED:
        p.set_green_kernel(green_kernel)
    return p


def _clean_run(p, fields):
    p.reset()
    p.propagate(fields)
    assert p.status() == 0
    return p.green(), p.weights()


# the digit chain (M = 27, beside the one-block G), the item-list mixed chain (M = 81, CUDA-core G)
@pytest.mark.parametrize("precision,M,N,W,green_kernel", [("fp64", 27, 14, 400, 0), ("mixed", 81, 14, 400, 2)])
def test_chain_gives_up_and_recovers(ftq, precision, M, N, W, green_kernel):
    p = _context(ftq, ftq.FTQ_FP64 if precision == "fp64" else ftq.FTQ_MIXED, M, N, W, green_kernel)
    f = torch.from_numpy(gaussian_fields(41 + M, 3, W, p.n_alpha)).cuda()
    G0, w0 = _clean_run(p, f)
    p.reset()
    p.set_wait_limit(0)
    p.propagate(f[:1].contiguous())
    torch.cuda.synchronize()
    assert p.status() == FTQ_ETIMEOUT
    assert p.status() == 0
    p.set_wait_limit(-1)
    G1, w1 = _clean_run(p, f)
    assert torch.equal(G1, G0) and torch.equal(w1, w0)
    p.close()
