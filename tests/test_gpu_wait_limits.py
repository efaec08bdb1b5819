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


# the update kernel of the blocked LU in both precisions, several items per group of its epilogue
@pytest.mark.parametrize("precision,M,N,W", [("fp64", 57, 14, 400), ("mixed", 123, 14, 200)])
def test_blocked_lu_gives_up_and_recovers(ftq, precision, M, N, W):
    p = _context(ftq, ftq.FTQ_FP64 if precision == "fp64" else ftq.FTQ_MIXED, M, N, W, 1)
    f = torch.from_numpy(gaussian_fields(43 + M, 5, W, p.n_alpha)).cuda()
    G0, w0 = _clean_run(p, f)                             # a stabilisation at slice 5
    # a slice whose chain and G both give up, and its launches: scales, form, G and tail, three per
    # panel of 32 columns, and an update beside every panel but the last, forward and backward
    p.reset()
    before = p.profile_read()["green"][1]
    p.set_wait_limit(0)
    p.propagate(f[:1].contiguous())
    torch.cuda.synchronize()
    panels = (M + 31) // 32
    assert p.profile_read()["green"][1] - before == 4 + 3 * panels + 2 * (panels - 1)
    assert p.status() == FTQ_ETIMEOUT
    # the T^-1 update alone: of a stabilisation's kernels only the update waits
    p.set_wait_limit(-1)
    p.reset()
    p.propagate(f[:1].contiguous())
    assert p.status() == 0
    p.set_wait_limit(0)
    p.stabilise()
    torch.cuda.synchronize()
    assert p.status() == FTQ_ETIMEOUT
    assert p.status() == 0
    p.set_wait_limit(-1)
    G1, w1 = _clean_run(p, f)
    assert torch.equal(G1, G0) and torch.equal(w1, w0)
    p.close()
