"""A ragged batch whose members all run a slice's Horner steps in one launch
(M <= 64): no work list of the batched chain is left, the results are those of
single contexts, and the wait limit set on the batch rules the members' chains."""
import pytest

from synthetic_inputs import gaussian_fields

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FTQ_ETIMEOUT = -4
SYSTEMS = [dict(N=2, M=7, rs=1.0, theta=0.5, dtau=0.05, walkers=5),
           dict(N=14, M=33, rs=1.0, theta=0.25, dtau=0.05, walkers=3),
           dict(N=14, M=57, rs=1.0, theta=0.125, dtau=0.05, walkers=2)]


def test_batch_of_small_members():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2012_12228_gb300 as ftq
    b = ftq.Batch(SYSTEMS)
    fields = [torch.from_numpy(gaussian_fields(61 + k, 7, m.W, m.n_alpha)).cuda() for k, m in enumerate(b.members)]
    b.propagate(fields)                                   # seven slices: across a stabilisation
    for s, m, f in zip(SYSTEMS, b.members, fields):
        p = ftq.Propagator(s["N"], s["M"], s["rs"], s["theta"], s["dtau"], walkers=s["walkers"],
                           precision=ftq.FTQ_MIXED)
        p.propagate(f)
        assert m.status() == 0 and p.status() == 0
        assert torch.equal(m.green(), p.green()) and torch.equal(m.weights(), p.weights())
        p.close()
    G0 = [m.green() for m in b.members]
    for m in b.members:
        m.reset()
    assert b.lib.ftq_set_wait_limit(b.h, 0) == 0
    b.propagate([f[:1].contiguous() for f in fields])
    torch.cuda.synchronize()
    assert [m.status() for m in b.members] == [FTQ_ETIMEOUT] * len(SYSTEMS)
    assert b.lib.ftq_set_wait_limit(b.h, -1) == 0
    for m in b.members:
        m.reset()
    b.propagate(fields)
    for m, g in zip(b.members, G0):
        assert m.status() == 0 and torch.equal(m.green(), g)
    b.close()


def test_autotune_times_the_chain_that_runs():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2012_12228_gb300 as ftq
    s = SYSTEMS[2]
    out = []
    for tune in (False, True):
        p = ftq.Propagator(s["N"], s["M"], s["rs"], s["theta"], s["dtau"], walkers=9, precision=ftq.FTQ_MIXED)
        f = torch.from_numpy(gaussian_fields(71, 4, 9, p.n_alpha)).cuda()
        p.propagate(f[:2].contiguous())
        if tune:
            before = p.profile_read()["chain"][1]
            tiles, ms = p.autotune()
            assert tiles == 1 and ms > 0
            assert p.profile_read()["chain"][1] - before == 4      # a warm-up and three timed slices
            p.set_green_kernel(0)
        p.propagate(f[2:].contiguous())                   # no stabilisation: the QR panel does not enter
        out.append((p.green(), p.weights()))
        assert p.status() == 0
        p.close()
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
