"""Estimators of walkers that are split over blocks: values and time.

Values: per walker against the oracle's formulas on the walker's own G, for
numbers of walkers that give one to eight parts. Tolerance 1e-11 of the
largest term summed: FP64 sums of fewer than 2e4 terms, each product 1e-16.

Time: a call on fewer walkers takes no longer than on more (a bad split took
1.6 times as long on 110 walkers as on 152, and longer on 152 than on 200),
least of ten calls each, with a quarter to spare."""
import numpy as np
import pytest

from oracle import afqmc
from oracle.ueg import UEG
from synthetic_inputs import gaussian_fields

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ftq():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2012_12228_gb300 as m
    return m


@pytest.mark.parametrize("M,N", [(7, 2), (19, 2), (33, 14), (57, 14)])
@pytest.mark.parametrize("W", [1, 5, 50, 76, 110, 200, 400])
def test_per_walker_estimates_for_every_split(ftq, M, N, W):
    rs, theta, dtau = 1.0, 0.25, 0.05
    s = UEG(N, M, rs, theta, dtau)
    p = ftq.Propagator(N, M, rs, theta, dtau, walkers=W)
    p.propagate(torch.from_numpy(gaussian_fields(29 + M, 2, W, p.n_alpha)).cuda())
    est = p.estimators()["per_walker"].cpu().numpy()
    G = p.green().cpu().numpy()
    assert p.status() == 0
    p.close()
    for w in sorted({0, 1 % W, W // 2, W - 1}):
        E, Nw = afqmc.local_energy(s, G[w])[:2]
        size = np.abs(np.asarray(s.eps)).sum() + np.abs(E)
        assert abs(complex(est[w, 3], est[w, 4]) - E) < 1e-11 * size
        assert abs(complex(est[w, 5], est[w, 6]) - Nw) < 1e-11 * M


def _least_ms(f, repeats=10):
    f()
    f()
    best = float("inf")
    for _ in range(repeats):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        f()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


def test_fewer_walkers_take_no_longer(ftq):
    def complex128(W):
        p = ftq.Propagator(14, 171, 0.5, 0.125, 0.05, walkers=W)
        t = _least_ms(lambda: p.estimators(per_walker=False))
        p.close()
        return t

    def tracked(W):
        p = ftq.Propagator(14, 123, 2.0, 0.25, 0.05, walkers=W, precision=ftq.FTQ_MIXED)
        x = torch.from_numpy(gaussian_fields(3, 4, W, p.n_alpha)).cuda()

        def path():
            p.reset()
            p.propagate(x)
        plain = _least_ms(path)
        p.track_estimates(1)
        t = _least_ms(path) - plain
        p.close()
        return t

    for call, few, more in ((complex128, 152, 200), (tracked, 110, 152)):
        a, b = call(few), call(more)
        print(f"{call.__name__}: {few} walkers {a:.3f} ms, {more} walkers {b:.3f} ms")
        assert a < 1.25 * b if call is tracked else a < b
