"""Static structure factor with transfers of at most 16 and of at most 8 pairs
sharing a warp: per walker against the oracle's formula on the walker's own G, on
bases with none, some and many transfers of each kind. Tolerance 1e-11 of the
largest entry: FP64 sums of at most 81^2 terms.

Time on a small basis with many walkers: the exchange sums are those of the
estimators, so a call takes about as long as theirs (it took 2.3 times as long
with a warp per transfer); bound 1.7, least of ten calls each."""
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


@pytest.mark.parametrize("M,N,W", [(7, 2, 3), (19, 2, 1), (27, 14, 160), (33, 14, 3), (57, 14, 330), (81, 14, 2)])
def test_per_walker_against_oracle(ftq, M, N, W):
    rs, theta, dtau = 1.0, 0.25, 0.05
    s = UEG(N, M, rs, theta, dtau)
    p = ftq.Propagator(N, M, rs, theta, dtau, walkers=W)
    p.propagate(torch.from_numpy(gaussian_fields(37 + M, 2, W, p.n_alpha)).cuda())
    pw = p.structure_factor(per_walker=True)["per_walker"].cpu().numpy()
    G = p.green().cpu().numpy()
    assert p.status() == 0
    p.close()
    for w in sorted({0, W // 2, W - 1}):
        ref = np.empty(pw.shape[1], dtype=np.complex128)
        ref[0::2], ref[1::2] = afqmc.density_correlation(s, G[w])
        assert np.abs(pw[w] - ref).max() < 1e-11 * max(1.0, np.abs(ref).max())


def test_small_basis_takes_about_the_estimators_time(ftq):
    p = ftq.Propagator(14, 33, 1.0, 0.25, 0.05, walkers=1216)
    p.propagate(torch.from_numpy(gaussian_fields(3, 1, 1216, p.n_alpha)).cuda())

    def least(f):
        f()
        f()
        best = float("inf")
        for _ in range(10):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record()
            f()
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        return best
    sf, est = least(lambda: p.structure_factor(per_walker=True)), least(lambda: p.estimators())
    print(f"structure factor {sf:.3f} ms, estimators {est:.3f} ms")
    assert sf < 1.7 * est
    p.close()
