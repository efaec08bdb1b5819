"""Stabilisation of the complex128 path on bases whose T^-1 update runs as a
forward substitution with tensor-core updates (M = 48 .. 640), with more than 257
columns, against the oracle; and one slice at
M = 515, where the chain's products take three accumulation chunks.

Tolerances: those of the repository's complex128 parity, 1e-10 relative for G and
ln det across stabilisations; 1e-13 for a slice without one, as for the other bases
of the digit chain."""
import numpy as np
import pytest

from oracle import afqmc
from oracle.ueg import UEG
from synthetic_inputs import gaussian_fields

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,slices,every,tol", [(305, 3, 1, 1e-10), (389, 2, 1, 1e-10), (515, 1, 0, 1e-13)])
def test_large_bases_against_oracle(M, slices, every, tol):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2012_12228_gb300 as ftq
    N, rs, theta, dtau, W = 66, 1.0, 0.125, 0.025, 2
    s = UEG(N, M, rs, theta, dtau)
    f = gaussian_fields(83 + M, slices, W, s.N_alpha)
    p = ftq.Propagator(N, M, rs, theta, dtau, walkers=W, stabilise_every=every)
    # one trial on both sides, as in the tests of the digit chain
    assert abs(p.query_f64("MU_T") - s.mu_T) < 1e-9
    s.mu_T, s.mu = p.query_f64("MU_T"), p.query_f64("MU")
    ref = afqmc.run(s, f, afqmc.Options(stabilise_every=every), n_slices=slices, want_estimator=False)
    p.propagate(torch.from_numpy(f).cuda())
    G, wt = p.green().cpu().numpy(), p.weights().cpu().numpy()
    assert p.status() == 0
    for w in range(W):
        assert np.abs(G[w] - ref[w].G).max() < tol * max(1.0, np.abs(ref[w].G).max())
        assert abs(wt[w, 3] - ref[w].logdet.real) < tol * max(1.0, abs(ref[w].logdet.real))
    p.close()
