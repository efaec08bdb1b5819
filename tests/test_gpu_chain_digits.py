"""The complex128 chain (FP64 FMA for small bases, bf16 digit products on the
tensor cores above) and the complex128 Green's function (one block per walker
below M = 48, the blocked LU with tensor-core updates above, panels of 32 columns
up to M = 384 and of 16 beyond) against the oracle at the edges of their tiles: the last
basis of the small kernel and the first of the tensor-core one, one 64-row
block with and without a second 32-column tile's worth of columns, a remainder
of 64 rows, a thin border row (M = 257) and two accumulation chunks (M = 305).

Tolerance: a Horner step's product is accurate to about 1e-15 normwise, a slice
has six and the path here at most four slices, so that G and ln det stay
within 1e-13 relative (an error of one digit level would show as 1e-14 times
128, one chunk or border row left out as 1e-2)."""
import numpy as np
import pytest

from oracle import afqmc
from oracle.ueg import UEG
from synthetic_inputs import gaussian_fields

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,rs,slices,order", [(7, 2, 1.0, 4, 6), (19, 2, 1.0, 4, 6), (27, 14, 1.0, 4, 1),
                                                (33, 14, 1.0, 4, 6), (81, 14, 2.0, 3, 9), (123, 14, 2.0, 3, 6),
                                                (257, 66, 1.0, 2, 6), (305, 66, 1.0, 1, 6),
                                                (389, 66, 1.0, 1, 6)])
def test_chain_at_tile_edges(M, N, rs, slices, order):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2012_12228_gb300 as ftq
    W, theta, dtau = 3, 0.125, 0.025
    s = UEG(N, M, rs, theta, dtau)
    f = gaussian_fields(97 + M, slices, W, s.N_alpha)
    p = ftq.Propagator(N, M, rs, theta, dtau, walkers=W, exp_order=order)
    # one trial on both sides: with the Fermi level in a gap <N>(mu) is flat, so the
    # two bisections' roots (and with them ln det) differ by far more than the chain
    assert abs(p.query_f64("MU_T") - s.mu_T) < 1e-9
    s.mu_T, s.mu = p.query_f64("MU_T"), p.query_f64("MU")
    ref = afqmc.run(s, f, afqmc.Options(exp_order=order), n_slices=slices, want_estimator=False)
    p.propagate(torch.from_numpy(f).cuda())
    G, wt = p.green().cpu().numpy(), p.weights().cpu().numpy()
    assert p.status() == 0
    for w in range(W):
        assert np.abs(G[w] - ref[w].G).max() < 1e-13 * max(1.0, np.abs(ref[w].G).max())
        assert abs(wt[w, 3] - ref[w].logdet.real) < 1e-13 * max(1.0, abs(ref[w].logdet.real))
    p.close()


def test_fp32_lu_with_narrow_panels():
    """M = 691, the first closed shell beyond the 32-column panels of the mixed path's blocked
    LU, against the complex128 path with the bounds of the other mixed Green's-function tests:
    1e-4 for G, and M 2^-20 for ln det, a sum of M FP32 log-pivots.  (The CUDA-core LU is no
    reference here: its ln det is 3e-4 off.)"""
    import __graft_entry__
    __graft_entry__.build()
    import paper_2012_12228_gb300 as ftq
    N, M, rs, theta, dtau, W = 66, 691, 1.0, 0.5, 0.05, 2
    out = []
    for precision in (ftq.FTQ_FP64, ftq.FTQ_MIXED):
        p = ftq.Propagator(N, M, rs, theta, dtau, walkers=W, precision=precision)
        if precision == ftq.FTQ_MIXED:
            p.set_green_kernel(1)
        p.propagate(torch.from_numpy(gaussian_fields(5, 1, W, p.n_alpha)).cuda())
        out.append((p.green().cpu().numpy(), p.weights().cpu().numpy()))
        assert p.status() == 0
        p.close()
    (Ga, wa), (Gb, wb) = out
    assert np.abs(Ga - Gb).max() < 1e-4 * np.abs(Ga).max()
    assert (np.abs(wa[:, 3] - wb[:, 3]) < M * 2.0 ** -20).all()
