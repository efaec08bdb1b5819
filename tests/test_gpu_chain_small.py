"""The mixed-precision chain of small bases (a slice's Horner steps in one
launch, V and the chain in shared memory) against the complex128 path: one to
four 32-float k tiles (M = 7, 19, 33, 57), more walkers than blocks and fewer, one
Horner step and several, across a stabilisation.

Tolerance: the chain rounds to 2^-22 relative per slice and G is FP32, so G
agrees within 1e-5 (as the tensor-core and CUDA-core chains do)."""
import numpy as np
import pytest

from synthetic_inputs import gaussian_fields

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,W,order", [(7, 2, 3, 6), (19, 2, 400, 2), (33, 14, 9, 1), (33, 14, 200, 6), (57, 14, 170, 6)])
def test_small_basis_chain_vs_complex128(M, N, W, order):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2012_12228_gb300 as ftq
    n = 7
    out = []
    for precision in (ftq.FTQ_FP64, ftq.FTQ_MIXED):
        p = ftq.Propagator(N, M, 1.0, 0.25, 0.05, walkers=W, precision=precision, exp_order=order)
        p.propagate(torch.from_numpy(gaussian_fields(11 + M, n, W, p.n_alpha)).cuda())
        out.append((p.green().cpu().numpy(), p.weights().cpu().numpy()))
        assert p.status() == 0
        p.close()
    (Ga, wa), (Gb, wb) = out
    assert np.abs(Ga - Gb).max() < 1e-5 * np.abs(Ga).max()
    assert np.array_equal(wa[:, 2], wb[:, 2])
