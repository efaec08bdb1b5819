"""Weights and ln det of the mixed path on small bases (a slice's Horner steps in
one launch) against the complex128 path, beside the Green's functions that the
other tests of this chain compare.

Bounds: ln det is a sum of M FP32 log-pivots, M 2^-20 as in the other mixed tests;
ln w telescopes to twice its difference plus the Gaussian factors of the seven
slices, which are given as much again."""
import numpy as np
import pytest

from synthetic_inputs import gaussian_fields

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,W,order", [(7, 2, 3, 6), (19, 2, 400, 2), (33, 14, 9, 1), (33, 14, 200, 6), (57, 14, 170, 6)])
def test_small_basis_weights_vs_complex128(M, N, W, order):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2012_12228_gb300 as ftq
    out = []
    for precision in (ftq.FTQ_FP64, ftq.FTQ_MIXED):
        p = ftq.Propagator(N, M, 1.0, 0.25, 0.05, walkers=W, precision=precision, exp_order=order)
        p.propagate(torch.from_numpy(gaussian_fields(11 + M, 7, W, p.n_alpha)).cuda())
        out.append(p.weights().cpu().numpy())
        assert p.status() == 0
        p.close()
    a, b = out
    live = a[:, 2] > 0.5
    assert live.any() and np.array_equal(a[:, 2], b[:, 2])
    assert np.abs(a[:, 3] - b[:, 3]).max() < M * 2.0 ** -20
    assert np.abs(a[live, 0] - b[live, 0]).max() < 4 * M * 2.0 ** -20
