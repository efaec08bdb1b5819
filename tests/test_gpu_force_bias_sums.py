"""The pair sums of the mixed path's force bias over the FP32 Green's function,
at FP64 accuracy: entries of G span many orders of magnitude, and every rounding
of the sum must stay below those of an FP64 sum.

gauss_k = x . xbar - xbar . xbar / 2 of a slice whose fields are zero but for one
of 1024 shows that field's xbar; the reference sums the same FP32 entries exactly.
Tolerance: a dozen FP64 roundings (2^-53) of the terms' magnitudes, taken as 16."""
import math

import numpy as np
import pytest

from synthetic_inputs import gaussian_fields

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,rs,theta", [(57, 14, 1.0, 0.125), (123, 14, 0.5, 0.125), (257, 66, 1.0, 0.0625)])
def test_force_bias_sums_of_fp32_entries(M, N, rs, theta):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2012_12228_gb300 as ftq
    from oracle.ueg import UEG
    W, dtau = 8, 0.025
    s = UEG(N, M, rs, theta, dtau)
    p = ftq.Propagator(N, M, rs, theta, dtau, walkers=W, precision=ftq.FTQ_MIXED)
    p.propagate(torch.from_numpy(gaussian_fields(19 + M, 3, W, p.n_alpha)).cuda())
    G = p.green().cpu().numpy()                           # FP32 entries widened
    assert np.array_equal(G, G.astype(np.complex64).astype(np.complex128))
    x = np.zeros((1, W, p.n_alpha))
    x[0, np.arange(W), np.arange(W)] = 1024.0             # walker w: field w (the transfers with the most pairs)
    p.propagate(torch.from_numpy(x).cuda())
    gauss = p.weights()[:, 5:7].cpu().numpy()
    p.close()

    n = np.array(s.nvec)
    d = n[:, None, :] - n[None, :, :]
    code = ((d[..., 0] + 64) * 128 + d[..., 1] + 64) * 128 + d[..., 2] + 64
    half = np.array(s.q_half)
    c = np.array(s.cq_half)
    q_code = ((half[:, 0] + 64) * 128 + half[:, 1] + 64) * 128 + half[:, 2] + 64
    pairs = [np.nonzero(code == k) for k in q_code]       # (a, b) with n_a - n_b = Q
    sdt = math.sqrt(s.dtau)
    for w in range(W):
        xb = np.zeros(p.n_alpha, dtype=np.complex128)
        size = np.zeros(p.n_alpha)
        for q, (a, b) in enumerate(pairs):
            rp = -complex(math.fsum(G[w][b, a].real), math.fsum(G[w][b, a].imag))
            rm = -complex(math.fsum(G[w][a, b].real), math.fsum(G[w][a, b].imag))
            xb[2 * q] = -sdt * 2j * c[q] * (rp + rm)
            xb[2 * q + 1] = sdt * 2.0 * c[q] * (rp - rm)
            size[2 * q:2 * q + 2] = sdt * 2.0 * c[q] * (abs(rp) + abs(rm))
        ref = 1024.0 * xb[w] - 0.5 * complex(math.fsum((xb * xb).real), math.fsum((xb * xb).imag))
        tol = 16 * 2.0 ** -53 * (1024.0 * size[w] + (size ** 2).sum())
        print(f"M={M} walker {w}: error / tolerance {abs(complex(*gauss[w]) - ref) / tol:.2f}")
        assert abs(complex(*gauss[w]) - ref) < tol

