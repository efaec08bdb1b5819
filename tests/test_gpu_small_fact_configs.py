"""The launch shapes of the one-block complex128 factorisations by the number of
walkers (lanes per row of G, matrices in shared memory or not, lanes per column
of the QRCP, block size of the low-rank kernels): walkers on both sides of every
line, against the same walkers alone, through a stabilisation.

Tolerance 1e-12 relative, a hundredth of the repository's complex128 parity: the
shapes differ in the order of FP64 sums over at most M terms."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,low_rank", [(7, 2, 0.0), (19, 2, 0.0), (27, 14, 0.0), (33, 14, 0.0), (33, 14, 1e-6),
                                          (81, 14, 1e-6)])
def test_launch_shapes_agree(M, N, low_rank):
    import __graft_entry__
    __graft_entry__.build()
    import paper_2012_12228_gb300 as ftq
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    sizes = [2 * sms, 2 * sms + 1] if low_rank else [3 * sms // 2, 3 * sms // 2 + 1, 4 * sms, 4 * sms + 1]
    g = torch.Generator(device="cuda")
    g.manual_seed(17 + M)

    def run(W, x):
        p = ftq.Propagator(N, M, 1.0, 0.25, 0.05, walkers=W, low_rank=low_rank)
        x = 0.5 * torch.randn((6, W, p.n_alpha), generator=g, device="cuda", dtype=torch.float64) if x is None else x
        p.propagate(x)                                    # a stabilisation after slice 5
        assert p.status() == 0
        out = x, p.green(), p.weights()
        p.close()
        return out

    for W in sizes:
        x, G, w = run(W, None)
        few = [0, 1, W // 2, W - 1]
        _, G1, w1 = run(len(few), x[:, few].contiguous())
        assert (G[few] - G1).abs().max() < 1e-12 * max(1.0, G1.abs().max().item())
        assert (w[few] - w1)[:, [0, 2, 3]].abs().max() < 1e-12 * max(1.0, w1[:, [0, 3]].abs().max().item())
