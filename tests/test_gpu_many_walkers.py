"""More walkers than the y and z dimensions of a grid hold (65,535): a whole
mixed path without stabilisation (FP32 blocked LU of G, the complex128 one at
tau = beta) and the structure factor, walker by walker as in a small context."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_mixed_path_and_structure_factor_beyond_65535_walkers():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2012_12228_gb300 as ftq
    N, M, rs, theta, W = 14, 57, 1.0, 0.5, 65537
    picked = torch.tensor([0, 1, 40000, 65534, 65535, 65536], device="cuda")
    dtau = 0.5                                            # two slices to tau = beta

    def run(walkers, fields):
        p = ftq.Propagator(N, M, rs, theta, dtau, walkers=walkers, stabilise_every=0, precision=ftq.FTQ_MIXED)
        x = fields(p)
        p.propagate(x[:1].contiguous())
        G1 = p.green()[picked if walkers == W else slice(None)].clone()
        p.propagate(x[1:].contiguous())
        out = [G1, p.green()[picked if walkers == W else slice(None)].clone(),
               p.weights()[picked if walkers == W else slice(None)].clone(),
               p.structure_factor(per_walker=True)["per_walker"][picked if walkers == W else slice(None)].clone()]
        assert p.status() == 0
        p.close()
        return x, out

    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    x, many = run(W, lambda p: 0.2 * torch.randn((p.n_slices, W, p.n_alpha), generator=g, device="cuda",
                                                 dtype=torch.float64))
    assert x.shape[0] == 2
    _, few = run(len(picked), lambda p: x[:, picked].contiguous())
    for a, b in zip(many, few):
        assert torch.equal(a, b)
