"""A NaN among the generator's parameters reaches the outputs that its tap serves and no others, however many
samples a call has: calls with one, two and four samples a thread against calls of four samples, which take
one output per thread. The tap is in the middle of the first kernel, so the outputs at both ends of the long
axis stay finite."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [32, 33, 65, 130])
@pytest.mark.parametrize("channel", [0, 7])
def test_nan_stays_within_reach(n, channel):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2106_00712_gb300 import nmc
    # hidden layer 28 x 6 x 5, 33 long kernel: enough work for lanes on samples from 32 samples on
    arch = nmc.gen_arch(z=(3, 2, 2), c1=8, k1=(26, 5, 4), k2=(33, 7, 2))
    with nmc.Generator(6, 6, 1.0, 4.0, 6.0, 0.1, 5, arch=arch, seed=4, max_batch=4,
                       lattice="honeycomb") as g:
        assert n * 6 * 5 * (33 * 7 * 2) >= 140000
        params = g.params()
        rng = np.random.default_rng(n)
        params[0][0][:] = rng.uniform(-0.2, 0.2, params[0][0].shape)
        params[1][0][:] = rng.uniform(-0.2, 0.2, params[1][0].shape)
        params[0][0][0, channel, 13, 2, 1] = np.nan
        g.set_params(params)
        p = torch.zeros((n, g.L_tau, g.A, g.B), device="cuda")
        q = torch.zeros_like(p)
        g.probs(0, n, 1, p.data_ptr())
        for k in range(0, n, 4):
            g.probs(k, min(4, n - k), 1, q[k:].data_ptr())
    assert bool(torch.isnan(q).any()) and bool(torch.isfinite(q).any())
    assert torch.equal(torch.isnan(p), torch.isnan(q))
    assert torch.equal(p.nan_to_num(2.0), q.nan_to_num(2.0))
