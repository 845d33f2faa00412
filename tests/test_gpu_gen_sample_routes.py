"""Generator outputs at the edges of the rules that choose how samples are laid over lanes: just below
and above the work from which lanes hold samples (162 and 163 samples of this network), one, two and
four samples per thread (the last group full, nearly empty and of odd size), past one internal chunk
(256). Equal bit for bit to the same samples in calls of eight, which are below the rule: the
multiply-adds and their order are the same."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SMALL = ("square", 6, 6, 0.9, dict(z=(2, 2, 2), c1=3, k1=(3, 2, 3), k2=(6, 4, 3)))
PAPER = ("honeycomb", 6, 6, 6.0, dict())   # one sample per thread up to 32, two up to 64


@pytest.mark.parametrize("case,n", [(SMALL, n) for n in (161, 162, 163, 164, 193, 255, 256, 259)]
                         + [(PAPER, n) for n in (31, 32, 33, 35, 62, 64, 65, 129)])
def test_routes_agree(case, n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2106_00712_gb300 import nmc
    lattice, Lx, Ly, beta, arch = case
    with nmc.Generator(Lx, Ly, 1.0, 4.0, beta, 0.1, 3, arch=nmc.gen_arch(**arch), seed=3,
                       max_batch=4, lattice=lattice) as g:
        rng = np.random.default_rng(n)
        g.set_params([(W, rng.uniform(-0.3, 0.3, b.shape).astype(np.float32))
                      for W, b in g.params()])
        p = torch.full((n, g.L_tau, g.A, g.B), float("nan"), device="cuda")
        g.probs(2, n, 1, p.data_ptr())
        q = torch.empty_like(p)
        for k in range(0, n, 8):
            g.probs(2 + k, min(8, n - k), 1, q[k:].data_ptr())
        assert torch.equal(p, q)
        assert 0 < float(p.min()) and float(p.max()) < 1
