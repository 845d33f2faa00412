"""Lanes on samples at axes off the output tile of 4 and at axes of length 1, above the work from which a call
takes them (140,000 a step: samples x hidden sites of a plane x second-kernel entries): batches at the edges
of a group and odd ones, and one past an internal chunk (256) whose rest is below the rule. Equal bit for bit
to the same samples in calls of four, which take one output per thread."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

RULE = 140000
OFF = ("square", 12, 6, 1.7, dict(z=(3, 2, 1), c1=5, k1=(3, 3, 2), k2=(13, 9, 5)))    # hidden 5 x 4 x 2
ONES = ("square", 14, 1, 3.0, dict(z=(1, 1, 1), c1=3, k1=(6, 2, 1), k2=(25, 13, 1)))  # hidden 6 x 2 x 1
FLAT = ("square", 8, 8, 0.9, dict(z=(1, 3, 2), c1=2, k1=(1, 2, 3), k2=(9, 5, 5)))     # hidden 1 x 4 x 4


@pytest.mark.parametrize("case,n", [(OFF, n) for n in (32, 33, 63, 65, 127, 130, 300)]
                         + [(ONES, n) for n in (216, 217, 255, 256, 300)]
                         + [(FLAT, n) for n in (39, 64, 131)])
def test_axes(case, n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2106_00712_gb300 import nmc
    lattice, Lx, Ly, beta, arch = case
    hidden = [a + k - 1 for a, k in zip(arch["z"], arch["k1"])]
    work = hidden[1] * hidden[2] * int(np.prod(arch["k2"]))
    assert min(n, 256) * work >= RULE and 4 * work < RULE
    with nmc.Generator(Lx, Ly, 1.0, 4.0, beta, 0.1, 1, arch=nmc.gen_arch(**arch), seed=9,
                       max_batch=4, lattice=lattice) as g:
        rng = np.random.default_rng(n)
        g.set_params([(W, rng.uniform(-0.3, 0.3, b.shape).astype(np.float32))
                      for W, b in g.params()])
        p = torch.full((n, g.L_tau, g.A, g.B), float("nan"), device="cuda")
        f = torch.zeros((n, g.L_tau, g.N), dtype=torch.int8, device="cuda")
        g.probs(5, n, 1, p.data_ptr())
        g.sample_fields(5, n, 1, f.data_ptr())
        q, h = torch.empty_like(p), torch.empty_like(f)
        for k in range(0, n, 4):
            m = min(4, n - k)
            g.probs(5 + k, m, 1, q[k:].data_ptr())
            g.sample_fields(5 + k, m, 1, h[k:].data_ptr())
        assert torch.equal(p, q) and torch.equal(f, h)
        assert 0 < float(p.min()) and float(p.max()) < 1
