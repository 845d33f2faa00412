"""Generator outputs for many samples at once (lanes on samples) against the same samples in
calls too small for that path: equal bit for bit (the same multiply-adds in the same order), at
batch sizes at the edges of the groups (32 and 128 samples), past one internal chunk (256) and
odd ones, for the paper's network and for one whose axes are no multiple of the output tile (4).
The small calls themselves are held to the oracle elsewhere (test_gpu_nimc.py)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ARCHS = [("honeycomb", 6, 6, 6.0, dict()),
         ("square", 6, 2, 0.9, dict(z=(3, 2, 1), c1=5, k1=(3, 3, 2), k2=(5, 3, 1))),
         ("square", 2, 1, 0.6, dict(z=(1, 1, 1), c1=1, k1=(6, 2, 1), k2=(1, 1, 1)))]


@pytest.mark.parametrize("lattice,Lx,Ly,beta,arch", ARCHS)
@pytest.mark.parametrize("n", [32, 37, 95, 96, 130, 300])
def test_many_samples_equal_few(lattice, Lx, Ly, beta, arch, n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2106_00712_gb300 import nmc
    with nmc.Generator(Lx, Ly, 1.0, 4.0, beta, 0.1, 3, arch=nmc.gen_arch(**arch), seed=9,
                       max_batch=4, lattice=lattice) as g:
        rng = np.random.default_rng(n)
        g.set_params([(W, rng.uniform(-0.3, 0.3, b.shape).astype(np.float32))
                      for W, b in g.params()])
        p = torch.full((n, g.L_tau, g.A, g.B), float("nan"), device="cuda")
        f = torch.zeros((n, g.L_tau, g.N), dtype=torch.int8, device="cuda")
        g.probs(5, n, 1, p.data_ptr())
        g.sample_fields(5, n, 1, f.data_ptr())
        q, h = torch.empty_like(p), torch.empty_like(f)
        for k in range(0, n, 16):
            m = min(16, n - k)
            g.probs(5 + k, m, 1, q[k:].data_ptr())
            g.sample_fields(5 + k, m, 1, h[k:].data_ptr())
        assert torch.equal(p, q) and torch.equal(f, h)
        assert 0 < float(p.min()) and float(p.max()) < 1
