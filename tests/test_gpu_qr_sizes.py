"""The fixed-point column-pivoted QR at the edges of its lane and row blocks (16, 32, 48, 64, 80,
128, 160 and 256 sites, shared and global memory): the equal-time Green's functions of fields whose
UDT stacks are strongly graded (beta = 6, U = 6: singular values over some 20 decades), against the
FP64 oracle's stabilized product with LAPACK's pivoted QR.

Bar: both sides are backward stable per column, and the split-D formula turns such errors into
a few hundred roundings of G times the middle factor's condition (below 1e5 here): 1e-10 of
max|G|, ten times 2^-53 x 1e5."""
import numpy as np
import pytest

from oracle import dqmc
from paper_2106_00712_gb300.workloads import random_fields

pytestmark = pytest.mark.gpu

SIZES = [("square", 2, 1), ("square", 4, 4), ("honeycomb", 3, 3), ("square", 8, 4),
         ("honeycomb", 17, 1), ("square", 8, 6), ("honeycomb", 5, 5), ("square", 8, 8),
         ("honeycomb", 11, 3), ("square", 10, 8), ("honeycomb", 41, 1), ("square", 16, 8),
         ("honeycomb", 13, 5), ("square", 16, 10), ("honeycomb", 9, 9), ("square", 16, 16)]


@pytest.mark.parametrize("lattice,Lx,Ly", SIZES)
def test_graded_stacks_against_oracle(lattice, Lx, Ly):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2106_00712_gb300 import nmc
    beta = 6.0 if Lx * Ly <= 100 else 2.0   # (the oracle's time)
    m = dqmc.Model(Lx, Ly, 1.0, 6.0, beta, 0.1, 5, lattice=lattice)
    P = dqmc.Propagators(m)
    s = random_fields(2, m.L_tau, m.N, seed=m.N)
    dE = torch.from_numpy(nmc.nmc_expk(Lx, Ly, 1.0, -0.1, lattice)).cuda()
    dS = torch.from_numpy(s).cuda()
    dG = torch.full((2, 2, m.N, m.N), float("nan"), dtype=torch.float64, device="cuda")
    nmc.nmc_green_noalloc(m.N, m.L_tau, m.n_wrap, P.lam, dE.data_ptr(), dS.data_ptr(), 2,
                          dG.data_ptr())
    torch.cuda.synchronize()
    G = dG.cpu().numpy()
    for c in range(2):
        for a, sigma in enumerate(dqmc.SIGMAS):
            ref = dqmc.green_scratch(P, s[c], sigma, 0, m.n_wrap)
            assert np.max(np.abs(G[c, a] - ref)) <= 1e-10 * np.max(np.abs(ref))
