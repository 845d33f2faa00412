"""FP64 products as exact tensor-core slices: the equal-time Green's functions of
nmc_green_noalloc, whose every product (plain, transposed on either side, with row and column
scales, with an added matrix) goes through them for N > 16, against the FP64 oracle at lattice
sizes at the edges of the kernel's blocks (16), stages (64 terms at once, 48 at a time above) and
range (256), and odd ones between.

Bar: the oracle and the kernel both evaluate the split-D formula in FP64 or better, with errors
of a few hundred roundings times the middle factor's condition (below 1e4 at beta = 1):
1e-12 relative to max|G| = O(1) is 2^-53 x 1e4, the bar 1e-11 ten times that."""
import numpy as np
import pytest

from oracle import dqmc
from paper_2106_00712_gb300.workloads import random_fields

pytestmark = pytest.mark.gpu

SIZES = [("square", 2, 1), ("square", 4, 4), ("honeycomb", 3, 3), ("square", 8, 4),
         ("square", 8, 6), ("honeycomb", 5, 5), ("square", 8, 8), ("honeycomb", 11, 3),
         ("square", 10, 8), ("square", 12, 8), ("honeycomb", 7, 7), ("honeycomb", 13, 5),
         ("square", 16, 16)]


@pytest.mark.parametrize("lattice,Lx,Ly", SIZES)
@pytest.mark.parametrize("chains", [1, 3])
def test_green_against_oracle(lattice, Lx, Ly, chains):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2106_00712_gb300 import nmc
    m = dqmc.Model(Lx, Ly, 1.0, 4.0, 1.0, 0.1, 5, lattice=lattice)
    P = dqmc.Propagators(m)
    s = random_fields(chains, m.L_tau, m.N, seed=m.N + chains)
    dE = torch.from_numpy(nmc.nmc_expk(Lx, Ly, 1.0, -0.1, lattice)).cuda()
    dS = torch.from_numpy(s).cuda()
    dG = torch.full((chains, 2, m.N, m.N), float("nan"), dtype=torch.float64, device="cuda")
    nmc.nmc_green_noalloc(m.N, m.L_tau, m.n_wrap, P.lam, dE.data_ptr(), dS.data_ptr(), chains,
                          dG.data_ptr())
    torch.cuda.synchronize()
    G = dG.cpu().numpy()
    for c in range(chains):
        for a, sigma in enumerate(dqmc.SIGMAS):
            ref = dqmc.green_scratch(P, s[c], sigma, 0, m.n_wrap)
            assert np.max(np.abs(G[c, a] - ref)) <= 1e-11 * np.max(np.abs(ref))
