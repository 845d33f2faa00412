"""The blocked stabilized solve at the edges of its blocks and storage: the last size on the
column-by-column kernel (40) and the first beyond (42), remainders of 16 columns, odd sizes (41, 73:
rows not 16-byte aligned), the last two-CTA size (72) and the next (74), the last in shared memory
(112) and the first in global memory (114), and the first with two rows per thread (514, by a
context). e^{-dtau K} of a ring with random hoppings, so any size is allowed, and strong couplings;
the equal-time Green's functions against the FP64 oracle's stabilized product.

Bar: as for the pivoted QR, both sides are backward stable: 1e-10 of max|G|."""
from types import SimpleNamespace

import numpy as np
import pytest

from oracle import dqmc
from paper_2106_00712_gb300.workloads import random_fields

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [40, 41, 42, 47, 49, 63, 72, 73, 74, 95, 97, 112, 113, 114])
def test_any_size_against_oracle(N):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2106_00712_gb300 import nmc
    L, n_wrap, lam = 20, 5, 0.9
    rng = np.random.default_rng(N)
    K = np.zeros((N, N))      # a ring with random hoppings
    for i in range(N):
        K[i, (i + 1) % N] = K[(i + 1) % N, i] = -1.0 - 0.3 * rng.random()
    w, V = np.linalg.eigh(K)
    E = (V * np.exp(-0.2 * w)) @ V.T
    s = random_fields(2, L, N, seed=N)
    dE, dS = torch.from_numpy(E).cuda(), torch.from_numpy(s).cuda()
    dG = torch.full((2, 2, N, N), float("nan"), dtype=torch.float64, device="cuda")
    nmc.nmc_green_noalloc(N, L, n_wrap, lam, dE.data_ptr(), dS.data_ptr(), 2, dG.data_ptr())
    torch.cuda.synchronize()
    G = dG.cpu().numpy()
    P = SimpleNamespace(expK_m=E, lam=lam)
    for c in range(2):
        for a, sigma in enumerate(dqmc.SIGMAS):
            ref = dqmc.green_scratch(P, s[c], sigma, 0, n_wrap)
            assert np.max(np.abs(G[c, a] - ref)) <= 1e-10 * np.max(np.abs(ref))


def test_two_rows_per_thread():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2106_00712_gb300 import nmc
    m = dqmc.Model(257, 1, 1.0, 4.0, 0.4, 0.1, 2, seed=1, lattice="honeycomb")
    s = random_fields(1, m.L_tau, m.N, seed=3)
    with nmc.Context(257, 1, 1.0, 4.0, 0.4, 0.1, 2, seed=1, lattice="honeycomb", n_chains=1,
                     precision=nmc.NMC_FP64) as c:
        c.set_fields(s)
        P = dqmc.Propagators(m)
        for a, sigma in enumerate(dqmc.SIGMAS):
            ref = dqmc.green_scratch(P, s[0], sigma, 0, 2)
            assert np.max(np.abs(c.green(0, a) - ref)) <= 1e-10 * np.max(np.abs(ref))
