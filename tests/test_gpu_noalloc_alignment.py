"""nmc_green_noalloc on a caller's packed buffers: fields at odd addresses (they are bytes), and the
constant and the output at addresses that are multiples of 8 but not of 16 (they are doubles). G equals
the call on separately allocated arrays bit for bit, at each size of tile (16 to 112 sites), with a
partly empty last tile, one slice to a block and several, and on the product-by-product route (odd N
and N > 112)."""
import math

import pytest

from paper_2106_00712_gb300.workloads import random_fields

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,L,n_wrap,chains", [(16, 6, 3, 3), (36, 4, 2, 2), (64, 6, 3, 2), (72, 3, 1, 2),
                                               (112, 4, 2, 1), (15, 4, 2, 2), (120, 2, 2, 1)])
@pytest.mark.parametrize("odd", [1, 3])
def test_green_at_any_address(N, L, n_wrap, chains, odd):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2106_00712_gb300 import nmc
    K = torch.diag(torch.full((N - 1,), -1.0, dtype=torch.float64), 1)
    expk = torch.linalg.matrix_exp(-0.1 * (K + K.T)).cuda()     # an open chain of N sites
    fields = torch.from_numpy(random_fields(chains, L, N, seed=N)).cuda()
    lam = math.acosh(math.exp(0.2))
    out = []
    for shift_bytes, shift in ((0, 0), (odd, 1)):
        f = torch.zeros(fields.numel() + 16, dtype=torch.int8, device="cuda")
        f = f[shift_bytes:shift_bytes + fields.numel()].copy_(fields.reshape(-1))
        e = torch.zeros(N * N + 2, dtype=torch.float64, device="cuda")
        e = e[shift:shift + N * N].copy_(expk.reshape(-1))
        G = torch.full((chains * 2 * N * N + 2,), float("nan"), dtype=torch.float64, device="cuda")
        G = G[shift:shift + chains * 2 * N * N]
        assert f.data_ptr() % 2 == shift_bytes % 2 and G.data_ptr() % 16 == 8 * shift
        nmc.nmc_green_noalloc(N, L, n_wrap, lam, e.data_ptr(), f.data_ptr(), chains, G.data_ptr(),
                              torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        out.append(G.cpu())
    assert bool(torch.isfinite(out[0]).all())
    assert torch.equal(out[0], out[1])
