"""A convolutional generator whose largest call is below the rules of the tiled kernels (125,000 outputs of a
middle layer, 2600 positions) holds none of their memory: the weights' copies in their layouts and 152 sets
of partial gradients, 17 MB at 32 channels. One position more than the rule holds it. Both train."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_small_generator_holds_no_tiled_workspace():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2106_00712_gb300 import nmc
    f = torch.ones((2, 82, 4, 4), dtype=torch.int8, device="cuda")
    with nmc.ConvGenerator(4, 4, 82, channels=32, max_batch=2) as g:   # (kernels loaded, pools grown)
        g.train_step(f.data_ptr(), 2, 0, 1e-4)
    held = {}
    for L, n in ((81, 2), (82, 2)):   # 2592 and 2624 positions
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        with nmc.ConvGenerator(4, 4, L, channels=32, max_batch=n) as g:
            held[L] = free - torch.cuda.mem_get_info()[0]
            th = g.get_params()
            loss = g.train_step(f.data_ptr(), n, 0, 1e-4)
            assert np.isfinite(loss) and not np.array_equal(th, g.get_params())
    assert held[81] < 8 << 20 < held[82], held
