"""Every gradient of the convolutional generator, exactly: noise and weights are small integers, hidden
activations with them, and the last bias makes every logit so large that a Bernoulli probability is 1 to the
last bit. The gradient flowing in is then 0 or c = 1 / (samples x positions), a power of two here, every
gradient that flows on c times an integer of at most 8 bits (exact in BF16), and every weight's and bias's
gradient c times an integer below 2^24: no sum rounds, whatever its order, and a lost or doubled position
shows. Shapes on both sides of the kernels' rules, tiles of 8 slices and fewer, short axes and rows of
length 1 (whose halo wraps onto itself), rows of odd length, channels off the groups of 8."""
import numpy as np
import pytest

from oracle import cgen

pytestmark = pytest.mark.gpu

SHAPES = [((32, 8, 8), 32, 16), ((32, 16, 16), 32, 2), ((1, 4, 4), 8, 1024), ((2, 16, 2), 9, 64),
          ((64, 2, 16), 24, 2), ((8, 1, 8), 12, 64), ((4, 2, 2), 32, 256), ((16, 4, 8), 16, 32),
          ((16, 4, 1), 16, 128), ((8, 4, 2), 40, 64), ((4, 4, 4), 7, 16)]


@pytest.mark.parametrize("shape,C,n", SHAPES)
def test_integer_gradients(shape, C, n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2106_00712_gb300 import nmc
    rng = np.random.default_rng(sum(shape) + C + n)
    params = []
    for co, ci in ((C, 1), (C, C), (C, C), (1, C)):
        # about two nonzero weights per output channel: activations and gradients stay small
        W = rng.integers(-1, 2, size=(co, ci, 3, 3, 3)) * (rng.random((co, ci, 3, 3, 3)) < 3 / (27 * ci))
        params.append((W.astype(np.float64), rng.integers(-1, 2, size=co).astype(np.float64)))
    params[3][1][:] = 2000.0
    params[3][0][0, rng.integers(0, C, 6), 1, 1, 1] = 1.0      # (some gradient flows)
    z = rng.integers(-1, 2, size=(n,) + shape).astype(np.float64)
    s = np.where(rng.random((n,) + shape) < 0.8, 1.0, -1.0)
    unit = 1.0 / z.size
    assert z.size & (z.size - 1) == 0
    logits, acts = cgen.forward(params, z, round_bf16=True)
    assert logits.min() > 200 and max(np.abs(a).max() for a in acts) <= 256
    want_loss, want = cgen.loss_and_grads(params, z, s, round_bf16=True)
    flat = np.concatenate([np.concatenate([W.reshape(-1), b]) for W, b in want])
    assert np.array_equal(flat / unit, np.rint(flat / unit)) and np.abs(flat).max() < 2 ** 24 * unit
    with nmc.ConvGenerator(shape[2], shape[1], shape[0], channels=C, max_batch=n) as g:
        g.set_params(np.concatenate([np.concatenate([W.reshape(-1), b]) for W, b in params]).astype(np.float32))
        dz = torch.from_numpy(z.astype(np.float32)).cuda()
        df = torch.from_numpy(s.astype(np.int8)).cuda()
        dg = torch.full((g.n_params(),), float("nan"), dtype=torch.float32, device="cuda")
        loss = g.loss_grad(dz.data_ptr(), df.data_ptr(), n, dg.data_ptr())
        np.testing.assert_array_equal(dg.cpu().numpy().astype(np.float64), flat)
    assert abs(loss - want_loss) <= 1e-4 * want_loss
