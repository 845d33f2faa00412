"""The tiled convolutions and the weight-gradient product of the convolutional generator at the
edges of their tiles: channel counts off the groups of 8 and past 32, an odd row length (no
paired positions), rows and slices of length 1 and 2 (a halo that wraps onto itself), slices
that straddle a CTA's positions, a batch that takes the wide tile (256 positions per CTA) and
ones that take the narrow one.

Forward: integer noise, weights and biases make every sum an integer far below 2^24 and every
activation an integer below 256 for these weights' sparsity, exact in FP32 and in BF16, so the
logits are equal bit for bit. Gradients: BF16 rounding of a gradient flowing in can differ by one
unit (2^-8 relative) where an FP32 and an FP64 sum straddle a rounding boundary; as in the
oracle comparison of the whole generator, 3e-2 of the largest entry of a layer."""
import numpy as np
import pytest

from oracle import cgen

pytestmark = pytest.mark.gpu

SHAPES = [((40, 8, 8), 32, 40), ((7, 6, 4), 16, 5), ((3, 10, 10), 24, 2), ((5, 1, 2), 3, 3),
          ((4, 2, 2), 40, 2), ((30, 6, 6), 9, 3), ((5, 4, 3), 12, 2), ((1, 4, 4), 8, 2)]


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2106_00712_gb300 import nmc
    return nmc, torch


def _flat(params):
    return np.concatenate([np.concatenate([W.reshape(-1), b]) for W, b in params]).astype(np.float32)


def _gen(nmc, shape, C, n):
    return nmc.ConvGenerator(shape[2], shape[1], shape[0], channels=C, max_batch=n)


@pytest.mark.parametrize("shape,C,n", SHAPES)
def test_forward_bits(env, shape, C, n):
    nmc, torch = env
    rng = np.random.default_rng(C)
    params = []
    for co, ci in ((C, 1), (C, C), (C, C), (1, C)):
        # about two nonzero weights per output channel: activations stay below 2^7
        W = rng.integers(-1, 2, size=(co, ci, 3, 3, 3)) * (rng.random((co, ci, 3, 3, 3)) < 3 / (27 * ci))
        params.append((W.astype(np.float64), rng.integers(-1, 2, size=co).astype(np.float64)))
    z = rng.integers(-1, 2, size=(n,) + shape).astype(np.float64)
    want, acts = cgen.forward(params, z, round_bf16=True)
    assert max(np.abs(a).max() for a in acts) <= 256
    with _gen(nmc, shape, C, n) as g:
        g.set_params(_flat(params))
        dz = torch.from_numpy(z.astype(np.float32)).cuda()
        dl = torch.empty_like(dz)
        g.forward(dz.data_ptr(), n, dl.data_ptr())
        np.testing.assert_array_equal(dl.cpu().numpy().astype(np.float64), want)


@pytest.mark.parametrize("shape,C,n", [(s, c, min(n, 6)) for s, c, n in SHAPES])
def test_gradients(env, shape, C, n):
    nmc, torch = env
    rng = np.random.default_rng(sum(shape) + C)
    params = [(cgen.bf16(W), b.astype(np.float32).astype(np.float64))
              for W, b in cgen.init_params(C, seed=C, scale=0.25)]
    z = rng.normal(size=(n,) + shape)
    s = np.where(rng.random((n,) + shape) < 0.6, 1.0, -1.0)
    want_loss, want = cgen.loss_and_grads(params, z, s, round_bf16=True)
    with _gen(nmc, shape, C, n) as g:
        g.set_params(_flat(params))
        dz = torch.from_numpy(z.astype(np.float32)).cuda()
        df = torch.from_numpy(s.astype(np.int8)).cuda()
        dg = torch.full((g.n_params(),), float("nan"), dtype=torch.float32, device="cuda")
        loss = g.loss_grad(dz.data_ptr(), df.data_ptr(), n, dg.data_ptr())
        got = dg.cpu().numpy().astype(np.float64)
    assert abs(loss - want_loss) <= 1e-4 * want_loss
    o = 0
    for gW, gb in want:
        for ref in (gW.reshape(-1), gb):
            assert np.max(np.abs(got[o:o + ref.size] - ref)) <= 3e-2 * np.max(np.abs(ref)) + 1e-12
            o += ref.size
    assert o == got.size
