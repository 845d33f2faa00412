"""The rounding error of the convolutional generator's weight gradients over large batches, against 64 bits.

Every weight tensor of the first three layers has one 1 per output channel, so that activations are the noise
itself, shifted (positive BF16 values, exact); the last bias saturates the probabilities, and the last weights
have one entry per channel, so that every gradient flowing back is a BF16 value too. What the sums add up is
then known exactly, and is all positive or of one sign per channel, where truncation shows most.

Bar: 2^-22 of the layer's largest entry, somewhat above what FP32 sums of one multiply-add per position reach
here (1.9e-7 at most over batches of this kind, 2e-8 rms); rms 2^-24."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,C,n", [((40, 8, 8), 32, 64), ((30, 6, 6), 16, 37), ((20, 10, 10), 32, 40),
                                       ((60, 4, 4), 8, 60)])
def test_weight_gradients_against_64_bits(shape, C, n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2106_00712_gb300 import nmc
    rng = np.random.default_rng(n)

    def bf16(a):
        return torch.from_numpy(np.asarray(a, dtype=np.float32)).bfloat16().double().numpy()

    params = []
    for co, ci in ((C, 1), (C, C), (C, C), (1, C)):
        W = np.zeros((co, ci, 27))
        if co > 1:
            W[np.arange(co), rng.integers(0, ci, co), rng.integers(0, 27, co)] = 1.0
        else:
            W[0, np.arange(ci), rng.integers(0, 27, ci)] = bf16(rng.normal(size=ci))
        params.append([W.reshape(co, ci, 3, 3, 3), np.zeros(co)])
    params[3][1][:] = 2000.0
    z = bf16(np.abs(rng.normal(size=(n,) + shape)))
    s = np.where(rng.random((n,) + shape) < 0.5, 1, -1).astype(np.int8)

    taps = [(t, y, x) for t in range(3) for y in range(3) for x in range(3)]
    W = [torch.from_numpy(w).cuda() for w, _ in params]

    def shift(a, k, sign):
        return torch.roll(a, tuple(-sign * (d - 1) for d in k), (2, 3, 4))

    acts = [torch.from_numpy(z)[:, None].cuda()]
    for w in W[:3]:
        acts.append(sum(torch.einsum("oc,ncabd->noabd", w[(slice(None), slice(None)) + k], shift(acts[-1], k, 1))
                        for k in taps))
    c = float(bf16(np.float32(1.0) / np.float32(z.size)))
    g = (torch.from_numpy((s < 0).astype(np.float64)).cuda() * c)[:, None]
    want = [None] * 4
    for j in (3, 2, 1, 0):
        want[j] = torch.stack([torch.einsum("noabd,ncabd->oc", g, shift(acts[j], k, 1)) for k in taps], dim=2)
        if j:
            g = sum(torch.einsum("oc,noabd->ncabd", W[j][(slice(None), slice(None)) + k], shift(g, k, -1))
                    for k in taps)
            g = g.float().bfloat16().double()

    with nmc.ConvGenerator(shape[2], shape[1], shape[0], channels=C, max_batch=n) as gen:
        gen.set_params(np.concatenate([np.concatenate([w.reshape(-1), b]) for w, b in params])
                       .astype(np.float32))
        dz = torch.from_numpy(z.astype(np.float32)).cuda()
        df = torch.from_numpy(s).cuda()
        dg = torch.empty(gen.n_params(), device="cuda")
        gen.loss_grad(dz.data_ptr(), df.data_ptr(), n, dg.data_ptr())
    o = 0
    for j in range(4):
        ref = want[j].reshape(-1)
        err = (dg[o:o + ref.numel()].double() - ref).abs() / ref.abs().max()
        assert float(err.max()) <= 2.0 ** -22 and float((err * err).mean().sqrt()) <= 2.0 ** -24, j
        o += ref.numel() + params[j][1].size
