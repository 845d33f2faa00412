"""Delays on both sides of the line between folding one flip at a time and deciding blocks of sites:
every field after every sweep equals the FP64 oracle's, and G at the end. Sizes where the delay alone
sets the line (16, 36 sites), where delay x sites does (64, 100) and where shared memory does (100 and
120 sites, one spin, in FP64), lattices smaller than the default delay (2 and 8 sites), and blocks cut
short of 16 sites (9 and 13). FP32X2 on both sides of its own lines: 24 and 26 sites, 64 and 66, both spins
and one (100), and G that fits a block's shared memory or not (100, 104, 112).

Bar on G: 1e-10 of max|G| in FP64, 1e-8 in FP32 pairs (the bars of the blocks' own tests: FP32 pairs
carry 2^-46 of a wrap's terms over five slices, amplified by the propagators by a few 1e2)."""
import numpy as np
import pytest

from oracle.dqmc import Chain, Model, initial_fields

pytestmark = pytest.mark.gpu

CASES = [("fp64", 4, 4, k, 0) for k in (1, 6, 7, 9)] + [("fp64", 6, 6, k, 0) for k in (6, 7)] + \
        [("fp64", 8, 8, k, 0) for k in (4, 5, 13)] + [("fp64", 10, 10, 3, 1), ("fp64", 10, 10, 4, 1)] + \
        [("fp64", 12, 10, 2, 1)] + \
        [("split", 4, 4, k, 0) for k in (1, 8, 9)] + [("split", 8, 8, k, 0) for k in (6, 7, 13)] + \
        [("split", 10, 10, k, 0) for k in (4, 5)] + [("split", 12, 10, 3, 1)] + \
        [("x2", 6, 6, 8, 0), ("x2", 6, 6, 9, 0), ("x2", 8, 8, 6, 1), ("x2", 8, 8, 7, 1)] + \
        [("x2", 6, 4, 16, 0), ("x2", 26, 1, 16, 0), ("x2", 16, 4, 16, 0), ("x2", 66, 1, 12, 0)] + \
        [("x2", 10, 10, 16, ph) for ph in (0, 1)] + [("x2", 26, 4, 16, 0), ("x2", 28, 4, 16, 0)] + \
        [(m, Lx, Ly, 16, 0) for m in ("fp64", "split", "x2") for Lx, Ly in ((2, 1), (4, 2))]


@pytest.fixture(scope="module")
def nmc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2106_00712_gb300 import nmc as m
    m.load()
    return m


def _precision(nmc, mode):
    return {"fp64": nmc.NMC_FP64, "split": nmc.NMC_SPLIT_BF16, "x2": nmc.NMC_FP32X2}[mode]


@pytest.mark.parametrize("mode,Lx,Ly,delay,ph", CASES)
def test_fields_and_green_follow_the_oracle(nmc, mode, Lx, Ly, delay, ph):
    m = Model(Lx, Ly, 1.0, 4.0, 0.5, 0.1, 5, seed=7)
    with nmc.Context(Lx, Ly, 1.0, 4.0, 0.5, 0.1, 5, seed=7, n_chains=2, delay_k=delay,
                     precision=_precision(nmc, mode), ph_symmetric=ph, drift_tol=1e-3) as c:
        c.generate()
        refs = [Chain(m, initial_fields(m, ch), ch) for ch in range(2)]
        for sw in range(4):
            c.sweep(1, measure=0)
            for r in refs:
                r.sweep(False)
            f = c.fields()
            for ch in range(2):
                assert np.array_equal(f[ch], refs[ch].s), (sw, ch)
        for ch in range(2):
            for spin in (0, 1):
                ref = refs[ch].G[spin]
                assert np.max(np.abs(c.green(ch, spin) - ref)) <= \
                    (1e-10 if mode == "fp64" else 1e-8) * np.max(np.abs(ref))


@pytest.mark.parametrize("mode", ["fp64", "split"])
def test_small_delays_stay_fast(nmc, mode):
    """The flips' device time at delay 1 against delay 16, 256 chains of 64 sites: 2.3 times as long one
    flip at a time, 5.7 (FP64) and 6.1 (pairs) in blocks of one site. The bar lies between."""
    t = {}
    for delay in (1, 16):
        with nmc.Context(8, 8, 1.0, 4.0, 1.0, 0.1, 5, seed=1, n_chains=256, delay_k=delay,
                         precision=_precision(nmc, mode), drift_tol=1.0) as c:
            c.generate()
            c.sweep(2, measure=0)
            c.profile(1)
            c.kernel_stats(reset=True)
            c.sweep(4, measure=0)
            t[delay] = c.kernel_stats()["flip"][2]
    assert t[1] < 4 * t[16], t
