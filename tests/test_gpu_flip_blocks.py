"""The block-of-sites flip kernel at the edges of its blocks and tiles: the last block full, one
pair of sites or in between (N = 16, 18, 30, 36, 50, 64), G in shared and in global memory (N = 144,
162: both spins do not fit), one flip per block (delay 1), blocks cut short (3), full ones (16) and a
delay above a block (40), both spins or one, and forced decisions. Every field after every sweep
equals the FP64 oracle's, so do the counts, and G is compared at the end.

Bar on G: 1e-10 of max|G| in FP64 (the FP64 path's bar everywhere); with FP32 pairs a wrap carries
2^-46 of its terms and a slice's flips N terms of 2^-47 each, over n_wrap = 5 slices between
rebuilds amplified by the propagators (a few 1e2): 1e-8."""
import numpy as np
import pytest

from oracle import dqmc
from oracle.dqmc import Chain, Model, initial_fields

pytestmark = pytest.mark.gpu

SIZES = [("square", 4, 4), ("honeycomb", 3, 3), ("honeycomb", 5, 3), ("square", 6, 6),
         ("honeycomb", 5, 5), ("square", 8, 8), ("square", 12, 12), ("honeycomb", 9, 9)]
DELAYS = {0: 16, 1: 3, 2: 1, 3: 40}


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


@pytest.mark.parametrize("mode", ["fp64", "split", "x2"])
@pytest.mark.parametrize("k,size", [(k, s) for k, s in enumerate(SIZES)])
def test_fields_and_green_follow_the_oracle(nmc, mode, k, size):
    lattice, Lx, Ly = size
    prec = {"fp64": nmc.NMC_FP64, "split": nmc.NMC_SPLIT_BF16, "x2": nmc.NMC_FP32X2}[mode]
    ph = int(k % 2 == 1 and mode != "fp64")
    m = Model(Lx, Ly, 1.0, 4.0, 1.0, 0.1, 5, seed=3 + k, lattice=lattice)
    with nmc.Context(Lx, Ly, 1.0, 4.0, 1.0, 0.1, 5, seed=3 + k, lattice=lattice, n_chains=2,
                     delay_k=DELAYS[k % 4], precision=prec, ph_symmetric=ph, drift_tol=1e-3) as c:
        c.generate()
        refs = [Chain(m, initial_fields(m, ch), ch) for ch in range(2)]
        for sw in range(3):
            c.sweep(1, measure=1)
            for r in refs:
                r.sweep(True)
            f = c.fields()
            for ch in range(2):
                assert np.array_equal(f[ch], refs[ch].s), (sw, ch)
        _, per = c.measure(per_chain=True)
        for ch in range(2):
            assert abs(per[ch].accept - refs[ch].means()["accept"]) < 1e-15
            for spin in (0, 1):
                ref = refs[ch].G[spin]
                assert np.max(np.abs(c.green(ch, spin) - ref)) <= \
                    (1e-10 if mode == "fp64" else 1e-8) * np.max(np.abs(ref))


@pytest.mark.parametrize("mode", ["fp64", "split", "x2"])
def test_forced_decisions(nmc, mode):
    """Decisions of another trajectory: the fields follow them, the disagreements are counted."""
    prec = {"fp64": nmc.NMC_FP64, "split": nmc.NMC_SPLIT_BF16, "x2": nmc.NMC_FP32X2}[mode]
    m = Model(5, 5, 1.0, 4.0, 1.0, 0.1, 5, seed=9, lattice="honeycomb")
    accept = (np.random.default_rng(5).random((2, m.L_tau, m.N)) < 0.3).astype(np.uint8)
    got = []
    for delay in (1, 16):
        with nmc.Context(5, 5, 1.0, 4.0, 1.0, 0.1, 5, seed=9, lattice="honeycomb", n_chains=2,
                         delay_k=delay, precision=prec, drift_tol=1.0) as c:
            c.generate()
            before = c.fields()
            c.sweep_replay(accept, measure=1)
            assert np.array_equal(c.fields(), np.where(accept, -before, before))
            obs, per = c.measure(per_chain=True)
            got.append(obs.n_disagree)
            for ch in range(2):
                assert abs(per[ch].accept - accept[ch].mean()) < 1e-15
    assert got[0] == got[1] > 0


@pytest.mark.parametrize("mode", ["fp64", "split"])
@pytest.mark.parametrize("lattice,Lx,Ly", [("honeycomb", 7, 7), ("square", 12, 12), ("honeycomb", 9, 9)])
def test_clusters_change_no_bit(nmc, mode, lattice, Lx, Ly):
    """Few chains take several CTAs each, many one: 4 (2 chains), 2 (60) and 1 (160), with 16-row
    tiles that do not divide evenly (N = 98, 144, 162): the same bits."""
    prec = nmc.NMC_FP64 if mode == "fp64" else nmc.NMC_SPLIT_BF16
    got = []
    for chains in (2, 60, 160):
        with nmc.Context(Lx, Ly, 1.0, 4.0, 0.5, 0.1, 5, seed=2, lattice=lattice, n_chains=chains,
                         precision=prec, drift_tol=1e-3) as c:
            c.generate()
            c.sweep(1, measure=1)
            got.append((c.fields()[:2].copy(), [c.green(ch, sp).copy() for ch in (0, 1) for sp in (0, 1)]))
    for f, G in got[1:]:
        assert np.array_equal(f, got[0][0])
        assert all(np.array_equal(a, b) for a, b in zip(G, got[0][1]))
