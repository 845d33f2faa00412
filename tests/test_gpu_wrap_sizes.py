"""The whole-matrix products (wraps, block products, half steps of the measurement) at the edges of
their 16-site tiles and of the tiles per warp (16, 32, 48, 64, 80, 96, 112 sites; at 114 the
product-by-product kernels take over), carries beyond 64 terms, in FP64 and in FP32 pairs on the tensor
cores, one spin and both: fields after every sweep, G and the measured energies against the FP64 oracle.

Bars: 1e-10 of max|G| in FP64 and 1e-8 with FP32 pairs (2^-46 per product and slice, grown by the
propagators' condition over n_wrap = 5 slices), 1e-9 on observables, as everywhere."""
import numpy as np
import pytest

from oracle.dqmc import Chain, Model, initial_fields

pytestmark = pytest.mark.gpu

SIZES = [("square", 2, 2), ("square", 4, 4), ("honeycomb", 3, 3), ("square", 8, 4),
         ("honeycomb", 17, 1), ("square", 8, 6), ("honeycomb", 5, 5), ("honeycomb", 11, 3),
         ("square", 10, 8), ("honeycomb", 41, 1), ("square", 12, 8), ("honeycomb", 7, 7),
         ("honeycomb", 8, 7), ("honeycomb", 19, 3)]


@pytest.mark.parametrize("mode", ["fp64", "split"])
@pytest.mark.parametrize("lattice,Lx,Ly", SIZES)
def test_sweeps_follow_the_oracle(lattice, Lx, Ly, mode):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2106_00712_gb300 import nmc
    prec = nmc.NMC_FP64 if mode == "fp64" else nmc.NMC_SPLIT_BF16
    ph = int(mode == "split" and Lx % 2 == 1)
    m = Model(Lx, Ly, 1.0, 4.0, 1.0, 0.1, 5, seed=Lx + Ly, lattice=lattice)
    with nmc.Context(Lx, Ly, 1.0, 4.0, 1.0, 0.1, 5, seed=Lx + Ly, lattice=lattice, n_chains=2,
                     precision=prec, ph_symmetric=ph, drift_tol=1e-3) as c:
        c.generate()
        refs = [Chain(m, initial_fields(m, ch), ch) for ch in range(2)]
        for sw in range(2):
            c.sweep(1, measure=1)
            for r in refs:
                r.sweep(True)
            f = c.fields()
            for ch in range(2):
                assert np.array_equal(f[ch], refs[ch].s), (sw, ch)
        _, per = c.measure(per_chain=True)
        for ch in range(2):
            want = refs[ch].means()
            for k in ("energy", "ekin", "double_occ", "s_pipi"):
                assert abs(getattr(per[ch], k).mean - want[k]) < 1e-9, (k, ch)
            for spin in (0, 1):
                ref = refs[ch].G[spin]
                assert np.max(np.abs(c.green(ch, spin) - ref)) <= \
                    (1e-10 if mode == "fp64" else 1e-8) * np.max(np.abs(ref))
