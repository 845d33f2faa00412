"""The kernels that only large lattices reach, on short runs against the FP64 oracle: every field after every
sweep, and G.

* 258 and 312 sites: the stabilization's products in FP32 pairs (stab_pairs above 256 sites, where the FP64
  products no longer go through exact slices), with the tensor cores' wraps and with FP32X2; G differs in its
  bits from the run with FP64 products, so both kernels were at work. These sizes also take the QR with 32
  lanes to a column and the solve in global memory.
* 576 sites in FP64: single flips with G in global memory, where a block's vectors do not fit shared memory.
* 440 sites in FP32X2: single flips of pairs with G in global memory and a delay clamped by their panels.

Bars: G of the stacks 1e-10 of max|G| (a pair product is off by 2^-44 of the sum of its terms, some 3e-14
against G's conditioning of 1e2 here); after the sweeps 1e-8 in pairs, 1e-10 in FP64."""
import numpy as np
import pytest

from oracle.dqmc import Chain, Model, initial_fields

pytestmark = pytest.mark.gpu


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


def _far(a, b):
    return np.max(np.abs(a - b)) / np.max(np.abs(b))


def _follow(c, refs, sweeps, bar):
    for sw in range(sweeps):
        c.sweep(1, measure=0)
        for r in refs:
            r.sweep(False)
        f = c.fields()
        for ch, r in enumerate(refs):
            assert np.array_equal(f[ch], r.s), (sw, ch)
    for ch, r in enumerate(refs):
        for spin in (0, 1):
            assert _far(c.green(ch, spin), r.G[spin]) <= bar


@pytest.mark.parametrize("mode", ["split", "x2"])
@pytest.mark.parametrize("Lx,Ly,lattice", [(43, 3, "honeycomb"), (26, 12, "square")])
def test_stabilization_in_pairs(nmc, mode, Lx, Ly, lattice):
    prec = nmc.NMC_SPLIT_BF16 if mode == "split" else nmc.NMC_FP32X2
    m = Model(Lx, Ly, 1.0, 4.0, 0.4, 0.1, 2, seed=6, lattice=lattice)
    assert m.N > 256
    first = {}
    for pairs in (0, 1):
        with nmc.Context(Lx, Ly, 1.0, 4.0, 0.4, 0.1, 2, seed=6, lattice=lattice, n_chains=1,
                         precision=prec, stab_pairs=pairs, drift_tol=1e-3) as c:
            c.generate()
            ref = Chain(m, initial_fields(m, 0), 0)
            first[pairs] = np.stack([c.green(0, spin) for spin in (0, 1)])
            assert _far(first[pairs], np.stack(ref.G)) <= 1e-10
            if pairs:
                _follow(c, [ref], 2, 1e-8)
    assert not np.array_equal(first[0], first[1])


@pytest.mark.parametrize("mode,Lx,Ly,bar", [("fp64", 24, 24, 1e-10), ("x2", 22, 20, 1e-8)])
def test_single_flips_in_global_memory(nmc, mode, Lx, Ly, bar):
    prec = nmc.NMC_FP64 if mode == "fp64" else nmc.NMC_FP32X2
    m = Model(Lx, Ly, 1.0, 4.0, 0.2, 0.1, 1, seed=8)
    with nmc.Context(Lx, Ly, 1.0, 4.0, 0.2, 0.1, 1, seed=8, n_chains=2, precision=prec,
                     drift_tol=1e-3) as c:
        c.generate()
        _follow(c, [Chain(m, initial_fields(m, 0), 0)], 1, bar)
