"""The bounds-checked build on the kernels that its small cases do not reach: the tensor-core products above
112 sites, clusters of CTAs, blocks folded in FP32 pairs, single flips, G in global memory, and the
stabilization's products in FP32 pairs. Every key index is checked, no check fails, and the fields equal the
regular build's. It runs in a child process that loads the debug library."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
import sys
import numpy as np
sys.path.insert(0, ROOT)
from paper_2106_00712_gb300 import nmc
lib = nmc.load()
assert lib.nmc_debug_build() == DEBUG
out = []
for Lx, Ly, prec, chains, delay, ph, pairs in (
        (12, 10, nmc.NMC_SPLIT_BF16, 2, 16, 0, 0), (12, 12, nmc.NMC_SPLIT_BF16, 160, 16, 1, 0),
        (18, 18, nmc.NMC_FP64, 1, 16, 0, 0), (12, 12, nmc.NMC_FP64, 3, 7, 0, 0),
        (10, 10, nmc.NMC_FP32X2, 2, 16, 0, 0), (12, 10, nmc.NMC_FP32X2, 2, 16, 0, 0),
        (8, 8, nmc.NMC_FP64, 2, 3, 0, 0), (8, 8, nmc.NMC_SPLIT_BF16, 2, 5, 1, 0),
        (26, 10, nmc.NMC_SPLIT_BF16, 1, 16, 0, 1)):
    with nmc.Context(Lx, Ly, 1.0, 4.0, 0.4, 0.1, 2, seed=5, n_chains=chains, delay_k=delay, precision=prec,
                     ph_symmetric=ph, stab_pairs=pairs, drift_tol=1e-3) as c:
        c.generate()
        c.sweep(2, measure=1)
        out.append(c.fields().reshape(-1))
if DEBUG:
    assert lib.nmc_debug_checks() == 0, lib.nmc_debug_checks()
np.save(OUT, np.concatenate(out))
print("ran, no check failed")
'''


def test_bounds_checked_build_on_large_lattices(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import numpy as np
    from paper_2106_00712_gb300 import build_lib
    got = []
    for debug in (0, 1):
        out = str(tmp_path / ("fields%d.npy" % debug))
        env = dict(os.environ, NMC_LIB_PATH=build_lib.build(debug=bool(debug)))
        code = "ROOT, OUT, DEBUG = %r, %r, %d\n" % (ROOT, out, debug) + CHILD
        r = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True,
                           timeout=600, cwd=ROOT)
        assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
        assert "no check failed" in r.stdout
        got.append(np.load(out))
    assert np.array_equal(got[0], got[1])
