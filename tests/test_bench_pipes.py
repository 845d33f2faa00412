"""The benchmark line's classes that do FP64-class work on other pipes say so: FP64 products by exact FP16
digits carry their fraction of the tensor peak, QR and solve are marked as equivalents, and the flips name
the kernel that the path runs (no GPU)."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

import bench  # noqa: E402

PEAKS = {"fp64": 1.2, "fp32": 75.0, "bf16": 1900.0}
STATS = {k: (1, 1, 1.0) for k in ("gemm", "flip", "qrp", "solve")}


@pytest.mark.parametrize("base,tc", [("fp64", False), ("fp32x2", True), ("fp32x2", False)])
def test_equivalents_are_marked(base, tc):
    rl = bench.class_rooflines(STATS, base, 2, 0.5, PEAKS, tc)
    a = 28 * 2.0 * bench.WL.N ** 3 * 2 * bench.WL.n_chains / 1e-3 / 1e12
    assert rl["gemm"]["frac_of_pipe"] == pytest.approx(a / PEAKS["bf16"])
    for cls in ("gemm", "qrp", "solve"):
        assert "FP64" in rl[cls]["equivalent"] and rl[cls]["pipe"]
    assert "equivalent" not in rl["flip"]
    if base == "fp32x2":
        assert ("k_flip_block" in rl["flip"]["kernel"]) == tc


def test_simt_products_are_not():
    rl = bench.class_rooflines(STATS, "fp32", 2, 0.5, PEAKS, False)
    assert "equivalent" not in rl["gemm"] and rl["gemm"]["bound"] == "alu"
