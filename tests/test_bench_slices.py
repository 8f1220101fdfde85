"""What bench.py counts per kernel by the number of slices the kernels take (CPU)."""

import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402
from paper_1704_08897_gb300 import synth  # noqa: E402


def test_the_inverse_low_mode_product_is_32_deep():
    p = synth.wobbly(192, 1)  # padded to 256 on every axis
    assert bench.issued_tensor_flop([p], "low_inv", fold=False) == 2 * 21 * 256 * 256 * 32
    # the forward product is the same box turned over
    assert bench.issued_tensor_flop([p], "low_fwd", fold=False) == 2 * 21 * 256 * 256 * 32


@pytest.mark.parametrize("kind,side", [("split", 128), ("fold", 256)])
def test_slicing_writes_what_its_grids_take(kind, side):
    p = synth.wobbly(side, 1)
    n = side * side
    assert bench.algorithmic_cost([p], kind, prec="fp32") == (20 * n, "byte")
    assert bench.algorithmic_cost([p], kind, prec="mixed_bf16") == (20 * n, "byte")           # up to 768^2
    assert bench.algorithmic_cost([p], kind, low=True, prec="mixed_bf16") == (20 * n, "byte")
    big = synth.wobbly(1024 if kind == "fold" else 1400, 1)  # 700-node classes pad to 768: not folded
    assert bench.algorithmic_cost([big], kind, prec="mixed_bf16") == (16 * big.nx * big.ny, "byte")


def test_the_roofline_reads_no_file_that_is_not_there():
    src = open(os.path.join(ROOT, "bench.py")).read()
    for line in src.splitlines():
        if "os.path.join(ROOT, " in line and ".json" in line:
            assert "MEASURED_PEAKS.json" in line, line
