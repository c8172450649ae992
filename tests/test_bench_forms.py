"""bench.py's account of the tensor-core form: the sources whose change makes a capture stale,
and the slice products that a convolution issues."""
import os
import shutil
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


@pytest.mark.parametrize("name", ["kernels.cu", "digits.cuh", "kernels.hpp", "dag_sync.cuh", "mma_kernels.cu",
                                  "slices.cuh"])
def test_kernel_source_hash_covers_every_kernel_source(tmp_path, monkeypatch, name):
    csrc = tmp_path / "paper_2101_10881_gb300" / "csrc"
    shutil.copytree(os.path.join(ROOT, "paper_2101_10881_gb300", "csrc"), csrc)
    whole = bench.kernel_source_hash()
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.kernel_source_hash() == whole
    with open(csrc / name, "a") as f:
        f.write("\nconstexpr int kUnusedForTheTest = 1;\n")
    assert bench.kernel_source_hash() != whole


@pytest.mark.parametrize("k,d,slices", [(4, 8, 30), (5, 152, 38), (8, 95, 56), (10, 152, 58)])
def test_slice_products(k, d, slices):
    digits = (53 * k + 28 + 27) // 28 + 1
    blocks = (slices + 15) // 16
    tiles = [list(range(max(0, hi - 7), hi + 1)) for hi in range(d, -1, -8)]
    assert sorted(j for t in tiles for j in t) == list(range(d + 1))
    macs = sum((t[-1] + 1) * 16 * 16 * 8 for t in tiles) * sum(range(1, blocks + 1))
    assert bench.slice_product_flops(3, d, k, digits) == 3 * 2 * macs
