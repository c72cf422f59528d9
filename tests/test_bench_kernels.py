"""Host logic of the benchmark (no GPU): the kernel it names beside a step's time is the one the
library's rules take."""
import os
import re
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402

CSRC = os.path.join(ROOT, "paper_2212_10680_gb300", "csrc")


def _constant(header, name):
    with open(os.path.join(CSRC, header)) as f:
        return eval(re.search(rf"constexpr \w+ {name} = ([^;]+);", f.read()).group(1))


def test_the_bounds_are_the_librarys():
    assert bench.MARCH_NODES == _constant("fmlbm_march.cuh", "kMarchNodes")
    assert bench.MARCH_COLS == _constant("fmlbm_march.cuh", "kMarchCols")
    assert bench.PACK_NODES == _constant("fmlbm_pack.cuh", "kPackNodes")


def test_step_kernel_follows_the_rules():
    k = bench.step_kernel
    assert k("plain", "fp32", 2, 1024, 1024) == "march_step"
    assert k("plain", "bf16dev", 3, 724, 725) == "march_step"
    # mostly empty last strips: 64 columns take three of 28, 3 columns one
    assert k("plain", "fp32", 2, 64, 9000) == "pack_step" and k("plain", "fp32", 3, 64, 9000) == "fused_step"
    assert k("plain", "fp32", 2, 3, 65536) == "pack_step"
    assert k("plain", "fp32", 2, 23, 23000) == "march_step"
    assert k("plain", "fp32", 2, 255, 256) == "fused_step" and k("plain", "fp32", 2, 256, 256) == "pack_step"
    assert k("plain", "fp32", 1, 1024, 1024) == k("plain", "fp32", 4, 1024, 1024) == "fused_step"
    assert k("plain", "fp32", 2, 1024, 1024, standard=True) == k("plain", "fp64", 2, 64, 64, standard=True) == "fused_step"
    assert k("plain", "fp32", 2, 1024, 1024, 16) == "fused_step"
    assert k("plain", "fp64", 2, 64, 64) == k("plain", "bf16dev_lnf64", 3, 4096, 4096) == "collide_fields"
    assert k("tma_tile", "fp32", 2, 1024, 1024) == "fused_step_tma"
