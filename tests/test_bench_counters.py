"""The benchmark's counter tables (DRAM traffic, L2 share) hold for the kernel that they were taken on."""

from __future__ import annotations

import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402

SOURCE = open(os.path.join(ROOT, "paper_2505_06711_gb300", "csrc", "density.cu"), encoding="utf-8").read()


def test_key_follows_the_kernel_and_nothing_else():
    sha = bench.kernel_sha("k_density_adj", SOURCE)
    others = SOURCE.replace("k_edges", "k_other").replace("constexpr int kBbarAtoms = 16;", "constexpr int kBbarAtoms = 8;")
    assert others != SOURCE and bench.kernel_sha("k_density_adj", others) == sha
    assert bench.kernel_sha("k_density_adj", SOURCE + "\n// a comment\n") == sha
    changed = SOURCE.replace("const float qt = ck * ph;", "const float qt = ph * ck;")
    assert changed != SOURCE and bench.kernel_sha("k_density_adj", changed) != sha


def test_tables_are_keyed_alike():
    assert set(bench.TRAFFIC) == set(bench.L2_FRAC)
    assert all(region == bench.region_key(region)[0] for region, _ in bench.TRAFFIC)
    assert bench.region_key("mlp_fwd") is None
