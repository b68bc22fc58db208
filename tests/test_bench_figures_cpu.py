"""The ncu summaries that the benchmark reads for its assembly rooflines: every figure is
there and parses, and both are of kernels in the source."""

import os

import pytest

import bench

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROF = {"assembly": {"launches": 1, "ms": 1.0, "work": 1.0e9, "bytes": 0.0},
        "assembly_fast": {"launches": 1, "ms": 1.0, "work": 1.0e9, "bytes": 0.0}}


@pytest.mark.parametrize("cat,flops", [("assembly", "fp64_flops_per_far_point_pair"),
                                       ("assembly_fast", "fp32_flops_per_far_point_pair")])
def test_figures_of_the_assembly_rooflines(cat, flops):
    r = bench.roofline_entry(cat, PROF, 6763.3, 1701.9, {64: 1.25e12, 32: 78.0e12})
    name = r["figures_source"].split("/")[-1]
    for key in (flops, "dram_bytes_per_far_point_pair", "pipe_active_frac"):
        v, src = bench.profile_figure(name, key)
        assert v is not None and v > 0 and src == "profiles/" + name, key
    assert r["pipe_active_frac"] <= 1.0 and r["achieved"] > 0 and r["traffic"] > 0
    kernel = r["kernel"].split()[0]
    text = open(os.path.join(ROOT, "profiles", name)).read()
    source = open(os.path.join(ROOT, "paper_2203_13283_gb300", "csrc", "assemble.cu")).read()
    assert "`" + kernel in text.splitlines()[0] and kernel + "(" in source
