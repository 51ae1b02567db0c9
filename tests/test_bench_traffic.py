"""The benchmark's measured DRAM traffic of the local solves belongs to the source of the local kernels: it is reported
for the present one, whatever else changes in the file, and dropped with a change of those kernels."""

import os
import sys

from conftest import ROOT

sys.path.insert(0, ROOT)
import bench  # noqa: E402


def test_measured_local_traffic_is_reported_for_the_present_kernels():
    assert bench._local_traffic("c2_kappa_rect_p1_h512", "mixed") > 1e9
    assert bench._local_traffic("c2_kappa_rect_p1_h512", "fp64") is None


def test_traffic_is_tied_to_the_local_kernels_alone():
    with open(os.path.join(ROOT, "paper_2203_06327_gb300", "csrc", "kernels.cu")) as f:
        text = f.read()
    sha = bench._local_source_hash(text)
    assert bench._local_source_hash(text.replace("k_spmm", "k_other")) == sha
    assert bench._local_source_hash(text.replace("k_local_sweep_blk_body(BID", "k_local_sweep_body(BID")) != sha
    assert bench._local_source_hash("") is None
