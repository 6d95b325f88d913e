"""bench.py's list of a step's kernels follows the library's dispatch."""
import os
import re

import bench

CSRC = os.path.join(bench.ROOT, "paper_2108_07605_gb300", "csrc")


def _source(name):
    return open(os.path.join(CSRC, name)).read()


def test_lines_are_the_library_s():
    m = re.search(r"boundary_warp_nodes\(bool fp64, bool chem64\) \{\s*"
                  r"return fp64 \? (\d+) : \(chem64 \? (\d+) : (\d+)\);", _source("lbm_internal.h"))
    fp64, c64, fp32 = (int(v) for v in m.groups())
    assert bench.WARP_BOUNDARY_NODES == {"fp64": fp64, "fp32c64": c64, "fp32": fp32, "fp16": fp32}
    m = re.search(r"kIfChemThreadNodes = (\d+)LL \* (\d+);", _source("lbm_kernels.cuh"))
    assert bench.IFACE_CHEM_THREADS == int(m.group(1)) * int(m.group(2))


def test_boundary_kernels_by_interface_nodes():
    launch = {"chem_lanes": 1, "collide_split": 1}

    def names(n, precision="fp64"):
        return bench.step_kernels(launch, n, precision)[0]

    assert names(0) == ["k_moments"]
    assert names(4096) == ["k_bnode_warp", "k_moments"]
    assert names(4097) == ["k_bnode", "k_chem", "k_moments"]
    assert names(4097, "fp32") == ["k_bnode_warp", "k_moments"]
    assert names(2049, "fp32c64") == ["k_bnode", "k_chem", "k_moments"]
    assert names(19455) == ["k_bnode", "k_chem", "k_moments"]
    assert names(19456) == ["k_bnode", "k_iface_chem", "k_moments"]
    assert bench.launches_per_step(launch, 20000, "fp64") == 5
