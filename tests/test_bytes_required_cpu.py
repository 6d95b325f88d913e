"""Boundary arrays in lbm_bytes_required: the reconstructed populations take the
lattice type (FP64, or FP32 for FP32 and FP16 storage)."""
import pytest

from lbm_workloads import fields
from lbm_workloads.mechanism import h2_air_synthetic

from helpers import boundary_spec


@pytest.mark.parametrize("precision,size", [("fp64", 8), ("fp32", 4), ("fp16", 4)])
def test_boundary_arrays(precision, size):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2108_07605_gb300 import lbm
    mech = h2_air_synthetic()
    w = fields.channel_2d(nx=50, ny=20)

    def need(**bc):
        cfg, _ = lbm.make_config(mech, lattice="D2Q9", shape=w["shape"], dx=w["dx"],
                                 precision=precision, use_torch_allocator=False, **bc)
        return lbm.lbm_bytes_required(cfg)

    def a256(n):
        return (n + 255) // 256 * 256

    n, n_if, lq = 50 * 20, 2 * 50 + 2 * 18, 10 * 9
    want = a256(4 * n) + 3 * a256(4 * n_if) + 4 * a256(8 * n_if) + a256(lq * n_if * size)
    assert need(**boundary_spec(w)) - need() == want
