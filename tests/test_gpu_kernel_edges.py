"""The kernels' dispatch edges against the CPU oracle: the boundary kernel with
a warp or a thread per interface node (the line lies at 6144 of them), the lane
groups' default at its grid limits, reaction rates inside and outside the range
of their fixed-point arguments (128 K <= T < 16384 K, coefficients that fit),
and the FP16 codec set up on the device.

FP64: 1e-10 relative per lattice, the bound of the other parity tests.  FP32:
the field tolerances stated for that storage.  FP16 initial populations: an
offset h = (f - o) / s keeps 11 bits of f - o, whose size the tables bound by
the lattice's largest deviation from the mean state's equilibrium, and FP32
arithmetic rounds f itself: 2^-11 and 2^-22 of them, doubled for the decode."""
import dataclasses

import numpy as np
import pytest

from lbm_workloads import fields
from lbm_workloads.mechanism import h2_air_synthetic

from helpers import make_gpu, make_oracle, max_rel_err_per_lattice, oracle_populations

pytestmark = pytest.mark.gpu
RTOL_FP64 = 1e-10


@pytest.fixture(scope="module")
def mech():
    return h2_air_synthetic()


def _parity(mech, w, nsteps, noise=0.0):
    if noise:
        rng = fields.philox(3)
        w["u"] = w["u"] + noise * rng.uniform(-1.0, 1.0, size=w["u"].shape)
        if w["lattice"] == "D2Q9":
            w["u"][2] = 0.0
    o, g = make_oracle(mech, w), make_gpu(mech, w)
    o.step(nsteps)
    g.step(nsteps)
    mask = None if w.get("solid") is None else ~np.asarray(w["solid"]).reshape(-1)
    err = max_rel_err_per_lattice(g.populations(), oracle_populations(o), mask)
    g.close()
    assert np.all(err < RTOL_FP64), err


# 2 nx + 2 (ny - 2) interface nodes: 6142, 6144, 6146
@pytest.mark.parametrize("nx", [3065, 3066, 3067])
def test_boundary_kernels_either_side_of_the_line_d2q9(mech, nx):
    _parity(mech, fields.channel_2d(nx=nx, ny=8, dx=25e-6), 3, noise=0.05)


@pytest.mark.parametrize("offgrid", [False, True])
@pytest.mark.parametrize("nx", [44, 61])
def test_thread_boundary_kernel_d3q27(mech, nx, offgrid):
    """More than 6144 interface nodes; ragged last blocks, warps with nodes of
    several wall rows, inlet and outlet."""
    w = fields.microtube(nx=nx, ny=40, nz=40, radius=19.0, dx=25e-6, offgrid=offgrid)
    _parity(mech, w, 2, noise=0.05)


@pytest.mark.parametrize("make,lanes", [
    (lambda m: fields.flame_1d(nx=304, ny=4, nz=4, x_ign=80), 4),      # 4864 nodes
    (lambda m: fields.flame_1d(nx=305, ny=4, nz=4, x_ign=80), 1),
    (lambda m: fields.perturbed_box((32, 24, 19), "D3Q27", mech=m), 4),   # 14592 nodes
    (lambda m: fields.perturbed_box((29, 24, 21), "D3Q27", mech=m), 1),
])
@pytest.mark.parametrize("precision", ["fp32", "fp32c64", "fp16"])
def test_default_lanes_at_the_limits(mech, make, lanes, precision):
    w = make(mech)
    g = make_gpu(mech, w, precision=precision)
    assert g.launch()["chem_lanes"] == lanes
    o = make_oracle(mech, w)
    o.step(4)
    g.step(4)
    mo, mg = o.moments(), g.moments()
    g.close()
    M = mech.n_species
    loose = 10.0 if precision == "fp16" else 1.0
    assert np.abs(mg["Y"] - mo["Y"].reshape(M, -1)).max() <= 2e-5 * loose
    assert np.abs(mg["T"] - mo["T"].ravel()).max() <= 0.05 * loose
    assert (np.abs(mg["rho"] - mo["rho"].ravel()) / mo["rho"].ravel()).max() <= 1e-4 * loose


@pytest.mark.parametrize("shape,lattice", [((9, 5, 3), "D3Q27"), ((13, 11, 1), "D2Q9")])
@pytest.mark.parametrize("T0,amp_T,dx,unfit", [
    # nodes either side of the fixed-point range (a step short enough for radicals
    # recombining at 128 K)
    (128.0, 0.1, 1e-6, False),
    (1400.0, 0.02, 1e-3, True),     # an activation energy whose coefficient does not fit
    (1400.0, 0.6, 1e-3, False),     # 560 K to 2240 K
])
def test_rate_arguments(mech, shape, lattice, T0, amp_T, dx, unfit):
    m = mech
    if unfit:
        arr = mech.arrhenius.copy()
        arr[-1, 2] = 9e5        # J/mol; 64 Ea / (R ln 2) above 2^23
        m = dataclasses.replace(mech, arrhenius=arr)
    _parity(m, fields.perturbed_box(shape, lattice, mech=m, T0=T0, amp_T=amp_T, dx=dx), 6)


@pytest.mark.parametrize("shape", [(5, 3, 2), (37, 19, 11)])
def test_fp16_codec_holds_the_initial_populations(mech, shape):
    w = fields.perturbed_box(shape, "D3Q27", mech=mech)
    o, g = make_oracle(mech, w), make_gpu(mech, w, precision="fp16")
    ref, got = oracle_populations(o), g.populations()
    g.close()
    for l in range(ref.shape[0]):
        spread = ref[l].max(axis=1) - ref[l].min(axis=1)     # >= the deviation from the mean's
        tol = 2.0 * (2.0 ** -11 * spread.max() + 2.0 ** -22 * np.abs(ref[l]).max())
        assert np.abs(got[l] - ref[l]).max() <= tol
