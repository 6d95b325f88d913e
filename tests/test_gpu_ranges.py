"""The kernels' arithmetic at the edges of its ranges, against the CPU oracle."""
import dataclasses

import numpy as np
import pytest

from lbm_workloads import fields
from lbm_workloads.mechanism import R_UNIVERSAL, h2_air_synthetic
from oracle.diagnostics import diagnostics
from paper_2108_07605_gb300 import lbm

from helpers import make_gpu, make_oracle, max_rel_err_per_lattice, oracle_populations

pytestmark = pytest.mark.gpu
RTOL_FP64 = 1e-10      # relative per lattice, the bound of the other parity tests


@pytest.fixture(scope="module")
def mech():
    return h2_air_synthetic()


def _errors(mech, w, nsteps, precision="fp64"):
    o, g = make_oracle(mech, w), make_gpu(mech, w, precision=precision)
    o.step(nsteps)
    g.step(nsteps)
    err = max_rel_err_per_lattice(g.populations(), oracle_populations(o))
    g.close()
    return err


def _inert(mech, D0):
    """The mechanism's species without reactions."""
    M = mech.n_species
    return dataclasses.replace(
        mech, nu_f=np.zeros((0, M)), nu_r=np.zeros((0, M)), arrhenius=np.zeros((0, 3)),
        third_body=np.zeros(0, dtype=np.int32), efficiency=np.ones((0, M)),
        reversible=np.zeros(0, dtype=np.int32), D0=D0)


# The fixed-point rate arguments hold 1/T below 2^-7 (T above 128 K) and T below
# 2^14 K.
def _at_temperature(mech, shape, T0):
    w = fields.perturbed_box(shape, "D2Q9", mech=mech, T0=T0, amp_T=0.0, amp_u=0.0,
                             dx=1e-6 if T0 < 200.0 else 1e-9)
    w["Y"][:] = w["Y"][:, :1, :1, :1]      # radicals present
    if T0 > 3000.0:
        w["T_max"] = 17000.0
    return w


@pytest.mark.parametrize("T0", [128.0, 16384.0])
def test_heat_release_at_the_bounds_of_the_rate_arguments(mech, T0):
    """Nodes on the bound itself and a spacing beside it: the temperature solve's
    rounding spreads them."""
    w = _at_temperature(mech, (37, 23, 1), T0)
    o, g = make_oracle(mech, w), make_gpu(mech, w)
    T = g.moments()["T"]
    assert (T == T0).any() and (T < T0).any()
    d, m = g.diagnostics(), o.moments()
    g.close()
    ref = diagnostics(mech, m["rho"], m["u"], m["T"], m["Y"], w["dx"], 2, w["shape"][0])
    for k in ("hrr_integral", "hrr_max"):
        assert abs(d[k] / ref[k] - 1.0) < RTOL_FP64, (k, d[k], ref[k])


@pytest.mark.parametrize("precision,tol", [("fp64", RTOL_FP64), ("fp32c64", 1e-4)])
def test_step_at_the_lower_bound_of_the_rate_arguments(mech, precision, tol):
    """Forty uniform states at 128 K, each with its own rounding of T."""
    worst = np.zeros(mech.n_species + 1)
    w = _at_temperature(mech, (5, 3, 1), 128.0)
    for k in range(40):
        w["P"][:] = 101325.0 * (1.0 + 1e-3 * k)
        worst = np.maximum(worst, _errors(mech, w, 1, precision))
    assert np.all(worst < tol), worst


# Trace species: rates of progress from 1e-36 down to 1e-56 mol/(m^3 s) below those
# of the main species, and a rate constant beyond e^200.  Relative to the species'
# own lattice, as everywhere; rounding of T (Ea / (R T) up to 175) leaves 4e-14.
def _without_radicals(mech, T0):
    w = fields.perturbed_box((9, 5, 3), "D3Q27", mech=mech, T0=T0, dx=25e-6)
    for s in ("H2O", "H", "O", "OH", "HO2", "H2O2"):
        w["Y"][mech.index(s)] = 0.0
    w["Y"] /= w["Y"].sum(axis=0)
    return w


def _one_step_errors(mech, w, lanes):
    o, g = make_oracle(mech, w), make_gpu(mech, w)
    g.set_launch(chem_lanes=lanes)
    o.step(1)
    g.step(1)
    got, ref = g.populations(), oracle_populations(o)
    g.close()
    present = np.abs(ref).max(axis=(1, 2)) > 0.0
    assert np.all(got[~present] == 0.0)
    return max_rel_err_per_lattice(got[present], ref[present])


@pytest.mark.parametrize("lanes", [1, 8])
@pytest.mark.parametrize("T0", [300.0, 700.0])
def test_radicals_formed_in_a_fresh_mixture(mech, T0, lanes):
    err = _one_step_errors(mech, _without_radicals(mech, T0), lanes)
    assert np.all(err < RTOL_FP64), err


@pytest.mark.parametrize("lanes", [1, 8])
def test_rate_constant_far_beyond_its_products(mech, lanes):
    arr, rev = mech.arrhenius.copy(), mech.reversible.copy()
    arr[-1], rev[-1] = (1e88, 0.0, 0.0), 0            # H2O2 + OH, both at 1e-45
    m = dataclasses.replace(mech, arrhenius=arr, reversible=rev)
    w = _without_radicals(m, 700.0)
    for s in ("H2O2", "OH"):
        w["Y"][m.index(s)] = 1e-45
    err = _one_step_errors(m, w, lanes)
    assert np.all(err < RTOL_FP64), err


# One step without reactions, composition as noise (diffusion velocities of the
# order of the lattice speed for the lightest species), 1/tau from 3 to 3e5.  A
# population is some ten roundings of terms of up to twice its size: 18 spacings
# of FP64.  (Coefficients of 48 bits would leave 2^-48 of the same terms, 6e-15
# and more.)
@pytest.mark.parametrize("split", [0, 1])
@pytest.mark.parametrize("scale", [10.0, 1.0, 0.1, 1e-2, 1e-4])
def test_species_relaxation_keeps_fp64(mech, scale, split):
    m = _inert(mech, mech.D0 * scale)
    w = fields.perturbed_box((9, 5, 3), "D3Q27", mech=m, T0=1300.0, dx=25e-6)
    o, g = make_oracle(m, w), make_gpu(m, w)
    g.set_launch(collide_split=split)
    o.step(1)
    g.step(1)
    err = max_rel_err_per_lattice(g.populations(), oracle_populations(o))
    g.close()
    assert np.all(err < 18 * 2.0 ** -52), err


# Trace species between main ones: their Stefan-Maxwell term scales with their mass
# fraction, its coefficient far below FP32's numbers.  And diffusivities so small
# that m_a m_b D_ab alone leaves FP32's range.
@pytest.mark.parametrize("split", [0, 1])
@pytest.mark.parametrize("trace", [1e-25, 1e-36, 1e-60])
def test_trace_species_diffuse_as_the_others(mech, trace, split):
    m = _inert(mech, mech.D0)
    w = fields.perturbed_box((9, 5, 3), "D3Q27", mech=m, T0=1300.0, dx=25e-6, amp_Y=0.2)
    for s in ("H", "O", "OH", "HO2", "H2O2"):
        w["Y"][m.index(s)] *= trace
    w["Y"][8] = 1.0 - w["Y"][:8].sum(axis=0)
    o, g = make_oracle(m, w), make_gpu(m, w)
    g.set_launch(collide_split=split)
    o.step(3)
    g.step(3)
    err = max_rel_err_per_lattice(g.populations(), oracle_populations(o))
    g.close()
    assert np.all(err < RTOL_FP64), err


def test_formed_radicals_diffuse(mech):
    err = _errors(mech, _without_radicals(mech, 300.0), 3)
    assert np.all(err < RTOL_FP64), err


@pytest.mark.parametrize("shape,lattice", [((9, 5, 3), "D3Q27"), ((13, 11, 1), "D2Q9")])
def test_tiny_diffusivities(mech, shape, lattice):
    m = _inert(mech, mech.D0 * 1e-28)
    m.D0[0, :] *= 1e-4
    m.D0[:, 0] = m.D0[0, :]
    err = _errors(m, fields.perturbed_box(shape, lattice, mech=m, T0=1300.0, dx=25e-6), 2)
    assert np.all(err < RTOL_FP64), err


def test_fp32_storage_holds_denormal_populations(mech):
    """A species at mass fractions of 1e-40 to 1e-38 in FP32 storage: populations
    rounded to FP32 (its denormals among them), read out as they are stored."""
    w = fields.perturbed_box((9, 5, 3), "D3Q27", mech=mech, T0=1300.0, dx=25e-6)
    Y = w["Y"][3]
    Y[:] = 1e-40 * (1.0 + 100.0 * np.arange(Y.size).reshape(Y.shape) / Y.size)
    o, g = make_oracle(mech, w), make_gpu(mech, w, precision="fp32")
    ref, got, m = oracle_populations(o), g.populations(), g.moments()
    g.close()
    assert np.all(np.abs(got[3] - ref[3]) <= 2.0 ** -24 * np.abs(ref[3]) + 2.0 ** -150)
    assert np.allclose(m["Y"][3], got[3].sum(axis=0) / got[8].sum(axis=0), rtol=1e-12, atol=0.0)


@pytest.mark.parametrize("lattice,shape", [("D3Q27", (5, 4, 3)), ("D2Q9", (7, 5, 1))])
@pytest.mark.parametrize("precision", ["fp32", "fp32c64"])
def test_substep_energies_of_unrounded_mass_fractions(mech, precision, lattice, shape):
    """A uniform state at rest: rho = 13, Y = (10/13, 3/13) and theta = 1/4 make
    its populations and their sums exact in FP32, the mass fractions not, and
    formation enthalpies that cancel in the mixture turn FP32 rounding of Y into
    0.02 K (6e-5), Ea / (R T) = 100 times that in a rate.  The first of eight
    sub-steps takes that temperature, the others that of rho_a / rho: a trace
    product, constant rate k C_a, is off by 6e-3 / 8, and what FP32 rounds of the
    energy (1e-7) times 100."""
    M, a, c, b = mech.n_species, 0, 1, mech.n_species - 1
    h, nu_f, nu_r = np.zeros(M), np.zeros((1, M)), np.zeros((1, M))
    h[a], h[b] = 1e7, -1e7 / 0.3
    nu_f[0, a] = nu_r[0, c] = 1
    T, N = 300.0, int(np.prod(shape))
    m = dataclasses.replace(
        mech, molar_mass=np.full(M, 28e-3), cp_coeffs=np.tile([3.5, 0.0, 0.0], (M, 1)),
        h_formation=h, s_standard=np.full(M, 150.0), nu_f=nu_f, nu_r=nu_r,
        arrhenius=np.array([[1e-3 * np.exp(100.0), 0.0, 100.0 * R_UNIVERSAL * T]]),
        third_body=np.zeros(1, dtype=np.int32), efficiency=np.ones((1, M)),
        reversible=np.zeros(1, dtype=np.int32), D0=np.full((M, M), 2e-5))
    c_ref = float(np.sqrt(4.0 * R_UNIVERSAL / 28e-3 * T))
    Y = np.zeros((M, N))
    Y[a], Y[b] = 10.0 / 13.0, 3.0 / 13.0
    s = lbm.Solver(m, lattice=lattice, shape=shape, dx=1e-6, precision="fp32",
                   chem_fp64=int(precision == "fp32c64"), substeps=8, c_ref=c_ref)
    s.set_launch(chem_lanes=1)
    s.init_fields(np.full(N, 13.0), np.zeros((3, N)), np.full(N, T), Y)
    s.step(1)
    made = s.populations()[c].sum(axis=0)
    s.close()
    assert np.abs(made / (1e-3 * 10.0 * 1e-6 / c_ref) - 1.0).max() < 1.5 * 6.4e-3 / 8


# 2 nx + 12 interface nodes either side of the precisions' lines between a warp and
# a thread per interface node
@pytest.mark.parametrize("nx,precision", [(2042, "fp64"), (2043, "fp64"), (1018, "fp32c64"),
                                          (1019, "fp32c64")])
def test_boundary_kernels_either_side_of_their_line(mech, nx, precision):
    w = fields.channel_2d(nx=nx, ny=8, dx=25e-6)
    w["u"][:2] += 0.05 * fields.philox(3).uniform(-1.0, 1.0, size=w["u"][:2].shape)
    o, g = make_oracle(mech, w), make_gpu(mech, w, precision=precision)
    o.step(3)
    g.step(3)
    if precision == "fp64":
        err = max_rel_err_per_lattice(g.populations(), oracle_populations(o))
        g.close()
        assert np.all(err < RTOL_FP64), err
        return
    mo, mg = o.moments(), g.moments()             # FP32 storage's field tolerances
    g.close()
    assert np.abs(mg["Y"] - mo["Y"].reshape(mech.n_species, -1)).max() <= 2e-5
    assert np.abs(mg["T"] - mo["T"].ravel()).max() <= 0.05
    assert (np.abs(mg["rho"] - mo["rho"].ravel()) / mo["rho"].ravel()).max() <= 1e-4
