"""Every form of the push (gamma by integers, roots next to one, the general
one; with and without a magnetic field) gives the oracle's steps bit for bit.
In vacuum with all azimuths zero, nothing in a history depends on a library
function, so all tallies and end states are equal; the speeds lie on both sides
of the lines between the forms, and an axial field takes particles across."""
import math

import numpy as np
import pytest

import oracle
from paper_2503_10263_gb300 import inputs
from tests.test_oracle_orbit import C, _orbit, _prims, _vacuum

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def karl():
    from paper_2503_10263_gb300 import karl as k
    k.load()
    return k


def _energy(u, species):
    m = float(inputs.SPECIES_MASS_EV[species])
    x = (u / C) ** 2
    return m * x / (math.sqrt(1 + x) + 1)


@pytest.mark.parametrize("b_t,e_r,e_z", [(0.0, 0.0, 0.0), (0.0, 50.0, 3000.0), (0.3, 0.0, 0.0),
                                         (-0.3, 40.0, -3000.0)])
@pytest.mark.parametrize("species", [inputs.E, inputs.T2P])
def test_vacuum_steps_are_the_oracles(karl, species, b_t, e_r, e_z):
    speeds = [300.0, 4e3, 8.4e3, 8.6e3, 9.2e3, 1.7e4, 5.1e4, 5.3e4, 3.9e5, 4.2e5, 3e6, 6e7, 5e8]
    if species == inputs.T2P:
        speeds = speeds[:11]
    omega = 0.3 * C * C / float(inputs.SPECIES_MASS_EV[species])
    u = np.repeat(speeds, 8)
    mu = np.tile([-0.95, -0.6, -0.2, 0.0, 0.1, 0.4, 0.7, 1.0], len(speeds))
    n = len(u)
    prob = _vacuum(length=0.8, nz=7, lifetime=100.0 / omega)
    orb = _orbit(0.3, frac=0.07, tube_radius_m=0.05, n_rbins=6, e_r_vm2=e_r,
                 e_z_vm=np.linspace(0.5, 1.5, 7) * e_z if e_z else None)
    orb.b_t = b_t
    pr = _prims(np.linspace(-0.045, 0.045, n), np.linspace(0.01, -0.02, n),
                np.linspace(0.05, 0.75, n), [_energy(v, species) for v in u], mu, 0.0, species)
    ctx = karl.Context(prob)
    try:
        g = ctx.run_orbit(orb, pr, seed=4)
    finally:
        ctx.close()
    o = oracle.orbit_run(prob, orb, pr, seed=4, n_threads=8)
    assert g["ledger"][karl.OB_N_STEPS] > 10 * n
    for k in ("ledger", "per_primary", "time_z", "time_r", "cross_pos", "cross_neg", "rcross_out",
              "rcross_in", "wall", "spectrum", "end_state"):
        np.testing.assert_array_equal(g[k], o[k], err_msg=k)


@pytest.mark.parametrize("radius,dt,x", [(0.05, 1e31, 0.01), (1e39, 3e30, 7e38), (3e-30, 1e-38, 1e-30),
                                         (1e-17, 1e-26, 3e-18)])
def test_lengths_beyond_fp32(karl, radius, dt, x):
    # the step tells wall and radial bin by FP32 squares where these are far
    # from an edge; lengths whose squares or values leave FP32 take the exact way
    prob = _vacuum(length=1.0, nz=7)
    orb = inputs.Orbit(b_t=0.0, dt_s=np.full(4, dt), tube_radius_m=radius, n_rbins=6, max_steps=40)
    n = 16
    a = np.linspace(0.0, 0.9, n)
    pr = _prims(x * a, 0.5 * x * a, np.linspace(0.1, 0.9, n), _energy(5e8, inputs.T2P),
                np.where(np.arange(n) % 2, 0.0, 1e-4), 0.0, inputs.T2P)
    ctx = karl.Context(prob)
    try:
        g = ctx.run_orbit(orb, pr, seed=4)
    finally:
        ctx.close()
    o = oracle.orbit_run(prob, orb, pr, seed=4, n_threads=4)
    for k in ("ledger", "per_primary", "time_r", "cross_pos", "cross_neg", "rcross_out", "rcross_in",
              "wall", "spectrum", "end_state"):
        np.testing.assert_array_equal(g[k], o[k], err_msg=k)
