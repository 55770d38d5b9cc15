"""Values, units and shapes at the ends of the ranges in which the FP32 and
double-float shortcuts may stand for the definition: each against the CPU
oracle, or bit for bit where both sides run the same rounded sequence.
"""
import numpy as np
import pytest

from paper_1612_03369_gb300 import workloads as W
import gpu_helpers as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_1612_03369_gb300 import pic

    return pic


def _chains_equal(P, oracle_mod, n, X, rho, per_cell, thinning):
    mesh, om = P.Mesh(n, X), oracle_mod.Mesh(n, X)
    per = np.full(om.ncells, per_cell, dtype=np.uint32)
    g = H.gpu_state(P.Particles.metropolis_hastings(mesh, per, rho, thinning=thinning, seed=33, n_props=0))
    o = oracle_mod.seed_particles_mh(om, per, rho, thinning, 33)
    np.testing.assert_array_equal(g["cell"], o.cell)
    np.testing.assert_array_equal(g["x"], o.x)


# 70 k steps: of decisions taken from FP32 values of a few of the smallest float,
# some tens would differ from the sequence's
@pytest.mark.parametrize("scale", [1e-36, 1e-39, 1e-40, 1e-41, 1e-42, 1e-43, 1e-44])
@pytest.mark.parametrize("n", [(9, 8), (5, 4, 3)])
def test_chains_of_densities_below_the_normal_floats(P, oracle_mod, n, scale):
    X = W.jittered_vertices(n, 8)
    rho = scale * np.random.default_rng(9).uniform(0.5, 2.0, X.shape[1])
    _chains_equal(P, oracle_mod, n, X, rho, 40, 25)


# the determinant, not the density, leaves the normal floats; and cells so thin
# that only a product of two rows does
@pytest.mark.parametrize("h", [(1e-14, 1e-14, 1e-14), (1e-12, 1e-12, 1e-12), (1e10, 1e-24, 1e-20), (1e-24, 1e-20, 1e10)])
def test_chains_of_cells_in_small_units(P, oracle_mod, h):
    n = (5, 4, 3)
    X = W.jittered_vertices(n, 8) * (np.array(h) * np.array(n))[:, None]
    rho = np.random.default_rng(9).uniform(0.5, 2.0, X.shape[1])
    _chains_equal(P, oracle_mod, n, X, rho, 40, 25)


# the sequence sums whole coordinates: its own error grows with |x| / h, to 2e-6 of
# rho-hat at 1e10 and 2e-4, past FP32's, at 1e12; among 1.4 M steps some fall into it
@pytest.mark.parametrize("offset", [1e6, 1e9, 1e10, 1e11, 1e12])
@pytest.mark.parametrize("n", [(9, 8), (5, 4, 3)])
def test_chains_of_meshes_far_from_the_origin(P, oracle_mod, n, offset):
    X = W.jittered_vertices(n, 8) + offset / max(n)
    rho = np.random.default_rng(9).uniform(0.5, 2.0, X.shape[1])
    _chains_equal(P, oracle_mod, n, X, rho, 200, 100)


# cells whose determinant lies where the FP32 reciprocal of it is 0 (2^126 to 2^128),
# and on either side
@pytest.mark.parametrize("n, h", [((5, 4), 2.0**58), ((5, 4), 2.0**63.5), ((5, 4), 2.0**66),
                                  ((5, 4, 3), 2.0**38), ((5, 4, 3), 2.0**42.3), ((5, 4, 3), 2.0**45)])
def test_steps_in_cells_of_large_units(P, oracle_mod, n, h):
    d = len(n)
    X = W.jittered_vertices(n, 4)
    U = W.zero_wall_normal(n, W.normalise_max(np.random.default_rng(6).standard_normal((d, W.q2_node_coords(n, X).shape[1]))))
    unit = h * np.array(n, dtype=float)[:, None]
    wl = W.Workload("units", d, n, X * unit, U * unit, 9, None, 1, 4, W.cfl_dt(n, X, U, 0.5), 3, 4, W.particle_seed(4))
    mesh, parts = H.gpu_seed(wl, n_props=0)
    om = oracle_mod.Mesh(n, wl.X, wl.U)
    op = oracle_mod.seed_particles(om, uniform_count=9, seed=wl.pseed, n_props=0)
    parts.advect(wl.dt, 4, 3)
    op = oracle_mod.advect(om, op, wl.dt, 4, 3)
    H.assert_same_store(H.gpu_state(parts), op, wl, tol_x=H.TOL_X * unit.max())
