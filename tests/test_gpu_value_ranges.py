"""Values, units and shapes at the ends of the ranges in which the FP32 and
double-float shortcuts may stand for the definition: each against the CPU
oracle, or bit for bit where both sides run the same rounded sequence.
"""
import numpy as np
import pytest

from paper_1612_03369_gb300 import workloads as W
import gpu_helpers as H
import test_gpu_transfer as T

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


def _affine(d, shear):
    """Rotation times shear: an affine map that leaves a box's cells as well shaped as
    its singular values, about `shear` and 1 / `shear`."""
    c, s = np.cos(0.6), np.sin(0.6)
    A = np.eye(d)
    A[0, 1] = shear
    R = np.eye(d)
    R[:2, :2] = [[c, -s], [s, c]]
    if d == 3:
        A[2, 0] = 0.5
        Q = np.eye(3)
        Q[1:, 1:] = [[c, -s], [s, c]]
        R = Q @ R
    return R @ A


def _jacobians(n, X, U, cell, t):
    """dPhi/dt and du/dt at reference coordinates t [N][d] of cells, in extended precision."""
    d, L = len(n), np.longdouble
    t = t.astype(L)
    lin = [(1 - t, -np.ones_like(t)), (t, np.ones_like(t))]
    quad = [(2 * (t - L(0.5)) * (t - 1), 4 * t - 3), (4 * t * (1 - t), 4 - 8 * t), (2 * t * (t - L(0.5)), 4 * t - 1)]
    ijk = np.stack(np.unravel_index(cell, n[::-1])[::-1])

    def deriv(basis, order, values):
        out = np.zeros((len(cell), d, d), dtype=L)
        for corner in np.ndindex(*[order + 1] * d):
            at = np.zeros(len(cell), dtype=np.int64)
            for a in reversed(range(d)):
                at = at * (order * n[a] + 1) + order * ijk[a] + corner[a]
            for j in range(d):
                w = np.ones(len(cell), dtype=L)
                for a in range(d):
                    w = w * basis[corner[a]][1 if a == j else 0][:, a]
                out[:, :, j] += values[:, at].T * w[:, None]
        return out

    return deriv(lin, 1, X), deriv(quad, 2, U)


def _check_reverse_step(P, n, shear, unit, seeds):
    """One Euler step: dL/dx0 = lambda + dt J^-T (du/dt)^T lambda at the seeds' own
    reference coordinates.  Double-float cofactors lose the condition of J times a few
    2^-47 relative to |J^-1| |du/dt| |lambda|; 60 of them are allowed, and of |lambda|
    itself its double-float rounding."""
    import torch

    d = len(n)
    A = _affine(d, shear) * 2.0**unit
    g = np.random.default_rng(12)
    X0 = W.jittered_vertices(n, 4)
    X = A @ X0
    # displacements of 0.02 cells a unit time, whatever the cells' shape
    U = A @ (W.zero_wall_normal(n, g.uniform(-0.02, 0.02, (d, W.q2_node_coords(n, X0).shape[1]))) / np.array(n)[:, None])
    mesh = P.Mesh(n, X, U)
    parts = P.Particles(mesh, uniform_count=50, seed=3, n_props=0)
    st = H.gpu_state(parts)
    N = st["id"].shape[0]
    tape = P.pic_advect_record(parts.h, mesh.h, 1.0, 1, 1)
    ids = H.gpu_state(parts)["id"].astype(np.int64)
    assert len(ids) > N // 4  # the step may lose particles of the most sheared cells
    lam = g.standard_normal((d, N)) * 2.0**seeds
    dU = torch.empty(U.shape, dtype=torch.float64, device="cuda")
    dx0 = torch.empty((d, N), dtype=torch.float64, device="cuda")
    P.pic_tape_adjoint(tape, torch.as_tensor(np.ascontiguousarray(lam[:, ids]), device="cuda"), dU, dx0)
    P.pic_destroy_tape(tape)
    J, Gu = _jacobians(n, X, U, st["cell"], st["xhat"])
    Jf = J.astype(float)
    inv = np.linalg.inv(Jf).astype(np.longdouble)
    for _ in range(4):  # to extended precision
        inv = inv + np.einsum("nij,njk->nik", inv, np.eye(d) - np.einsum("nij,njk->nik", J, inv))
    lt = lam.T.astype(np.longdouble)
    want = lt + np.einsum("nij,ni->nj", inv, np.einsum("nij,ni->nj", Gu, lt))
    size = np.linalg.norm(inv.astype(float), axis=(1, 2)) * np.linalg.norm(Gu.astype(float), axis=(1, 2)) * np.linalg.norm(lam, axis=0)
    tol = 60 * 2.0**-47 * np.linalg.cond(Jf) * size + 2.0**-46 * np.linalg.norm(lam, axis=0)
    err = np.abs((dx0.cpu().numpy().T - want).astype(float)).max(axis=1)
    assert np.all(err[ids] <= tol[ids]), (err[ids] / tol[ids]).max()


# nodal values without smoothness: the second and higher coefficients are the largest
@pytest.mark.parametrize("n", [(6, 5), (4, 3, 4), (2, 2, 2), (7, 2, 3)])
def test_gradient_of_rough_fields(P, n):
    _check_reverse_step(P, n, 0.0, 0, 0)


# J of condition 1 to 4e6, cells and seeds in units far from 1 (powers of two)
@pytest.mark.parametrize("shear, unit, seeds", [(30.0, 0, 0), (300.0, 0, 0), (2000.0, 0, 0), (0.0, -20, -80), (0.0, -30, 0),
                                                (30.0, -20, -80), (0.0, 20, 60)])
@pytest.mark.parametrize("n", [(6, 5), (4, 3, 4)])
def test_reverse_step_of_scaled_and_sheared_cells(P, n, shear, unit, seeds):
    _check_reverse_step(P, n, shear, unit, seeds)


# Newton's iterates are affine invariants, so a box and its affine image give every
# particle the same cells and reference coordinates but for rounding: FP32's, 1e-7
# times the condition A has, ends the FP32 phase and leaves that part of a last step
# of 1e-6 at most; ten of these over the four stages
@pytest.mark.parametrize("shear", [3.0, 10.0, 30.0])
@pytest.mark.parametrize("n", [(6, 5), (4, 3, 4)])
def test_steps_in_sheared_cells(P, n, shear):
    d = len(n)
    A = _affine(d, shear)
    X = W.jittered_vertices(n, 4)
    V = W.zero_wall_normal(n, np.random.default_rng(12).uniform(-0.3, 0.3, (d, W.q2_node_coords(n, X).shape[1]))) / np.array(n)[:, None]
    got = []
    for M in (np.eye(d), A):
        mesh = P.Mesh(n, M @ X, M @ V)
        parts = P.Particles(mesh, uniform_count=50, seed=3, n_props=0)
        parts.advect(1.0, 4, 1)
        got.append(H.gpu_state(parts))
    np.testing.assert_array_equal(got[1]["id"], got[0]["id"])
    np.testing.assert_array_equal(got[1]["cell"], got[0]["cell"])
    assert np.abs(got[1]["xhat"] - got[0]["xhat"]).max() <= 10 * 1e-6 * 1e-7 * np.linalg.cond(A)


# Translation across undistorted cells: x-hat follows from the position exactly.  What
# may remain is the rounding of the position and of its offset from a vertex to 48
# bits, 2^-48 of a coordinate of at most 1 each, in cells; crossing cells adds nothing
# of that size.
@pytest.mark.parametrize("cells", [0.3, 0.8, 1.6])
def test_reference_coordinates_after_crossing_cells(P, cells):
    n = (250, 2)  # vertices that are no double-floats
    X = W.uniform_vertices(n)
    U = np.zeros((2, W.q2_node_coords(n, X).shape[1]))
    U[0] = 1.0
    mesh = P.Mesh(n, X, U)
    parts = P.Particles(mesh, uniform_count=2000, seed=3, n_props=0)
    parts.advect(cells / n[0], 1, 1)
    s = H.gpu_state(parts)
    i = s["cell"] % n[0]
    assert len(i) > 900000
    x, v = s["x"][:, 0].astype(np.longdouble), X[0, : n[0] + 1].astype(np.longdouble)
    t = (x - v[i]) / (v[i + 1] - v[i])
    assert np.abs(s["xhat"][:, 0] - t).max() <= 2 * n[0] * 2.0**-48


# The FP32 phase ends with its residual's noise, ~1.5e-7, whatever the length of the
# last step; the FP32 Jacobian, off by 3e-7 times a condition of 2 here, leaves
# 9e-14 of that, and the position's 48 bits 1e-14.
@pytest.mark.parametrize("amplitude", [0.05, 0.1, 0.3])
@pytest.mark.parametrize("n", [(2, 2), (3, 3)])
def test_end_of_the_inverse_map(P, n, amplitude):
    X = W.jittered_vertices(n, 4, 0.25)
    nodes = W.q2_node_coords(n, X).shape[1]
    U = W.zero_wall_normal(n, np.random.default_rng(4).uniform(-amplitude, amplitude, (2, nodes))) / np.array(n)[:, None]
    mesh = P.Mesh(n, X, U)
    parts = P.Particles(mesh, uniform_count=8000, seed=4, n_props=0)
    parts.advect(1.0, 1, 1)
    s = H.gpu_state(parts)
    i, j = s["cell"] % n[0], s["cell"] // n[0]
    V = [X[:, (i + a) + (n[0] + 1) * (j + b)] for b in (0, 1) for a in (0, 1)]
    t = s["xhat"].copy()
    for _ in range(3):  # Newton in FP64 from the result
        a, b = t.T
        r = s["x"].T - (V[0] + (V[1] - V[0]) * a + (V[2] - V[0]) * b + (V[3] - V[2] - V[1] + V[0]) * a * b)
        J0, J1 = (V[1] - V[0]) * (1 - b) + (V[3] - V[2]) * b, (V[2] - V[0]) * (1 - a) + (V[3] - V[1]) * a
        det = J0[0] * J1[1] - J0[1] * J1[0]
        t = t + np.stack([(r[0] * J1[1] - r[1] * J1[0]) / det, (J0[0] * r[1] - J0[1] * r[0]) / det], axis=1)
    assert np.abs(s["xhat"] - t).max() <= 1e-13


# A cell 2,000 or 8,000 times as long as its neighbour holds points, within its 1e-10
# band, up to 2e-7 and 8e-7 of the neighbour's size into it: the lowest index decides.
@pytest.mark.parametrize("step", [False, True])
@pytest.mark.parametrize("ratio", [10.0, 2000.0, 8000.0])
@pytest.mark.parametrize("d", [2, 3])
def test_lowest_owner_among_uneven_cells(P, oracle_mod, d, ratio, step):
    import torch

    widths = [ratio, 1.0, 2.0, 0.5 * ratio]
    lines = np.concatenate([[0.0], np.cumsum(widths)])
    n = (4,) * d
    X = np.stack([g.ravel() for g in np.meshgrid(*[lines] * d, indexing="ij")][::-1])
    shift = 0.25 if step else 0.0
    pts = []
    for delta in np.array([-1.5, -0.9, -0.5, 0.5, 0.9, 1.5]) * 1e-10 * ratio:
        for a in range(d):
            for facet in lines[1:4]:
                p = np.full(d, ratio + 0.4)
                p[a] = facet + delta + shift
                pts.append(p)
    pts = np.array(pts)
    U = np.full((d, W.q2_node_coords(n, X).shape[1]), -1.0)
    mesh, om = P.Mesh(n, X, U), oracle_mod.Mesh(n, X, U)
    if not step:
        got = mesh.locate_points(torch.as_tensor(np.ascontiguousarray(pts.T), device="cuda"))[0].cpu().numpy()
        np.testing.assert_array_equal(got.view(np.uint32).astype(np.int64), om.locate(pts)[0])
        return
    parts, outside = P.Particles.import_points(mesh, torch.as_tensor(np.ascontiguousarray(pts.T), device="cuda"))
    c, t = om.locate(pts)
    o = np.argsort(c, kind="stable")
    op = oracle_mod.Particles(pts[o], t[o], c[o], o.astype(np.uint64), np.zeros((len(o), 0)))
    parts.advect(shift, 1, 1)
    op = oracle_mod.advect(om, op, shift, 1, 1)
    s = H.gpu_state(parts)
    np.testing.assert_array_equal(s["id"], op.id)
    np.testing.assert_array_equal(s["cell"], op.cell)


@pytest.mark.parametrize("ppc", [3, 5, 9, 20])
def test_vertex_sums_do_not_depend_on_the_room_for_particles(P, ppc):
    import torch

    n = (7, 6, 5)
    mesh = P.Mesh(n, W.jittered_vertices(n, 3))
    C = int(np.prod(n))
    v = torch.as_tensor(np.random.default_rng(2).standard_normal(C * ppc), device="cuda")
    got = []
    for capacity in (0, 6 * C + 40 * C):
        parts = P.Particles(mesh, uniform_count=ppc, seed=5, n_props=1, capacity=capacity)
        parts.set_property(0, v)
        got.append(parts.vertex_average(0))
    for a, b in zip(*got):
        assert torch.equal(a, b)


# the choice between one and four lanes a cell falls at 14 particles in the largest of
# 32 cells; from 77,824 cells a block takes four such groups
@pytest.mark.parametrize("n", [(8, 4), (9, 7), (331, 257)])
@pytest.mark.parametrize("per_cell", ["14", "15", "0..14", "one long", "long groups"])
def test_vertex_sums_of_cell_groups(P, oracle_mod, n, per_cell):
    C = int(np.prod(n))
    per = {"14": np.full(C, 14), "15": np.full(C, 15), "0..14": np.arange(C) % 15, "one long": np.arange(C) % 5,
           "long groups": np.where(np.arange(C) // 32 % 3 == 1, 17 + np.arange(C) % 4, np.arange(C) % 3)}[per_cell]
    if per_cell == "one long":
        per[C // 2] = 75
    if C > 10000:
        per = np.where(np.arange(C) < 70000, per % 8, per)  # most cells short: the oracle's time
    mesh, parts, om, op, vals = T._pair(P, oracle_mod, n, per_cell=per.astype(np.uint32))
    T._check_vertex(oracle_mod, parts, om, op, vals)


# one launch scans and scatters: an odd number of cells per thread, the last runs past
# the end, and more particles than its blocks take in one pass (622,592)
@pytest.mark.parametrize("n, ppc", [((1, 1), 3000), ((255, 1), 7), ((257, 1), 7), ((16, 16), 33), ((47, 87), 9), ((64, 64), 170)])
def test_steps_of_one_scan_tile(P, oracle_mod, n, ppc):
    X = W.jittered_vertices(n, 3)
    U = W.zero_wall_normal(n, W.normalise_max(W.stream_function_field(W.q2_node_coords(n, X), 3)))
    wl = W.Workload("tile", 2, n, X, U, ppc, None, 1, 1, W.cfl_dt(n, X, U, 0.5), 2, 3, W.particle_seed(3))
    mesh, parts = H.gpu_seed(wl)
    om, op = H.oracle_seed(oracle_mod, wl)
    parts.advect(wl.dt, 1, 2)
    op = oracle_mod.advect(om, op, wl.dt, 1, 2)
    H.assert_same_store(H.gpu_state(parts), op, wl)
    np.testing.assert_array_equal(np.diff(parts.cell_offsets().cpu().numpy()), np.bincount(op.cell, minlength=wl.ncells))


# zeros (of either sign) among values at and beyond the range of the split without
# conversions, and nothing but zeros
@pytest.mark.parametrize("values", ["mixed", "zeros"])
@pytest.mark.parametrize("n", [(9, 7), (5, 4, 3)])
def test_transfers_of_zeros(P, oracle_mod, n, values):
    import torch

    per = (np.arange(int(np.prod(n))) * 5 % 19).astype(np.uint32)
    mesh, parts, om, op, vals = T._pair(P, oracle_mod, n, per_cell=per)
    g = np.random.default_rng(4)
    v = np.array([0.0, -0.0, 1.0, -1.0, 2.0**-128, -(2.0**-100), 1e-30])[g.integers(0, 7, op.n)] if values == "mixed" else np.zeros(op.n)
    parts.set_property(0, torch.as_tensor(v, device="cuda"))
    T._check_vertex(oracle_mod, parts, om, op, v)
    T._check_lsq(oracle_mod, parts, om, op, v, len(n))
    if values == "zeros":
        avg, w = parts.vertex_average(0)
        assert (avg[w > 0] == 0).all()


def test_committed_field_with_a_second_field_set(P):
    """A staged field committed while a second field is set: as both set directly, bit
    for bit, so the mean's table follows the committed field."""
    import torch

    wl = W.curl_cube(6, 6, 2, 3)
    second = torch.as_tensor(np.ascontiguousarray(-0.4 * wl.U), device="cuda")
    fields = [torch.as_tensor(np.ascontiguousarray(s * wl.U), device="cuda") for s in (1.0, 0.7, 1.2)]
    got = []
    for staged in (False, True):
        mesh, parts = H.gpu_seed(wl)
        P.pic_set_velocity_dofs(mesh.h, fields[0], U_next=second)
        for f in fields[1:]:
            parts.advect(wl.dt, 4, 1)
            if staged:
                P.pic_stage_velocity_dofs(mesh.h, f)
                P.pic_commit_velocity_dofs(mesh.h)
            else:
                P.pic_set_velocity_dofs(mesh.h, f, U_next=second)
        parts.advect(wl.dt, 4, 1)
        got.append(H.gpu_state(parts))
    for k in got[0]:
        np.testing.assert_array_equal(got[0][k], got[1][k])


def test_two_fields_without_room_for_the_table_of_their_mean(P, oracle_mod):
    """With 95 MB left on the device the second field's arrays (72 MB) fit and the
    mean's table (46 MB) does not: the step evaluates both fields in its middle."""
    import torch

    wl = W.curl_cube(40, 1, 1, 3)
    mesh, parts = H.gpu_seed(wl)
    om, op = H.oracle_seed(oracle_mod, wl)
    second = -0.4 * wl.U
    first_d, second_d = (torch.as_tensor(np.ascontiguousarray(f), device="cuda") for f in (wl.U, second))
    P.pic_set_velocity_dofs(mesh.h, first_d)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    room = torch.cuda.mem_get_info()[0] - (95 << 20)
    try:
        fill = torch.empty(room, dtype=torch.uint8, device="cuda")
        before = P.pic_kernel_launches()
        P.pic_set_velocity_dofs(mesh.h, first_d, U_next=second_d)
        built = P.pic_kernel_launches() - before
    except (P.PicError, torch.OutOfMemoryError):
        pytest.skip("the device's memory could not be filled to within 95 MB")
    finally:
        fill = None
        torch.cuda.empty_cache()
    if built != 4:  # a fifth launch builds the mean's table
        pytest.skip("the device's memory could not be filled to within 95 MB")
    om.set_velocity_next(second)
    parts.advect(wl.dt, 4, 1)
    H.assert_same_store(H.gpu_state(parts), oracle_mod.advect(om, op, wl.dt, 4, 1), wl)
