"""Sizes and values at which the step's and its companions' branches change:
scan tiles, partial batches and lane groups, facets, rough and scaled fields,
export destinations, and the ranges of the generators' filters.  Each against
the CPU oracle, or bit for bit where both sides run the same rounded sequence.
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


def _square(n, per_cell=None, ppc=5, steps=3, rk=2, seed=3):
    X = W.jittered_vertices(n, seed)
    U = W.zero_wall_normal(n, W.normalise_max(W.stream_function_field(W.q2_node_coords(n, X), seed)))
    return W.Workload("edge", 2, n, X, U, None if per_cell is not None else ppc, per_cell, 2, rk,
                      W.cfl_dt(n, X, U, 0.5), steps, seed, W.particle_seed(seed))


# one scan tile is 4,096 cells: below and at it one launch scans and scatters,
# above it two do
@pytest.mark.parametrize("n", [(1, 1), (3, 1), (33, 31), (64, 64), (64, 65), (4097, 1), (130, 129)])
def test_steps_around_one_scan_tile(P, oracle_mod, n):
    wl = _square(n)
    mesh, parts = H.gpu_seed(wl)
    om, op = H.oracle_seed(oracle_mod, wl)
    for _ in range(2):  # the second call starts from a pending order and scratch cleared by the first
        parts.advect(wl.dt, wl.integrator, wl.n_steps)
        op = oracle_mod.advect(om, op, wl.dt, wl.integrator, wl.n_steps)
        H.assert_same_store(H.gpu_state(parts), op, wl)
        off = parts.cell_offsets().cpu().numpy()
        np.testing.assert_array_equal(np.diff(off), np.bincount(op.cell, minlength=wl.ncells))


# Nodal values without smoothness, and in units far from 1: the grid of the Q2
# sums follows each cell's own bound M.  M is at most ~30 max|U| here (sums of 27
# coefficients), a step moves dt |U| <= h / 2 with an error of 2^-45 M dt, and the
# 2 x 3 steps of 5 cells' width stay below 6 * 0.1 * 30 * 2^-45 = 6e-13.
@pytest.mark.parametrize("scale", [1.0, 1e15, 1e-15])
@pytest.mark.parametrize("n", [(5, 4), (5, 4, 3)])
def test_rough_and_scaled_fields(P, oracle_mod, n, scale):
    X = W.jittered_vertices(n, 4)
    nodes = W.q2_node_coords(n, X).shape[1]
    U = W.zero_wall_normal(n, W.normalise_max(np.random.default_rng(6).standard_normal((len(n), nodes))))
    U[0, ::7] = 0.0
    dt = W.cfl_dt(n, X, U, 0.5)
    wl = W.Workload("rough", len(n), n, X, scale * U, 9, None, 1, 4, dt / scale, 3, 4, W.particle_seed(4))
    mesh, parts = H.gpu_seed(wl)
    om, op = H.oracle_seed(oracle_mod, wl)
    for _ in range(2):
        parts.advect(wl.dt, wl.integrator, wl.n_steps)
        op = oracle_mod.advect(om, op, wl.dt, wl.integrator, wl.n_steps)
    H.assert_same_store(H.gpu_state(parts), op, wl)


# cells of 0 to 9 particles: partial batches of the averages, empty cells and
# ragged ones in the transfers
@pytest.mark.parametrize("n", [(7, 5), (33, 9), (5, 4, 3)])
def test_transfers_of_short_cells(P, oracle_mod, n):
    C = int(np.prod(n))
    per = (np.arange(C) % 10).astype(np.uint32)
    mesh, parts, om, op, vals = T._pair(P, oracle_mod, n, per_cell=per)
    T._check_vertex(oracle_mod, parts, om, op, vals)
    T._check_lsq(oracle_mod, parts, om, op, vals, len(n))
    ga, gc = parts.average(0, empty_fill=-3.0)
    oa, oc = oracle_mod.cell_average(C, op.cell, vals, empty_fill=-3.0)
    np.testing.assert_array_equal(gc.cpu().numpy(), oc)
    np.testing.assert_array_equal(ga.cpu().numpy(), oa)  # the same left fold


# four lanes share a cell from six particles of capacity per cell on
@pytest.mark.parametrize("n", [(9, 7), (5, 4, 3)])
@pytest.mark.parametrize("low, span", [(5, 1), (6, 1), (0, 13), (3, 10)])
def test_vertex_sums_either_side_of_shared_cells(P, oracle_mod, n, low, span):
    C = int(np.prod(n))
    per = (low + np.arange(C) % span).astype(np.uint32)
    mesh, parts, om, op, vals = T._pair(P, oracle_mod, n, per_cell=per)
    T._check_vertex(oracle_mod, parts, om, op, vals)


def test_geometric_mean_of_extreme_values(P, oracle_mod):
    """Subnormal to 1e300, and cells holding an infinity, a NaN, a zero or a
    negative value.  The oracle sums logarithms of up to 710, each within an ulp
    (1.1e-13), so the two agree to 2e-13 of the mean."""
    import torch

    n, ppc = (16, 8), 7
    mesh = P.Mesh(n, W.jittered_vertices(n, 2))
    parts = P.Particles(mesh, uniform_count=ppc, seed=5, n_props=1)
    C = int(np.prod(n))
    g = np.random.default_rng(8)
    v = 10.0 ** g.uniform(-300, 300, size=C * ppc)
    v[: 20 * ppc] = 10.0 ** g.uniform(-322, -306, size=20 * ppc)
    for cell, bad in zip(range(30, 36), (np.inf, np.nan, 0.0, -0.0, -1.0, -np.inf)):
        v[cell * ppc + 3] = bad
    parts.set_property(0, torch.as_tensor(v, device="cuda"))
    got = parts.average(0, kind=P.PIC_AVG_GEOMETRIC)[0].cpu().numpy()
    with np.errstate(all="ignore"):
        want, _ = oracle_mod.cell_average(C, np.repeat(np.arange(C), ppc), v, kind=1)
    np.testing.assert_array_equal(np.isnan(got), np.isnan(want))
    np.testing.assert_array_equal(np.isinf(got), np.isinf(want))
    ok = np.isfinite(want)
    assert np.all(np.abs(got[ok] - want[ok]) <= 2e-13 * want[ok] + 5e-324)


@pytest.mark.parametrize("settled", [False, True])
def test_export_destinations_agree(P, settled):
    """Device arrays (one kernel, through a pending order) against host arrays
    (the order applied, then copies), bit for bit; and a step after either."""
    import torch

    wl = W.curl_cube(6, 7, 2, 3)
    mesh, parts = H.gpu_seed(wl)
    parts.advect(wl.dt, 4, 2)
    if settled:
        parts.vertex_average(0)  # applies the pending order
    dev = parts.export()
    N = dev["id"].shape[0]
    host = {"x": torch.empty((3, N), dtype=torch.float64), "xhat": torch.empty((3, N), dtype=torch.float64),
            "id": torch.empty(N, dtype=torch.int64), "cell": torch.empty(N, dtype=torch.int32),
            "props": torch.empty((3, N), dtype=torch.float64)}
    again = parts.export()
    P.pic_export(parts.h, **host)
    torch.cuda.synchronize()
    for k in host:
        assert torch.equal(dev[k].cpu(), host[k]) and torch.equal(dev[k], again[k]), k
    ref_mesh, ref = H.gpu_seed(wl)
    ref.advect(wl.dt, 4, 3)
    parts.advect(wl.dt, 4, 1)
    a, b = parts.export(), ref.export()
    for k in a:
        assert torch.equal(a[k], b[k]), k


@pytest.mark.parametrize("field", ["x", "xhat", "id", "cell", "props"])
def test_export_to_an_address_no_kernel_can_write(P, field):
    """A device array off its element's alignment takes the copies, bit for bit."""
    import torch

    wl = W.curl_cube(4, 7, 2, 3)
    mesh, parts = H.gpu_seed(wl)
    parts.advect(wl.dt, 4, 1)
    ref = parts.export()
    out = {k: torch.zeros_like(v) for k, v in ref.items()}
    size = ref[field].numel() * ref[field].element_size()
    raw = torch.zeros(size + 16, dtype=torch.uint8, device="cuda")
    shifted = raw[2:2 + size]
    P.pic_export(parts.h, **{**out, field: shifted})
    torch.cuda.synchronize()
    out[field] = shifted.clone().view(ref[field].dtype).reshape(ref[field].shape)
    for k in ref:
        assert torch.equal(out[k], ref[k]), k


@pytest.mark.parametrize("n", [(3, 3), (4, 3, 3)])
def test_points_close_to_facets(P, oracle_mod, n):
    """Points within 1e-11 to 2e-6 of facets, inside and across: the fast path's
    band, the FP64 fallback and the lowest-index rule meet here."""
    import torch

    X = W.jittered_vertices(n, 5)
    om, mesh = oracle_mod.Mesh(n, X), P.Mesh(n, X)
    g = np.random.default_rng(3)
    pts = []
    for K in range(int(np.prod(n))):
        for d in (1e-11, 9e-11, 2e-10, 1e-9, 1e-8, 5e-8, 9e-8, 2e-7, 2e-6):
            for s in (-d, d):
                r = g.uniform(0.1, 0.9, size=len(n))
                r[g.integers(len(n))] = g.integers(2) + s
                pts.append(om.phi(K, r))
    pts = np.array(pts)
    oc, ot = om.locate(pts)
    gc, gt = mesh.locate_points(torch.as_tensor(np.ascontiguousarray(pts.T), device="cuda"))
    gc = gc.cpu().numpy().view(np.uint32).astype(np.int64)
    gc[gc == 0xFFFFFFFF] = -1
    np.testing.assert_array_equal(gc, oc)
    found = oc >= 0
    assert np.abs(gt.cpu().numpy().T[found] - ot[found]).max() <= 1e-14 * 30  # FP64 Newton on both sides


def _weights(kind, C):
    g = np.random.default_rng(C)
    if kind == "uniform":
        return g.uniform(0.0, 1.0, C)
    if kind == "ties":  # remainders of exactly half a spacing
        return g.integers(0, 8, C) * 2.0**-3 * 2.0 ** g.integers(-30, 20, C)
    if kind == "late":  # zeros, then weights over 100 binades
        w = 2.0 ** g.uniform(-50, 50, C)
        w[: C // 2] = 0.0
        return w
    return g.uniform(0.0, 1.0, C) * 2.0**-1060  # subnormal sums


@pytest.mark.parametrize("kind", ["uniform", "ties", "late", "subnormal"])
@pytest.mark.parametrize("C", [1, 255, 256, 257, 256 + 4096, 256 + 4097, 30000])
def test_drawn_counts_at_fold_edges(P, oracle_mod, kind, C):
    """The fold's 256-value prologue and 4,096-value batches; counts equal the
    oracle's, whose fold is a loop."""
    w = _weights(kind, C)
    if not w.sum() > 0:
        w[-1] = 1.0
    got = P.draw_cell_counts(w, 4 * C, 99).cpu().numpy().view(np.uint32).astype(np.int64)
    np.testing.assert_array_equal(got, oracle_mod.draw_cell_counts(w, 4 * C, 99))


@pytest.mark.parametrize("n", [(9, 8), (5, 4, 3)])
@pytest.mark.parametrize("density", ["constant", "zero_cells", "tiny", "huge"])
def test_chains_where_the_filters_cannot_decide(P, oracle_mod, n, density):
    """Undistorted cells of constant density accept with equality at u -> 1, zero
    densities compare 0 < 0, and values outside FP32's range leave every step
    to the written sequence: chains equal the oracle's bit for bit."""
    X = W.uniform_vertices(n) if density == "constant" else W.jittered_vertices(n, 8)
    rho = np.full(X.shape[1], 0.7) if density == "constant" else np.random.default_rng(9).uniform(0.0, 2.0, X.shape[1])
    if density == "zero_cells":
        rho[: X.shape[1] // 2] = 0.0
    rho = rho * {"tiny": 1e-60, "huge": 1e60}.get(density, 1.0)
    mesh, om = P.Mesh(n, X), oracle_mod.Mesh(n, X)
    per = (np.arange(om.ncells) % 7).astype(np.uint32)
    g = H.gpu_state(P.Particles.metropolis_hastings(mesh, per, rho, thinning=3, seed=21, n_props=0))
    o = oracle_mod.seed_particles_mh(om, per, rho, 3, 21)
    np.testing.assert_array_equal(g["cell"], o.cell)
    np.testing.assert_array_equal(g["x"], o.x)
