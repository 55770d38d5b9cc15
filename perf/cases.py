"""The work that users of this package have it do, as cases that can be timed and compared.

Each case is one use of the public Python entry points (`paper_1612_03369_gb300.pic`): time steps of a particle store
in 2D and 3D, in both precision forms, with steady and with changing fields; gradients through the steps; ensembles of
problems; property ODEs; particle-to-field transfers; particle generation.  Sizes come from the package's workloads
(32^2 x 16, 64^3 x 20, 128^3 x 20, 32^3 x 32, 64 members of 64^2..512^2) or are plain ragged boxes.

`exact` computes what `run` returns with torch tensors in 64 bits: the full nodal sums of the Q2 field, Newton's
method on the (bi/tri)linear map, the classical RK tableaux, sums over the particles of a cell.
"""
import math

import torch

from paper_1612_03369_gb300 import pic as P

F64 = torch.float64
DEV = "cuda"


# --------------------------------------------------------------------------- inputs


def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + stream) % (1 << 62))
    return g


def _rand(seed, stream, *shape):
    return torch.rand(*shape, generator=_gen(seed, stream), device=DEV, dtype=F64)


def _grid_index(shape):
    """Index of every point of a grid along each axis, x running fastest: list of int64 [points]."""
    flat = torch.arange(math.prod(shape), device=DEV)
    out = []
    for m in shape:
        out.append(flat % m)
        flat = flat // m
    return out


def _vertices(n, seed):
    """Unit box, every coordinate of every interior vertex moved by U(-0.1 h, 0.1 h): [dim][vertices]."""
    idx = _grid_index([m + 1 for m in n])
    inside = torch.ones_like(idx[0], dtype=torch.bool)
    for a, m in enumerate(n):
        inside &= (idx[a] > 0) & (idx[a] < m)
    move = _rand(seed, 1, len(n), idx[0].numel()) * 0.2 - 0.1
    return torch.stack([idx[a].to(F64) / m + torch.where(inside, move[a] / m, 0.0) for a, m in enumerate(n)])


def _q2_nodes(n, X):
    """Coordinates of the Q2 nodes (averages of the vertices around them) and their indices."""
    idx = _grid_index([2 * m + 1 for m in n])
    out = torch.zeros(len(n), idx[0].numel(), dtype=F64, device=DEV)
    for corner in range(1 << len(n)):
        v, stride = torch.zeros_like(idx[0]), 1
        for a, m in enumerate(n):
            v += (idx[a] // 2 + (idx[a] % 2) * ((corner >> a) & 1)) * stride
            stride *= m + 1
        out += X[:, v]
    return out / (1 << len(n)), idx


def _field(n, X, seed, stream=2):
    """Divergence-free field of 8 random-phase modes with no flow through the walls, max speed 1: [dim][nodes]."""
    p, idx = _q2_nodes(n, X)
    pi, d = math.pi, len(n)
    k = torch.randint(1, 4, (8, d), generator=_gen(seed, stream), device=DEV).to(F64) * pi
    phase = _rand(seed, stream + 100, 8, d) * 2 * pi
    s, c = torch.sin(pi * p), torch.cos(pi * p)
    potentials = 1 if d == 2 else 3
    g = torch.zeros(potentials, p.shape[1], dtype=F64, device=DEV)
    dg = torch.zeros(potentials, d, p.shape[1], dtype=F64, device=DEV)
    for m in range(8):
        arg = (k[m][:, None] * p).sum(0)
        for i in range(potentials):
            g[i] += torch.cos(arg + phase[m, i])
            sn = torch.sin(arg + phase[m, i])
            for j in range(d):
                dg[i, j] -= k[m, j] * sn
    if d == 2:
        u = torch.stack([s[0] * (pi * c[1] * g[0] + s[1] * dg[0, 1]), -s[1] * (pi * c[0] * g[0] + s[0] * dg[0, 0])])
    else:
        u = torch.stack([
            s[0] * (dg[2, 1] * s[1] + g[2] * pi * c[1] - dg[1, 2] * s[2] - g[1] * pi * c[2]),
            s[1] * (dg[0, 2] * s[2] + g[0] * pi * c[2] - dg[2, 0] * s[0] - g[2] * pi * c[0]),
            s[2] * (dg[1, 0] * s[0] + g[1] * pi * c[0] - dg[0, 1] * s[1] - g[0] * pi * c[1])])
    for a, m in enumerate(n):
        u[a][(idx[a] == 0) | (idx[a] == 2 * m)] = 0.0
    return u / u.square().sum(0).sqrt().max()


def _dt(n, X):
    """Half the shortest cell edge at unit speed."""
    V = X.reshape(len(n), *[m + 1 for m in reversed(n)])
    return 0.5 * min(float(V.diff(dim=a + 1).square().sum(0).min()) for a in range(len(n))) ** 0.5


def _counts(ncells, median, seed, stream=3):
    """Uneven particles per cell: log-normal, at most 16 times the median, some cells empty.  The seed deals the same
    numbers out to other cells, so the total depends on the mesh alone."""
    z = torch.randn(ncells, generator=_gen(0, stream), device=DEV, dtype=F64)
    n = torch.clamp((median * z.exp()).round(), 0, 16 * median).to(torch.int32)
    return n[torch.randperm(ncells, generator=_gen(seed, stream), device=DEV)]


def _pseed(seed, stream=4):
    return (int(seed) * 6364136223846793005 + stream * 1442695040888963407) % (1 << 63)


def _n(case):
    return tuple(int(case[k]) for k in ("n0", "n1", "n2") if case.get(k))


def _members(case):
    """Sides of an ensemble's square meshes, log-uniform between the two given ones."""
    P_, lo, hi = case["members"], math.log2(case["side_min"]), math.log2(case["side_max"])
    return [int(round(2 ** (lo + (hi - lo) * ((0.6180339887498949 * (p + 1)) % 1.0)))) for p in range(P_)]


def _mesh(n, X, U=None, U_next=None):
    mesh = P.Mesh(n, X.cpu().numpy())
    if U is not None:
        P.pic_set_velocity_dofs(mesh.h, U, U_next=U_next)
    return mesh


def _store(mesh, case, seed, n_props):
    if case.get("uneven"):
        return P.Particles(mesh, per_cell=_counts(mesh.ncells, case["ppc"], seed).cpu().numpy(), seed=_pseed(seed),
                           n_props=n_props)
    return P.Particles(mesh, uniform_count=case["ppc"], seed=_pseed(seed), n_props=n_props)


def _coordinates_as_properties(parts, n_props):
    """Properties q < dim are the particles' first positions (all positive); further ones cos(3 x_0) + 2."""
    x = parts.export()["x"]
    for q in range(n_props):
        parts.set_property(q, x[q].contiguous() if q < x.shape[0] else torch.cos(3 * x[0]) + 2.0)


def _density(n, X):
    """A vertex density that a run would seed more tracers by: larger near one corner, zero nowhere."""
    return 0.2 + torch.exp(-3.0 * (X - 0.25).square().sum(0))


ALPHA, BETA = 0.7, 0.3  # the damage ODE's growth and healing rates


# --------------------------------------------------------------------------- the cases


def listed():
    return [
        # A 2D test problem as one starts with: few particles, RK2, a cell average after every step.  Launches count.
        dict(name="square32_rk2", kind="steps", n0=32, n1=32, ppc=16, rk=2, precision=0, steps=10, props=1, average=1),
        # A small 3D box, one RK4 step and its averages: the smallest call of a coupled 3D run.
        dict(name="cube16_rk4", kind="steps", n0=16, n1=16, n2=16, ppc=20, rk=4, precision=0, steps=1, props=3,
             average=1),
        # The ordinary 3D run: 64^3 cells, 20 particles per cell, RK4, then the state is read.
        dict(name="cube64_rk4", kind="steps", n0=64, n1=64, n2=64, ppc=20, rk=4, precision=0, steps=5, props=3,
             average=0),
        # The largest mesh.
        dict(name="cube128_rk4", kind="steps", n0=128, n1=128, n2=128, ppc=20, rk=4, precision=0, steps=2, props=3,
             average=0),
        # A box of odd side lengths with uneven, partly empty cells, RK2.
        dict(name="box_uneven_rk2", kind="steps", n0=37, n1=61, n2=50, ppc=10, uneven=1, rk=2, precision=0, steps=4,
             props=2, average=0),
        # The FP32-basis precision form.
        dict(name="cube64_fp32", kind="steps", n0=64, n1=64, n2=64, ppc=20, rk=4, precision=1, steps=5, props=3,
             average=0),
        # One step of a run coupled to a flow solver: new fields (time-interpolated), RK4, averages of the properties.
        dict(name="cube64_coupled", kind="coupled", n0=64, n1=64, n2=64, ppc=20, rk=4, precision=0, two=1, props=3),
        # Inverse flow reconstruction: a loss on the final positions and its gradient in the nodal velocities.
        dict(name="adjoint32", kind="adjoint", n0=32, n1=32, n2=32, ppc=32, rk=4, steps=20, tape=0),
        # Many independent 2D problems of uneven size advanced in one persistent launch.
        dict(name="ensemble64", kind="ensemble", members=64, side_min=64, side_max=512, ppc=8, rk=4, steps=10),
        # Strain-driven damage and the deformation gradient integrated with the particles.
        dict(name="cube64_odes", kind="odes", n0=64, n1=64, n2=64, ppc=20, rk=4, steps=2),
        # Particle-to-field transfers of one property: cell means of three kinds, vertex averages, linear fits.
        dict(name="cube64_transfers", kind="transfers", n0=64, n1=64, n2=64, ppc=20),
        # Generation: tracers drawn by a density and thinned chains in the cells; tracers at prescribed positions.
        dict(name="generate48", kind="generate", n0=48, n1=48, n2=48, ppc=16, thinning=8),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def box(dim, lo, hi):
        side = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        n = [max(3, int(round(side * rng.uniform(0.7, 1.4)))) for _ in range(dim)]
        return dict(zip(("n0", "n1", "n2"), n))

    kind = rng.choice(["steps"] * 5 + ["coupled", "adjoint", "ensemble", "odes", "transfers", "generate"])
    dim = rng.choice([2, 3, 3])
    ppc = size(4, 36)
    if kind == "steps":
        return dict(kind=kind, **box(dim, 20 if dim == 2 else 8, 700 if dim == 2 else 72), ppc=ppc,
                    uneven=rng.choice([0, 0, 1]), rk=rng.choice([1, 2, 4, 4]), precision=rng.choice([0, 0, 0, 1]),
                    steps=rng.randint(1, 6), props=rng.randint(1, 4), average=rng.choice([0, 1]))
    if kind == "coupled":
        return dict(kind=kind, **box(dim, 16 if dim == 2 else 8, 500 if dim == 2 else 60), ppc=ppc,
                    uneven=rng.choice([0, 1]), rk=rng.choice([2, 4]), precision=rng.choice([0, 0, 1]),
                    two=rng.choice([0, 1]), props=rng.randint(1, 3))
    if kind == "adjoint":
        return dict(kind=kind, **box(dim, 12 if dim == 2 else 6, 120 if dim == 2 else 28), ppc=ppc,
                    rk=rng.choice([2, 4]), steps=rng.randint(2, 12), tape=rng.choice([0, 1]))
    if kind == "ensemble":
        return dict(kind=kind, members=rng.randint(3, 24), side_min=size(16, 64), side_max=size(80, 300), ppc=8,
                    rk=rng.choice([2, 4]), steps=rng.randint(1, 8))
    if kind == "odes":
        return dict(kind=kind, **box(dim, 16 if dim == 2 else 8, 300 if dim == 2 else 50), ppc=ppc,
                    rk=rng.choice([2, 4]), steps=rng.randint(1, 3))
    if kind == "transfers":
        return dict(kind=kind, **box(dim, 20 if dim == 2 else 8, 600 if dim == 2 else 64), ppc=ppc,
                    uneven=rng.choice([0, 1]))
    return dict(kind=kind, **box(dim, 16 if dim == 2 else 8, 250 if dim == 2 else 40), ppc=ppc,
                thinning=rng.randint(2, 10))


# --------------------------------------------------------------------------- prepare and run


def prepare(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        meshes, dts, per_cell = [], [], []
        for p, side in enumerate(_members(case)):
            X = _vertices((side, side), seed * 131 + p)
            meshes.append(_mesh((side, side), X, _field((side, side), X, seed * 131 + p)))
            dts.append(_dt((side, side), X))
            per_cell.append(_counts(side * side, case["ppc"], seed * 131 + p).cpu().numpy())
        ens = P.Ensemble(meshes, per_cell=per_cell, seeds=[_pseed(seed, p) for p in range(len(meshes))])
        ens.set_dt(dts)
        return {"case": case, "meshes": meshes, "ens": ens}
    n = _n(case)
    X = _vertices(n, seed)
    s = {"case": case, "dt": _dt(n, X)}
    if kind == "generate":
        s["mesh"] = _mesh(n, X)
        s["rho"], s["seed"] = _density(n, X), _pseed(seed)
        s["x"] = _import_points(case, seed)
        return s
    U = _field(n, X, seed)
    if kind == "adjoint":
        s["mesh"], s["U"], s["seed"] = _mesh(n, X, U), U.clone().requires_grad_(True), _pseed(seed)
        s["target"] = _rand(seed, 5, len(n), math.prod(n) * case["ppc"])
        return s
    if kind == "coupled":
        s["fields"], s["k"] = [U, _field(n, X, seed, 20), _field(n, X, seed, 40)], 0
        s["mesh"] = _mesh(n, X, U)
        s["parts"] = _store(s["mesh"], case, seed, case["props"])
        _coordinates_as_properties(s["parts"], case["props"])
        return s
    s["mesh"] = _mesh(n, X, U)
    d = len(n)
    props = case.get("props", 1) if kind != "odes" else 1 + d * d
    s["parts"] = _store(s["mesh"], case, seed, props)
    if kind == "odes":
        N = s["parts"].state()[0]
        for q in range(props):  # damage 0.1, deformation gradient the identity
            v = 0.1 if q == 0 else float((q - 1) % (d + 1) == 0)
            s["parts"].set_property(q, torch.full((N,), v, dtype=F64, device=DEV))
    else:
        _coordinates_as_properties(s["parts"], props)
    return s


def _import_points(case, seed):
    """Prescribed positions: as many as ppc per cell, one in 33 of them beyond the unit box."""
    n = _n(case)
    x = _rand(seed, 6, len(n), math.prod(n) * case["ppc"])
    x[0, ::33] += 1.0
    return x


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "steps":
        parts, avg = s["parts"], []
        if case["average"]:
            for _ in range(case["steps"]):
                parts.advect(s["dt"], case["rk"], 1, case["precision"])
                avg.append(parts.average(0))
        else:
            parts.advect(s["dt"], case["rk"], case["steps"], case["precision"])
        return {"average": avg, "store": parts.export()}
    if kind == "coupled":
        parts, f, k = s["parts"], s["fields"], s["k"]
        P.pic_set_velocity_dofs(s["mesh"].h, f[k % 3], U_next=f[(k + 1) % 3] if case["two"] else None)
        s["k"] = k + 1
        parts.advect(s["dt"], case["rk"], 1, case["precision"])
        avg = [parts.average(q) for q in range(case["props"])]
        return {"average": avg, "store": parts.export()}
    if kind == "adjoint":
        U = s["U"]
        U.grad = None
        parts = P.Particles(s["mesh"], uniform_count=case["ppc"], seed=s["seed"])
        x, ids = P.advect_differentiable(U, parts, s["dt"], case["rk"], case["steps"], case["tape"])
        loss = (x - s["target"][:, ids]).square().sum()
        loss.backward()
        return {"loss": loss.detach(), "x": x.detach(), "id": ids, "grad": U.grad}
    if kind == "ensemble":
        s["ens"].run(case["rk"], case["steps"])
        got = [s["ens"].export(p) for p in range(case["members"])]
        return {k: torch.cat([g[k] for g in got], dim=-1) for k in ("x", "xhat", "id", "cell")}
    if kind == "odes":
        s["parts"].advect_properties(s["dt"], case["rk"], case["steps"], damage=0, alpha=ALPHA, beta=BETA,
                                     deformation=1)
        return s["parts"].export()
    if kind == "transfers":
        parts = s["parts"]
        return {"mean": parts.average(0), "geometric": parts.average(0, kind=P.PIC_AVG_GEOMETRIC),
                "harmonic": parts.average(0, kind=P.PIC_AVG_HARMONIC), "vertex": parts.vertex_average(0),
                "linear": parts.project_linear(0)}
    w = P.cell_weights(s["mesh"], s["rho"])
    N = s["mesh"].ncells * case["ppc"]
    counts = P.draw_cell_counts(w, N, s["seed"])
    drawn = P.Particles.metropolis_hastings(s["mesh"], counts, s["rho"], case["thinning"], s["seed"] + 1)
    placed, outside = P.Particles.import_points(s["mesh"], s["x"])
    out = {"weights": w, "counts": counts, "outside": outside}
    for name, parts in (("drawn", drawn), ("placed", placed)):
        st = parts.export()
        out[name] = {k: st[k] for k in ("x", "xhat", "id", "cell")}
        parts.close()
    return out


# --------------------------------------------------------------------------- work


def _particles(case):
    if case["kind"] == "ensemble":
        cells = sum(s * s for s in _members(case))
        return cells, cells * case["ppc"] * 1.6  # the log-normal's mean is e^(1/2) medians, less the cut
    cells = math.prod(_n(case))
    return cells, cells * case["ppc"] * (1.6 if case.get("uneven") else 1.0)


def work(case):
    """Each input and output once; per stage the Q2 field's nested Horner form and an inverse map of three Newton steps."""
    kind = case["kind"]
    cells, N = _particles(case)
    d = 2 if kind == "ensemble" else len(_n(case))
    stages, steps = {1: 1, 2: 2, 4: 4}[case.get("rk", 4)], case.get("steps", 1)
    p = case.get("props", 1 + d * d if kind == "odes" else 0)
    state = N * (16 * d + 8 + 4 + 8 * p)
    mesh = 8 * d * cells * (1 + 2 ** d)  # vertices, and 2^d Q2 nodes per cell
    horner = 2 * d * (3 ** d - 1)
    stage = horner + 3 * (8 * d * 2 ** d) + 20 * d
    step = N * stages * stage
    if kind in ("steps", "ensemble"):
        return {"bytes": 2 * state + mesh + 12 * cells * case.get("average", 0) * steps, "flops": step * steps}
    if kind == "coupled":
        return {"bytes": 2 * state + mesh * (2 if case["two"] else 1) + 12 * cells * p, "flops": step * (1.5 if case["two"] else 1)}
    if kind == "adjoint":
        return {"bytes": N * 40 * d + 2 * mesh, "flops": 4 * step * steps}
    if kind == "odes":
        return {"bytes": 2 * state + mesh, "flops": steps * N * stages * (stage + horner * 2 + 8 * d ** 3)}
    if kind == "transfers":
        return {"bytes": N * (8 * d + 8) + cells * (3 * 12 + 16 + 8 * (d + 1) + 4), "flops": N * (20 + 4 * 2 ** d + (d + 1) * (d + 2))}
    chain = case["thinning"] * N * (d * d + 3) * 2 ** d
    return {"bytes": 2 * N * (16 * d + 12) + N * 8 * d + 8 * d * cells + 28 * cells, "flops": chain + N * 6 * 8 * d * 2 ** d}


# --------------------------------------------------------------------------- exact


class _Boxes:
    """One structured mesh, or several one after another, in plain torch: cells are numbered through all of them."""

    def __init__(self, sizes, Xs):
        self.d = len(sizes[0])
        self.X = torch.cat(Xs, dim=1)
        per_cell, v0, q0, self.base = [], 0, 0, [0]
        for n in sizes:
            ijk = _grid_index(n)
            v = v0 + sum(ijk[a] * math.prod(m + 1 for m in n[:a]) for a in range(self.d))
            q = q0 + sum(2 * ijk[a] * math.prod(2 * m + 1 for m in n[:a]) for a in range(self.d))
            C = ijk[0].numel()
            per_cell.append(torch.stack([v, q] + ijk + [torch.full((C,), m, device=DEV) for m in n]))
            v0 += math.prod(m + 1 for m in n)
            q0 += math.prod(2 * m + 1 for m in n)
            self.base.append(self.base[-1] + C)
        self.table = torch.cat(per_cell, dim=1)
        self.C = self.base[-1]

    def cell(self, K):
        t, d = self.table[:, K], self.d
        return t[0], t[1], t[2:2 + d], t[2 + d:2 + 2 * d]

    def corners(self, K):
        v, _, _, n = self.cell(K)
        e = []
        for c in range(1 << self.d):
            o, stride = torch.zeros_like(v), torch.ones_like(v)
            for a in range(self.d):
                o = o + ((c >> a) & 1) * stride
                stride = stride * (n[a] + 1)
            e.append(self.X[:, v + o])
        return e

    def map(self, e, t):
        """Phi(t) - e[0] and its Jacobian J[i][j], from the corners."""
        d = self.d
        phi, J = 0.0, [0.0] * d
        for c in range(1, 1 << d):
            off = e[c] - e[0]
            f = [t[a] if (c >> a) & 1 else 1 - t[a] for a in range(d)]
            phi = phi + off * math.prod(f)
        for c in range(1 << d):
            off = e[c] - e[0]
            f = [t[a] if (c >> a) & 1 else 1 - t[a] for a in range(d)]
            for j in range(d):
                J[j] = J[j] + off * math.prod(f[a] for a in range(d) if a != j) * (1 if (c >> j) & 1 else -1)
        return phi, [[J[j][i] for j in range(d)] for i in range(d)]

    def solve(self, J, r):
        d = self.d
        Ji = self.inverse(J)
        return torch.stack([sum(Ji[i][j] * r[j] for j in range(d)) for i in range(d)])

    def inverse(self, J):
        d = self.d
        if d == 2:
            det = J[0][0] * J[1][1] - J[0][1] * J[1][0]
            return [[J[1][1] / det, -J[0][1] / det], [-J[1][0] / det, J[0][0] / det]]
        c = [[J[(i + 1) % 3][(j + 1) % 3] * J[(i + 2) % 3][(j + 2) % 3] - J[(i + 1) % 3][(j + 2) % 3] * J[(i + 2) % 3][(j + 1) % 3]
              for j in range(3)] for i in range(3)]
        det = sum(J[0][j] * c[0][j] for j in range(3))
        return [[c[j][i] / det for j in range(3)] for i in range(3)]

    def locate(self, y, K, t):
        """Owner cell (lowest index on shared faces; -1: none) and reference coordinates of y, starting in cell K at t."""
        d = self.d
        K, t = K.clone(), t.clone()
        todo = torch.arange(K.numel(), device=DEV)
        for _ in range(6):
            k, yy, tt = K[todo], y[:, todo], t[:, todo]
            e = self.corners(k)
            for it in range(20):
                phi, J = self.map(e, tt)
                step = self.solve(J, (yy - e[0]) - phi)
                tt = tt + step
                if float(step.abs().max()) <= 3e-15 or it >= 6 and float(step.abs().max()) <= 1e-13:
                    break
            _, _, ijk, n = self.cell(k)
            hop, stride, move = 0, 1, torch.zeros_like(tt)
            for a in range(d):
                o = torch.where(tt[a] <= 1e-10, -1, torch.where(tt[a] > 1 + 1e-10, 1, 0))
                o = torch.where((ijk[a] + o < 0) | (ijk[a] + o >= n[a]), 0, o)
                move[a] = o.to(F64)
                hop = hop + o * stride
                stride = stride * n[a]
            t[:, todo] = tt
            going = hop != 0
            if not bool(going.any()):
                break
            left = todo[going]
            K[left] = (k + hop)[going]
            t[:, left] = (tt - move)[:, going]
            todo = left
        lost = ((t < -1e-10) | (t > 1 + 1e-10)).any(0)
        return torch.where(lost, -1, K), t

    def basis(self, t):
        return [[(1 - x) * (1 - 2 * x), 4 * x * (1 - x), x * (2 * x - 1)] for x in t]

    def nodes(self, K):
        """The cell's Q2 nodes with the basis index of each along every axis."""
        _, q, _, n = self.cell(K)
        for o in range(3 ** self.d):
            i, off, stride = o, torch.zeros_like(q), torch.ones_like(q)
            idx = []
            for a in range(self.d):
                idx.append(i % 3)
                off = off + (i % 3) * stride
                stride = stride * (2 * n[a] + 1)
                i //= 3
            yield q + off, idx

    def velocity(self, U, K, t):
        b, u = self.basis(t), 0.0
        for node, idx in self.nodes(K):
            u = u + U[:, node] * math.prod(b[a][i] for a, i in enumerate(idx))
        return u

    def gradient(self, U, K, t):
        """G[i][j] = d u_i / d x_j with the cell held fixed."""
        d, b = self.d, self.basis(t)
        db = [[4 * x - 3, 4 - 8 * x, 4 * x - 1] for x in t]
        g = [0.0] * d
        for node, idx in self.nodes(K):
            v = U[:, node]
            for j in range(d):
                g[j] = g[j] + v * math.prod(db[a][i] if a == j else b[a][i] for a, i in enumerate(idx))
        Ji = self.inverse(self.map(self.corners(K), t)[1])
        return [[sum(g[k][i] * Ji[k][j] for k in range(d)) for j in range(d)] for i in range(d)]


_TABLEAU = {1: ([], [1.0]), 2: ([0.5], [0.0, 1.0]), 4: ([0.5, 0.5, 1.0], [1 / 6, 1 / 3, 1 / 3, 1 / 6])}


def _splitmix(seed, index):
    """Output `index` of SplitMix64 seeded with `seed`, top 53 bits as a number in [0, 1)."""
    def wrap(v):
        v %= 1 << 64
        return v - (1 << 64) if v >> 63 else v

    def shift(z, k):
        return (z >> k) & ((1 << (64 - k)) - 1)

    z = (index + 1) * wrap(0x9E3779B97F4A7C15) + wrap(seed)
    z = (z ^ shift(z, 30)) * wrap(0xBF58476D1CE4E5B9)
    z = (z ^ shift(z, 27)) * wrap(0x94D049BB133111EB)
    return shift(z ^ shift(z, 31), 11).to(F64) * 2.0 ** -53


class _Tracers:
    """Particles in id order: x, reference coordinates t, cell K (-1: lost), properties."""

    def __init__(self, boxes, cells, seeds):
        """cells: the cell of every particle, per member; seeds: the generator seed of each member."""
        self.B = boxes
        t = [torch.stack([_splitmix(s, torch.arange(k.numel(), device=DEV) * boxes.d + a) for a in range(boxes.d)])
             for k, s in zip(cells, seeds)]
        self.t, self.K = torch.cat(t, dim=1), torch.cat(cells)
        self.id = torch.cat([torch.arange(k.numel(), device=DEV) for k in cells])
        self.x = torch.empty_like(self.t)
        for c in self.chunks(self.K.numel()):
            e = boxes.corners(self.K[c])
            self.x[:, c] = e[0] + boxes.map(e, self.t[:, c])[0]
        self.props = None

    @staticmethod
    def chunks(n, size=1 << 21):
        return [slice(i, min(n, i + size)) for i in range(0, n, size)]

    def step(self, U, dt, rk, U_next=None, odes=False, record=None):
        for c in self.chunks(self.K.numel()):
            alive = torch.nonzero(self.K[c] >= 0).flatten() + c.start
            self._step(U, dt if not torch.is_tensor(dt) else dt[alive], rk, alive, U_next, odes, record)

    def _step(self, U, dt, rk, at, U_next, odes, record):
        B, (nodes, weights) = self.B, _TABLEAU[rk]
        x, K, t = self.x[:, at], self.K[at], self.t[:, at]
        z = self.props[:, at] if odes else None
        sum_k, sum_z, kz = 0.0, 0.0, None
        ok = torch.ones_like(K, dtype=torch.bool)
        stages = []
        for s, w in enumerate(weights):
            if s:
                K2, t2 = B.locate(x + nodes[s - 1] * k, K, t)
                ok &= K2 >= 0
                K, t = torch.where(ok, K2, K), torch.where(ok, t2, t)
            stages.append((K, t))
            theta = 0.0 if s == 0 else nodes[s - 1]
            u = B.velocity(U, K, t) if U_next is None or theta < 1 else 0.0
            if U_next is not None and theta > 0:
                u = (1 - theta) * u + theta * B.velocity(U_next, K, t)
            k = dt * u
            sum_k = sum_k + w * k
            if odes:
                zs = z if s == 0 else z + nodes[s - 1] * kz
                kz = dt * _ode(B.gradient(U, K, t), zs, B.d)
                sum_z = sum_z + w * kz
        x = x + sum_k
        K2, t2 = B.locate(x, K, t)
        ok &= K2 >= 0
        self.x[:, at], self.t[:, at], self.K[at] = x, t2, torch.where(ok, K2, -1)
        if odes:
            self.props[:, at] = z + sum_z
        if record is not None:
            record.append((at, ok, stages))

    def order(self):
        alive = torch.nonzero(self.K >= 0).flatten()
        return alive[torch.argsort(self.K[alive] * (int(self.id.max()) + 1) + self.id[alive])]

    def store(self):
        o = self.order()
        out = {"x": self.x[:, o], "xhat": self.t[:, o], "id": self.id[o], "cell": self.K[o].to(torch.int32)}
        if self.props is not None:
            out["props"] = self.props[:, o]
        return out

    def sums(self, v):
        alive = self.K >= 0
        n = torch.bincount(self.K[alive], minlength=self.B.C)
        return torch.bincount(self.K[alive], weights=v[alive], minlength=self.B.C), n

    def mean(self, q):
        s, n = self.sums(self.props[q])
        return torch.where(n > 0, s / n, 0.0), n.to(torch.int32)


def _ode(G, z, d):
    """d/dt of (damage, deformation gradient row by row)."""
    strain = sum((0.5 * (G[i][j] + G[j][i])).square() for i in range(d) for j in range(d)).sqrt()
    F = [[sum(G[i][k] * z[1 + k * d + j] for k in range(d)) for j in range(d)] for i in range(d)]
    return torch.stack([ALPHA * strain - BETA * z[0]] + [F[i][j] for i in range(d) for j in range(d)])


def _cells_of(case, ncells, seed):
    if case.get("uneven") or case["kind"] == "ensemble":
        n = _counts(ncells, case["ppc"], seed).long()
    else:
        n = torch.full((ncells,), case["ppc"], device=DEV)
    return torch.repeat_interleave(torch.arange(ncells, device=DEV), n)


def exact(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        sides = _members(case)
        Xs = [_vertices((s, s), seed * 131 + p) for p, s in enumerate(sides)]
        U = torch.cat([_field((s, s), X, seed * 131 + p) for p, (s, X) in enumerate(zip(sides, Xs))], dim=1)
        B = _Boxes([(s, s) for s in sides], Xs)
        cells = [_cells_of(case, s * s, seed * 131 + p) + B.base[p] for p, s in enumerate(sides)]
        T = _Tracers(B, cells, [_pseed(seed, p) for p in range(len(sides))])
        member = torch.cat([torch.full((k.numel(),), p, device=DEV) for p, k in enumerate(cells)])
        dt = torch.tensor([_dt((s, s), X) for s, X in zip(sides, Xs)], dtype=F64, device=DEV)[member]
        for _ in range(case["steps"]):
            T.step(U, dt, case["rk"])
        out, o = T.store(), T.order()
        out["cell"] = (T.K[o] - torch.tensor(B.base, device=DEV)[member[o]]).to(torch.int32)
        return out
    n = _n(case)
    X = _vertices(n, seed)
    B = _Boxes([n], [X])
    if kind == "generate":
        return _exact_generate(case, seed, n, X, B)
    U, dt = _field(n, X, seed), _dt(n, X)
    T = _Tracers(B, [_cells_of(case, B.C, seed)], [_pseed(seed)])
    if kind == "adjoint":
        return _exact_adjoint(case, seed, B, U, dt, T)
    if kind == "odes":
        d = len(n)
        z = [0.1] + [float(q % (d + 1) == 0) for q in range(d * d)]
        T.props = torch.tensor(z, dtype=F64, device=DEV)[:, None].repeat(1, T.K.numel())
        for _ in range(case["steps"]):
            T.step(U, dt, case["rk"], odes=True)
        return T.store()
    q = case.get("props", 1)
    T.props = torch.stack([T.x[i] if i < len(n) else torch.cos(3 * T.x[0]) + 2.0 for i in range(q)])
    if kind == "transfers":
        return _exact_transfers(T, n)
    avg = []
    if kind == "coupled":
        T.step(U, dt, case["rk"], U_next=_field(n, X, seed, 20) if case["two"] else None)
        avg = [T.mean(i) for i in range(q)]
    else:
        for _ in range(case["steps"]):
            T.step(U, dt, case["rk"])
            if case["average"]:
                avg.append(T.mean(0))
    return {"average": avg, "store": T.store()}


def _exact_transfers(T, n):
    v, d, B = T.props[0], len(n), T.B
    mean = T.mean(0)
    cnt = mean[1]
    some = cnt > 0
    geometric = torch.where(some, (T.sums(v.log())[0] / cnt).exp(), 0.0)
    harmonic = torch.where(some, cnt / T.sums(1 / v)[0], 0.0)
    num = torch.zeros(B.X.shape[1], dtype=F64, device=DEV)
    den = torch.zeros_like(num)
    v0, _, _, m = B.cell(T.K)
    for c in range(1 << d):
        o, stride, w = torch.zeros_like(v0), torch.ones_like(v0), 1.0
        for a in range(d):
            hi = (c >> a) & 1
            o, stride, w = o + hi * stride, stride * (m[a] + 1), w * (T.t[a] if hi else 1 - T.t[a])
        num.index_add_(0, v0 + o, w * v)
        den.index_add_(0, v0 + o, w)
    rows = [torch.ones_like(v)] + [T.t[a] - 0.5 for a in range(d)]
    A = torch.stack([torch.stack([T.sums(r * q)[0] for q in rows], -1) for r in rows], -2)
    rhs = torch.stack([T.sums(r * v)[0] for r in rows], -1)
    fit = cnt > d
    A = torch.where(fit[:, None, None], A, torch.eye(d + 1, dtype=F64, device=DEV))
    c = torch.linalg.solve(A, rhs).T.contiguous()
    flat = torch.zeros_like(c)
    flat[0] = mean[0]
    return {"mean": mean, "geometric": (geometric, cnt), "harmonic": (harmonic, cnt),
            "vertex": (torch.where(den > 0, num / den, 0.0), den), "linear": (torch.where(fit, c, flat), cnt)}


def _exact_adjoint(case, seed, B, U, dt, T):
    nodes, weights = _TABLEAU[case["rk"]]
    d, tape = B.d, []
    for _ in range(case["steps"]):
        record = []
        T.step(U, dt, case["rk"], record=record)
        tape.append(record)
    o = T.order()
    target = _rand(seed, 5, d, T.K.numel())
    diff = T.x[:, o] - target[:, o]
    lam = torch.zeros_like(T.x)
    lam[:, o] = 2 * diff
    grad = torch.zeros_like(U)
    for record in reversed(tape):
        for at, ok, stages in record:
            l = torch.where(ok, lam[:, at], 0.0)
            total, ly = l, 0.0
            for s in reversed(range(len(weights))):
                K, t = stages[s]
                lk = weights[s] * l + (nodes[s] * ly if s < len(nodes) else 0.0)
                G = B.gradient(U, K, t)
                ly = dt * torch.stack([sum(G[c][q] * lk[c] for c in range(d)) for q in range(d)])
                total = total + ly
                b = B.basis(t)
                for node, idx in B.nodes(K):
                    grad.index_add_(1, node, dt * lk * math.prod(b[a][i] for a, i in enumerate(idx)))
            lam[:, at] = total
    return {"loss": diff.square().sum(), "x": T.x[:, o], "id": T.id[o], "grad": grad}


def _exact_generate(case, seed, n, X, B):
    rho, K = _density(n, X), torch.arange(B.C, device=DEV)
    e, d, w = B.corners(K), B.d, 0.0
    v0, _, _, m = B.cell(K)
    for q in range(1 << d):
        t = [torch.full((B.C,), 0.5 + (0.5 if (q >> a) & 1 else -0.5) / math.sqrt(3.0), dtype=F64, device=DEV) for a in range(d)]
        J = B.map(e, t)[1]
        det = J[0][0] * J[1][1] - J[0][1] * J[1][0] if d == 2 else sum(
            J[0][j] * (J[1][(j + 1) % 3] * J[2][(j + 2) % 3] - J[1][(j + 2) % 3] * J[2][(j + 1) % 3]) for j in range(3))
        r = 0.0
        for c in range(1 << d):
            o, stride, f = torch.zeros_like(v0), torch.ones_like(v0), 1.0
            for a in range(d):
                hi = (c >> a) & 1
                o, stride, f = o + hi * stride, stride * (m[a] + 1), f * (t[a] if hi else 1 - t[a])
            r = r + rho[v0 + o] * f
        w = w + r * det.abs() / (1 << d)
    x = _import_points(case, seed)
    inside = ((x >= 0) & (x <= 1)).all(0)
    x = x[:, inside]
    ijk = [(x[a] * m_).floor().clamp(0, m_ - 1).long() for a, m_ in enumerate(n)]
    start = sum(ijk[a] * math.prod(n[:a]) for a in range(d))
    K, t = torch.empty_like(start), torch.empty_like(x)
    for c in _Tracers.chunks(start.numel()):
        K[c], t[:, c] = B.locate(x[:, c], start[c], torch.full_like(x[:, c], 0.5))
    o = torch.argsort(K * K.numel() + torch.arange(K.numel(), device=DEV))
    placed = {"x": x[:, o], "xhat": t[:, o], "id": o, "cell": K[o].to(torch.int32)}
    return {"weights": w, "counts": None, "outside": int((~inside).sum()), "drawn": {k: None for k in ("x", "xhat", "id", "cell")},
            "placed": placed}
