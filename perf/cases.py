"""Performance cases of the CTENO / CTENOZ solver: what a user's program has it do.

A pass takes a program's cell means to the solver, advances them by some Runge-Kutta steps and
reads the new cell means back, through the public entry points of paper_2312_17042_gb300.native.
The mesh, its stencils and least-squares operators (``Solver``) are what such a program keeps from
pass to pass. The flows are those of the paper's experiments, at sizes from the smallest test mesh
to the largest that is quick to set up: order tests on a periodic wave, the Sod tube, the triple
point, the double Mach reflection, a 3D blast, and batches of small Riemann problems.

A case's plain values:
  flow       wave2 | tube | triple | dmr | quadrants | wave3 | blast
  nx, ny     squares (2D) along x and y, two triangles each; 3D: nx cubes a side, six tetrahedra each
  meshes     number of meshes of a batch (quadrants; sides log-uniform from nx to ny)
  degree, scheme (0 CTENO, 1 CTENOZ, 2 CWENO, 3 TENO), mixed (False: FP64), rk, characteristic
  steps      Runge-Kutta steps of a pass
  io         device (the state lives in device tensors) | host (pinned host buffers)
  loop       run (the captured step) | stages (the program's own loop over the stages)
  tuned      True: the program calls cteno_autotune once, as for a long run
"""
import math

import numpy as np
import torch

from paper_2312_17042_gb300 import native

GAMMA = 1.4
CFL = {"wave2": 0.5, "tube": 0.4, "triple": 0.4, "dmr": 0.4, "quadrants": 0.4, "wave3": 0.5, "blast": 0.3}
BOX = {"wave2": (1.0, 1.0), "tube": (1.0, 0.25), "triple": (7.0, 3.0), "dmr": (4.0, 1.0), "quadrants": (1.0, 1.0)}
POST = (8.0, 8.25 * math.cos(math.pi / 6), -8.25 * math.sin(math.pi / 6), 116.5)
PRE = (1.4, 0.0, 0.0, 1.0)


def _case(name, flow, nx, ny=0, **kw):
    c = dict(name=name, flow=flow, nx=nx, ny=ny or nx, meshes=1, degree=2, scheme=0, mixed=False, rk=3,
             characteristic=False, steps=5, io="device", loop="run", tuned=False)
    c.update(kw)
    return c


def listed():
    return [
        # the order test on its smallest mesh, as a first script or a unit test runs it: latency
        _case("wave 32^2 r2 fp64", "wave2", 32, steps=10),
        # a program's own loop over the stages, classical RK4, high order, walls: a small study
        _case("triple 70x30 r5 rk4 fp64", "triple", 70, 30, degree=5, rk=4, steps=3, loop="stages"),
        # the Sod tube of the paper's comparison, third order, a long mixed run
        _case("tube 512x128 r2 mixed", "tube", 512, 128, mixed=True, steps=10, tuned=True),
        # the same in FP64 at fourth order, run as a script does, with the solver's defaults
        _case("tube 512x128 r3 fp64", "tube", 512, 128, degree=3, scheme=1),
        # the same in characteristic variables (the paper's setting for strong shocks)
        _case("tube 512x128 char mixed", "tube", 512, 128, mixed=True, characteristic=True, tuned=True),
        # a parameter study: a batch of ragged small meshes per launch
        _case("quadrants x32 r2 mixed", "quadrants", 16, 256, meshes=32, scheme=1, mixed=True, steps=10, tuned=True),
        # the paper's triple point, fifth order, walls
        _case("triple 500x215 r4 mixed", "triple", 500, 215, degree=4, scheme=1, mixed=True, tuned=True),
        # double Mach reflection, seventh order, inflow, wall and moving-shock boundaries
        _case("dmr 600x150 r6 mixed", "dmr", 600, 150, degree=6, mixed=True, steps=3, tuned=True),
        # the 3D order test, third order
        _case("wave 32^3 r2 mixed", "wave3", 32, mixed=True, tuned=True),
        # the 3D blast in FP64: a reference solution on a coarse mesh, solver defaults
        _case("blast 16^3 r3 fp64", "blast", 16, degree=3, steps=2),
        # the 3D blast coupled to a host program: the state comes from and goes to pinned memory
        # around every step
        _case("blast 31^3 r3 mixed host", "blast", 31, degree=3, mixed=True, steps=1, io="host", tuned=True),
        # the 3D blast, fourth order: the production run
        _case("blast 48^3 r3 mixed", "blast", 48, degree=3, mixed=True, steps=2, tuned=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: any flow, odd sizes, every degree, weighting and option."""
    while True:
        flow = rng.choice(list(CFL))
        d = _dim({"flow": flow})
        c = _case("", flow, 1, mixed=rng.random() < 0.6, scheme=rng.choice([0, 0, 1, 1, 2, 3]),
                  rk=rng.choice([3, 3, 3, 4]), steps=rng.randint(1, 10), io=rng.choice(["device"] * 4 + ["host"]),
                  loop=rng.choice(["run"] * 4 + ["stages"]), tuned=rng.random() < 0.5)
        del c["name"]
        if d == 3:
            c["degree"] = rng.choice([2, 3])
            c["nx"] = c["ny"] = _log(rng, 8, 48)
        else:
            c["degree"] = rng.choice([2, 2, 3, 3, 4, 5, 6])
            c["ny"] = _log(rng, 24, 300)
            c["nx"] = {"tube": 4, "dmr": 4}.get(flow, 1) * c["ny"] + (rng.randint(0, 40) if flow == "triple" else 0)
            if flow == "quadrants":
                c["meshes"], c["nx"], c["ny"] = rng.randint(2, 32), rng.randint(24, 40), rng.randint(60, 256)
        c["characteristic"] = rng.random() < 0.15
        w, most = work(c), work(listed()[-1])
        slow = 1 if c["mixed"] else 12  # the FP64 rate of this GPU against its FP32 rate and memory
        if c["characteristic"]:
            slow *= 4
        if w["bytes"] * slow <= most["bytes"] and w["flops"] * slow <= 4 * most["flops"] and _cells(c) <= 700000:
            return c


# ---- sizes ---------------------------------------------------------------------------------------
def _dim(case):
    return 3 if case["flow"] in ("wave3", "blast") else 2


def _sides(case):
    """Squares along a side of each mesh of a batch: log-uniform quantiles, the same for every seed."""
    m, lo, hi = case["meshes"], math.log(case["nx"]), math.log(case["ny"])
    return [int(round(math.exp(lo + (hi - lo) * (k + 0.5) / m))) for k in range(m)]


def _cells(case):
    if case["flow"] == "quadrants":
        return sum(2 * n * n for n in _sides(case))
    return 6 * case["nx"] ** 3 if _dim(case) == 3 else 2 * case["nx"] * case["ny"]


def _shape(case):
    d, r = _dim(case), case["degree"]
    nk = math.comb(r + d, d) - 1
    kd = 5 if r >= 4 else d
    nq = 4 if d == 3 else max(2, (r + 2) // 2)
    return d, nk, 2 * (nk + 1), kd, nq


def work(case):
    """Every stage streams each cell's least-squares operators, stencil ids, state and geometry once
    and writes the new state; the operations are the products with the operators, the smoothness
    indicators, the weights, the face values and the face fluxes (HLLC about 90 + 20 d a point)."""
    d, nk, M, kd, nq = _shape(case)
    n, nv, nf, s = _cells(case), d + 2, d + 1, 4 if case["mixed"] else 8
    stages = case["steps"] * case["rk"]
    cell = (M * nk + nf * 2 * kd * kd) * s + 4 * M + nf * (4 + 4 * s) + 8 * nv * 3
    var = 2 * nk * M + nf * 2 * kd * 2 * kd + nk * (nk + 1) + 2 * nk + 30 * (nf + 1) + 2 * nf * nq * nk
    if case["characteristic"]:
        var += (nf - 1) * (nk * (nk + 1) + 2 * nk + 30 * (nf + 1)) + nf * 2 * nv * (nk + nf * kd + nq)
    ops = nv * var + nf * nq // 2 * (90 + 20 * d)
    return {"bytes": stages * n * cell + 2 * 8 * nv * n, "flops": stages * n * ops}


# ---- inputs --------------------------------------------------------------------------------------
class Mesh:
    def __init__(self, xyz, cells, period):
        self.xyz, self.cells, self.period = xyz, cells, period


def _tri(nx, ny, box, periodic, rng):
    hx, hy = box[0] / nx, box[1] / ny
    vx, vy = (nx, ny) if periodic else (nx + 1, ny + 1)
    i, j = (a.ravel() for a in np.meshgrid(np.arange(vx), np.arange(vy), indexing="ij"))
    xyz = np.stack([i * hx, j * hy], 1)
    inner = (i > 0) & (i < nx) & (j > 0) & (j < ny)
    xyz[inner] += 0.1 * np.array([hx, hy]) * rng.uniform(-1, 1, (int(inner.sum()), 2))
    si, sj = (a.ravel() for a in np.meshgrid(np.arange(nx), np.arange(ny), indexing="ij"))

    def vid(a, b):
        return (a % vx) * vy + b % vy
    v00, v10, v11, v01 = vid(si, sj), vid(si + 1, sj), vid(si + 1, sj + 1), vid(si, sj + 1)
    diag = rng.integers(0, 2, si.size)[:, None] == 0
    cells = np.empty((2 * si.size, 3), np.int32)
    cells[0::2] = np.where(diag, np.stack([v00, v10, v11], 1), np.stack([v00, v10, v01], 1))
    cells[1::2] = np.where(diag, np.stack([v00, v11, v01], 1), np.stack([v10, v11, v01], 1))
    return Mesh(xyz, cells, np.array(box if periodic else (0.0, 0.0), float))


def _tet(n, periodic, rng):
    v = n if periodic else n + 1
    g = np.stack([a.ravel() for a in np.meshgrid(*[np.arange(v)] * 3, indexing="ij")], 1)
    xyz = g / n
    inner = ((g > 0) & (g < n)).all(1)
    xyz[inner] += 0.08 / n * rng.uniform(-1, 1, (int(inner.sum()), 3))
    base = np.stack([a.ravel() for a in np.meshgrid(*[np.arange(n)] * 3, indexing="ij")], 1)
    cells = np.empty((6 * len(base), 4), np.int32)
    for t, perm in enumerate([(0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)]):
        p = base.copy()
        for k in range(4):
            if k:
                p[:, perm[k - 1]] += 1
            q = p % v
            cells[t::6, k] = (q[:, 0] * v + q[:, 1]) * v + q[:, 2]
    return Mesh(xyz, cells, np.full(3, 1.0 if periodic else 0.0))


def _corners(mesh):
    """[cells, d+1, d] vertices, periodic images next to vertex 0."""
    v = mesh.xyz[mesh.cells]
    per = mesh.period
    if (per > 0).any():
        v = v - per * np.round((v - v[:, :1]) / per)
    return v


def _means(mesh, prim):
    """Cell means [nv, cells] of a primitive field by the centroid and points towards the vertices."""
    v = _corners(mesh)
    d = v.shape[2]
    c = v.mean(1)
    out = 0.0
    for k in range(d + 2):
        q = prim(c if k == d + 1 else 0.5 * (c + v[:, k]))
        rho, vel, p = q[0], q[1:-1], q[-1]
        out = out + np.concatenate([rho[None], rho * vel, (p / (GAMMA - 1) + 0.5 * rho * (vel * vel).sum(0))[None]])
    return out / (d + 2)


def _field(case, rng):
    """Primitive field x [n, d] -> [nv, n] of a flow."""
    flow, d = case["flow"], _dim(case)

    def make(x, rho, vel, p):
        q = np.empty((d + 2, len(x)))
        q[0], q[-1] = rho, p
        for k in range(d):
            q[1 + k] = vel[k] if isinstance(vel, (list, tuple)) else vel
        return q
    if flow in ("wave2", "wave3"):
        return lambda x: make(x, 1 + 0.2 * np.sin(2 * np.pi * x.sum(1)), 1.0, 1.0)
    if flow == "tube":
        return lambda x: make(x, np.where(x[:, 0] < 0.5, 1, 0.125), 0.0, np.where(x[:, 0] < 0.5, 1, 0.1))
    if flow == "triple":
        return lambda x: make(x, np.where((x[:, 0] > 1) & (x[:, 1] > 1.5), 0.125, 1.0), 0.0,
                              np.where(x[:, 0] <= 1, 1.0, 0.1))
    if flow == "blast":
        return lambda x: make(x, 1.0, 0.0, np.where(((x - 0.5) ** 2).sum(1) < 0.04, 10.0, 0.1))
    if flow == "dmr":
        def f(x):
            post = x[:, 1] >= math.sqrt(3) * (x[:, 0] - 1 / 6)
            return np.where(post, np.array(POST)[:, None], np.array(PRE)[:, None])
        return f
    st = np.concatenate([rng.uniform(0.1, 2, (1, 4)), rng.uniform(-1, 1, (2, 4)), rng.uniform(0.1, 2, (1, 4))])
    return lambda x: st[:, (x[:, 0] >= 0.5) + 2 * (x[:, 1] >= 0.5)]


def _inputs(case, seed):
    """The meshes and their initial cell means [nv, cells]."""
    rng = np.random.default_rng(seed)
    flow = case["flow"]
    if flow == "quadrants":
        meshes = [_tri(n, n, BOX[flow], False, rng) for n in _sides(case)]
    elif _dim(case) == 3:
        meshes = [_tet(case["nx"], flow == "wave3", rng)]
    else:
        meshes = [_tri(case["nx"], case["ny"], BOX[flow], flow == "wave2", rng)]
    return meshes, [_means(m, _field(case, rng)) for m in meshes]


def _conserved(q):
    return np.array([q[0], q[0] * q[1], q[0] * q[2], q[3] / (GAMMA - 1) + 0.5 * q[0] * (q[1] ** 2 + q[2] ** 2)])


def prepare(case, seed):
    meshes, U0 = _inputs(case, seed)
    kw = dict(cfl=CFL[case["flow"]], rk=case["rk"], characteristic=int(case["characteristic"]))
    if case["flow"] == "triple":
        kw.update(boundary=native.CTENO_BOUNDARY_WALL, lambda1p=1e4)
    if case["flow"] == "dmr":
        tiny = 1e-9
        kw["regions"] = [((-1.0, -1.0), (tiny, 2.0), native.CTENO_BOUNDARY_STATE_A),
                         ((-1.0, -1.0), (1 / 6, tiny), native.CTENO_BOUNDARY_STATE_A),
                         ((1 / 6, -1.0), (5.0, tiny), native.CTENO_BOUNDARY_WALL),
                         ((-1.0, 1 - tiny), (5.0, 2.0), native.CTENO_BOUNDARY_SHOCK_AB)]
        kw["states"] = (_conserved(POST), _conserved(PRE), 1 / 6, 1 / math.sqrt(3), 20 / math.sqrt(3))
    s = native.Solver(meshes, _dim(case), degree=case["degree"], scheme=case["scheme"],
                      precision=native.CTENO_MIXED if case["mixed"] else native.CTENO_FP64,
                      stream=torch.cuda.current_stream().cuda_stream, **kw)
    U = torch.from_numpy(np.concatenate([u.ravel() for u in U0]))
    if case["io"] == "host":
        U = U.pin_memory()
        out = torch.empty_like(U).pin_memory()
    else:
        U = U.cuda()
        out = torch.empty_like(U)
    if case["tuned"]:
        native.cteno_set_state_all(s.ctx, *_arg(U))
        native.cteno_autotune(s.ctx)
    return {"case": case, "solver": s, "U": U, "out": out}


def _arg(t):
    return (t.data_ptr(), True) if t.is_cuda else (t.numpy(),)


def run(state):
    case, s = state["case"], state["solver"]
    native.cteno_set_state_all(s.ctx, *_arg(state["U"]))
    if case["flow"] == "dmr":
        native.cteno_set_time(s.ctx, 0.0)
    if case["loop"] == "run":
        s.run(case["steps"])
    else:
        for _ in range(case["steps"]):
            s.step()
    native.cteno_get_state_all(s.ctx, *_arg(state["out"]))
    return state["out"]


# ---- the same pass in 64 bits, in plain numpy ----------------------------------------------------
# Conserved variables, periodic, transmissive and wall boundaries; None where it would take long
# (many cells) and for the flows it leaves out (moving shock, characteristic variables).
def exact(case, seed):
    d, nk, M, kd, nq = _shape(case)
    cost = _cells(case) * (M * M * nk / 2e4 + case["steps"] * case["rk"] * nk * M / 700)
    if case["flow"] == "dmr" or case["characteristic"] or cost > 200000:
        return None
    meshes, U0 = _inputs(case, seed)
    return np.concatenate([_advance(case, m, u.T.copy()).T.ravel() for m, u in zip(meshes, U0)])


def _powers(d, r):
    return np.array([e for t in range(1, r + 1) for e in np.ndindex(*[t + 1] * d) if sum(e) == t])


def _simplex_integral(e):
    """Integral of x^e over the unit simplex."""
    return math.prod(math.factorial(k) for k in e) / math.factorial(sum(e) + len(e))


def _basis(x, ex):
    powers = [np.ones_like(x), x]
    while len(powers) <= ex.max():
        powers.append(powers[-1] * x)
    powers = [[np.ascontiguousarray(p[..., j]) for j in range(x.shape[-1])] for p in powers]
    return np.stack([math.prod(powers[p][j] for j, p in enumerate(e) if p) for e in ex])


def _smoothness(ex, d):
    """Sum over 1 <= |alpha| <= degree of the integrals of D^alpha x^i D^alpha x^j."""
    O = np.zeros((len(ex),) * 2)
    for i, p in enumerate(ex):
        for j, q in enumerate(ex):
            for al in ex:
                if (al <= p).all() and (al <= q).all():
                    c = math.prod(math.perm(int(a), int(b)) for a, b in zip(list(p) + list(q), list(al) * 2))
                    O[i, j] += c * _simplex_integral([int(t) for t in p + q - 2 * al])
    return O


def _rule(d, n):
    """Collapsed Gauss-Legendre points of the unit simplex and weights (sum 1 / d!)."""
    g, w = np.polynomial.legendre.leggauss(n)
    g, w = (g + 1) / 2, w / 2
    if d == 2:
        u, v = (a.ravel() for a in np.meshgrid(g, g, indexing="ij"))
        return np.stack([u, v * (1 - u)], 1), (w[:, None] * w).ravel() * (1 - u)
    u, v, t = (a.ravel() for a in np.meshgrid(g, g, g, indexing="ij"))
    return (np.stack([u, v * (1 - u), t * (1 - u) * (1 - v)], 1),
            (w[:, None, None] * w[:, None] * w).ravel() * (1 - u) ** 2 * (1 - v))


def _face_rule(d, nq):
    """Barycentric points on a face (its vertices sorted by global id) and weights (sum 1)."""
    if d == 2:
        g, w = np.polynomial.legendre.leggauss(nq)
        g = (g + 1) / 2
        return np.stack([1 - g, g], 1), w / 2
    g = (np.polynomial.legendre.leggauss(2)[0] + 1) / 2
    x = (4 - np.array([1, -1]) * math.sqrt(6)) / 10  # Gauss points of the weight 1 - u on [0, 1]
    w = np.array([(1 / 6 - 0.5 * x[1]) / (x[0] - x[1]), (1 / 6 - 0.5 * x[0]) / (x[1] - x[0])])
    u, v = (a.ravel() for a in np.meshgrid(x, g, indexing="ij"))
    return np.stack([(1 - u) * (1 - v), u, (1 - u) * v], 1), np.repeat(w, 2)


def _connect(cells):
    """Neighbour cell of each local face (-1: boundary), and the faces' vertices sorted by id."""
    n, nvc = cells.shape
    fv = np.sort(np.stack([np.delete(cells, f, 1) for f in range(nvc)], 1), axis=2)
    key = np.zeros(n * nvc, np.int64)
    for k in range(nvc - 1):
        key = key * (int(cells.max()) + 1) + fv.reshape(n * nvc, -1)[:, k]
    order = np.argsort(key, kind="stable")
    same = key[order][1:] == key[order][:-1]
    nb = np.full(n * nvc, -1)
    a, b = order[:-1][same], order[1:][same]
    nb[a], nb[b] = b, a
    return nb.reshape(n, nvc)  # the neighbour's (cell, face) as cell * nvc + face


def _stencils(cells, cen, per, M):
    """The M nearest cells among the vertex-adjacency layers that hold at least M."""
    n, nvc = cells.shape
    flat = cells.ravel()
    order = np.argsort(flat, kind="stable")
    count = np.bincount(flat)
    start = np.concatenate([[0], np.cumsum(count)])
    v2c = np.full((len(count), count.max()), -1)
    pos = np.arange(len(flat)) - start[flat[order]]
    v2c[flat[order], pos] = order // nvc
    out = np.empty((n, M), np.int64)
    shift = np.where(per > 0, per, 1.0)

    def offsets(ids, c):
        dx = cen[ids] - cen[c][:, None]
        s = np.where(per > 0, -per * np.trunc(dx / shift + np.copysign(0.5, dx)), 0.0)
        return (cen[ids] + s) - cen[c][:, None]
    for c0 in range(0, n, 4096):
        todo = np.arange(c0, min(n, c0 + 4096))
        found = todo[:, None]
        while len(todo):
            more = np.where(found[:, :, None] >= 0, v2c[cells[found]].reshape(len(todo), found.shape[1], -1), -1)
            more = np.sort(np.concatenate([found, more.reshape(len(todo), -1)], 1), axis=1)
            more[:, 1:][more[:, 1:] == more[:, :-1]] = -1
            more = -np.sort(-more, axis=1)
            found = more[:, :int((more >= 0).sum(1).max())]
            enough = (found >= 0).sum(1) > M
            ids, c = found[enough], todo[enough]
            if len(c):
                off = offsets(np.maximum(ids, 0), c)
                d2 = off[..., 0] * off[..., 0]
                for k in range(1, off.shape[2]):
                    d2 = d2 + off[..., k] * off[..., k]
                d2 = np.where((ids < 0) | (ids == c[:, None]), np.inf, d2)
                near = np.lexsort((ids, d2), axis=1)[:, :M]
                out[c] = np.take_along_axis(ids, near, 1)
            found, todo = found[~enough], todo[~enough]
    return out, offsets(out, np.arange(n))


def _pinv(A, rows):
    """Least-squares inverses of A [n, m, k] whose rows beyond `rows` are zero, and full rank."""
    q, r = np.linalg.qr(A)
    dg = np.abs(np.einsum("nkk->nk", r))
    ok = (rows >= A.shape[2]) & (dg.min(1) > 1e-10 * np.maximum(dg.max(1), 1e-300))
    eye = np.eye(A.shape[2])
    return np.where(ok[:, None, None], np.linalg.solve(np.where(ok[:, None, None], r, eye), q.swapaxes(1, 2)), 0.0), ok


def _flux(uL, uR, n):
    """HLLC flux along unit normals n [..., d] between states [..., nv]."""
    def parts(u):
        r, m, E = u[..., 0], u[..., 1:-1], u[..., -1]
        v = m / r[..., None]
        un, p = (v * n).sum(-1), (GAMMA - 1) * (E - 0.5 * (m * v).sum(-1))
        F = np.concatenate([(r * un)[..., None], m * un[..., None] + p[..., None] * n, ((E + p) * un)[..., None]], -1)
        return r, v, un, p, E, np.sqrt(GAMMA * p / r), F
    rL, vL, unL, pL, EL, cL, FL = parts(uL)
    rR, vR, unR, pR, ER, cR, FR = parts(uR)
    D = np.sqrt(rR / rL)
    vt = (vL + vR * D[..., None]) / (1 + D)[..., None]
    Ht = ((EL + pL) / rL + (ER + pR) / rR * D) / (1 + D)
    ct, ut = np.sqrt((GAMMA - 1) * (Ht - 0.5 * (vt * vt).sum(-1))), (vt * n).sum(-1)
    SL, SR = np.minimum(unL - cL, ut - ct), np.maximum(unR + cR, ut + ct)
    SM = (rR * unR * (SR - unR) - rL * unL * (SL - unL) + pL - pR) / (rR * (SR - unR) - rL * (SL - unL))
    ps = rL * (unL - SL) * (unL - SM) + pL

    def star(u, F, S, un, p):
        a = (S - un)[..., None]
        zero = np.zeros_like(p)[..., None]
        us = (a * u + np.concatenate([zero, (ps - p)[..., None] * n, (ps * SM - p * un)[..., None]], -1)) / (S - SM)[..., None]
        return F + S[..., None] * (us - u)
    pick = [(SL > 0)[..., None], (SM > 0)[..., None], (SR > 0)[..., None]]
    return np.select(pick, [FL, star(uL, FL, SL, unL, pL), star(uR, FR, SR, unR, pR)], FR)


def _advance(case, mesh, U):
    d, nk, M, kd, nq = _shape(case)
    nf, nv, n = d + 1, d + 2, len(mesh.cells)
    wall, lam1p = case["flow"] == "triple", 1e4 if case["flow"] == "triple" else 1e15
    per, eps, CT, scheme = mesh.period, 1e-24, 1e-6, case["scheme"]
    # positively oriented cells, their maps, faces and neighbours
    cells, X = mesh.cells.astype(np.int64), _corners(mesh)
    neg = np.linalg.det(X[:, 1:] - X[:, :1]) < 0
    cells[neg, 1], cells[neg, 2] = cells[neg, 2], cells[neg, 1].copy()
    X[neg, 1], X[neg, 2] = X[neg, 2], X[neg, 1].copy()
    J = (X[:, 1:] - X[:, :1]).swapaxes(1, 2)
    vol = np.linalg.det(J) / math.factorial(d)
    Ji = np.linalg.inv(J)
    cen = X[:, 0].copy()
    for k in range(1, nf):
        cen = cen + X[:, k]
    cen = cen / nf
    nb = _connect(cells)
    st, off = _stencils(cells, cen, per, M)
    normal, area = np.empty((n, nf, d)), np.empty((n, nf))
    for f in range(nf):
        P = np.delete(X, f, 1)
        e = P[:, 1:] - P[:, :1]
        w = np.stack([e[:, 0, 1], -e[:, 0, 0]], 1) if d == 2 else np.cross(e[:, 0], e[:, 1])
        size = np.linalg.norm(w, axis=1)
        w = w * np.sign(((P[:, 0] - X[:, f]) * w).sum(1))[:, None]
        normal[:, f], area[:, f] = w / size[:, None], size / (1 if d == 2 else 2)
    # the basis, its moments over every member in the target's reference space, the inverses
    ex = _powers(d, case["degree"])
    mean = np.array([_simplex_integral([int(t) for t in e]) for e in ex]) * math.factorial(d)
    O = _smoothness(ex, d)
    pts, wts = _rule(d, case["degree"] // 2 + 2)
    A, Vp = np.empty((n, M, nk)), vol[st] / (vol[:, None] * math.factorial(d))
    for m in range(M):
        sh = off[:, m] - (cen[st[:, m]] - cen)
        x = X[st[:, m], 0] + sh
        xi = ((x - X[:, 0])[:, None] + pts @ J[st[:, m]].swapaxes(1, 2)) @ Ji.swapaxes(1, 2)
        A[:, m] = (_basis(xi, ex) @ wts).T * (Vp[:, m] * math.factorial(d))[:, None] - Vp[:, m, None] * mean
    Pc = _pinv(A, np.full(n, M))[0] * Vp[:, None]
    # directional stencils: a member belongs to the first face whose cone from the centroid holds it
    Pd, adm, left = [], [], np.ones((n, M), bool)
    for f in range(nf):
        rays = (np.delete(X, f, 1) - cen[:, None]).swapaxes(1, 2)
        inside = (np.linalg.solve(rays[:, None], off[..., None])[..., 0] >= 0).all(2) & left
        left &= ~inside
        inside &= np.cumsum(inside, 1) <= 2 * kd
        p, ok = _pinv(np.where(inside[..., None], A[:, :, :kd], 0.0), inside.sum(1))
        Pd.append(p * Vp[:, None])
        adm.append(ok)
    Pd, adm = np.stack(Pd, 1), np.stack(adm, 1)
    del A
    # basis values at the face points, which both cells take in the same order
    bary, fw = _face_rule(d, nq)
    phi = np.empty((n, nf, nq, nk))
    ref = np.concatenate([np.zeros((1, d)), np.eye(d)])
    for f in range(nf):
        loc = np.delete(np.arange(nf), f)
        srt = loc[np.argsort(cells[:, loc], axis=1)]
        phi[:, f] = np.moveaxis(_basis(bary @ ref[srt], ex), 0, -1) - mean
    st_n = 1 + adm.sum(1)
    lam1 = 1 - 1 / lam1p
    lams = np.where(st_n > 1, (1 - lam1) / np.maximum(st_n - 1, 1), 0.0)[:, None]

    def weights(SI0, SId):
        """[n, nv] weight of p_1 and [n, nf, nv] of the directional polynomials."""
        on, lam = adm[..., None], lams[:, None]
        if scheme == 2:
            g0, g = lam1 / (SI0 + eps) ** 4, np.where(on, lam / (SId + eps) ** 4, 0.0)
            return g0 / (g0 + g.sum(1)), g / (g0 + g.sum(1))[:, None]
        if scheme == 1:
            tau = (np.where(on, np.abs(SId - SI0[:, None]), 0.0).sum(1) / np.maximum(st_n - 1, 1)[:, None]) ** 6
            g0, g = 1 + tau / (SI0 + eps), 1 + tau[:, None] / (SId + eps)
        else:
            g0, g = (SI0 + eps) ** -6.0, (SId + eps) ** -6.0
        if scheme != 3:
            g0, g = g0 * lam1, g * lam
        total = g0 + np.where(on, g, 0.0).sum(1)
        keep = ~(g0 / total < CT)
        sel = on & ~(g / total[:, None] < CT) & ~keep[:, None]
        return keep.astype(float), sel / np.maximum(sel.sum(1), 1)[:, None]

    def rate(U):
        """-(1 / |V|) sum over the faces of the flux."""
        dU = U[st] - U[:, None]
        a, ad = Pc @ dU, Pd @ dU[:, None]
        if scheme != 3:
            many = (st_n > 1)[:, None, None]
            split = a.copy()
            split[:, :kd] -= lams[..., None] * ad.sum(1)
            a = np.where(many, split / lam1, a)
        SI0 = np.einsum("nkv,kl,nlv->nv", a, O, a, optimize=True)
        SId = np.einsum("nfkv,kl,nflv->nfv", ad, O[:kd, :kd], ad, optimize=True)
        w0, wd = weights(SI0, SId)
        a = a * w0[:, None]
        a[:, :kd] += (wd[:, :, None] * ad).sum(1)
        W = U[:, None, None] + (phi.reshape(n, nf * nq, nk) @ a).reshape(n, nf, nq, nv)
        p = W[..., -1] * W[..., 0] - 0.5 * (W[..., 1:-1] ** 2).sum(-1)
        bad = (~((W[..., 0] > 0) & (p > 0))).any((1, 2))
        W = np.where(bad[:, None, None, None], U[:, None, None], W)
        out = W.reshape(n * nf, nq, nv)[np.maximum(nb, 0)]
        nn = np.broadcast_to(normal[:, :, None], (n, nf, nq, d))
        edge = (nb < 0)[..., None, None]
        if wall:
            mirror = W.copy()
            mirror[..., 1:-1] -= 2 * (W[..., 1:-1] * nn).sum(-1)[..., None] * nn
            out = np.where(edge, mirror, out)
        else:
            out = np.where(edge, U[:, None, None], out)
        F = (_flux(W, out, nn) * fw[:, None]).sum(2) * area[..., None]
        return -F.sum(1) / vol[:, None]

    for _ in range(case["steps"]):
        v = U[:, 1:-1] / U[:, :1]
        c = np.sqrt(GAMMA * (GAMMA - 1) * (U[:, -1] - 0.5 * (U[:, 1:-1] * v).sum(1)) / U[:, 0])
        dt = CFL[case["flow"]] * (vol / (area * (np.abs(np.einsum("nd,nfd->nf", v, normal)) + c[:, None])).sum(1)).min()
        if case["rk"] == 3:
            U1 = U + dt * rate(U)
            U2 = 0.75 * U + 0.25 * (U1 + dt * rate(U1))
            U = U / 3 + 2 / 3 * (U2 + dt * rate(U2))
        else:
            k1 = rate(U)
            k2 = rate(U + 0.5 * dt * k1)
            k3 = rate(U + 0.5 * dt * k2)
            U = U + dt / 6 * (k1 + 2 * k2 + 2 * k3 + rate(U + dt * k3))
    return U
