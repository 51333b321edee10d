"""The FP64 path's reconstruction forms its inner products in block fixed-point integers and takes
its decisions in FP32 where they are certain: face states and flags against the FP64 oracle where
the blocks, the scales and the decisions are at their limits.

Tolerances, of the largest |U_v| over the cell's stencil: 1e-12 as for the other FP64
parity tests (degrees 2 and 3; max(1e-12, 50 cond(A) u) at degrees 4 to 6); for means that differ by
1e-12 of themselves, whose face values both sides only round, the K-1 roundings of the oracle's sum
(it adds each term to U_0) and two of the library's, 2^-53 each.
"""
from __future__ import annotations

import numpy as np
import pytest

import workloads as W
from tests.test_gpu_parity import _native, _ragged, _solver

pytestmark = pytest.mark.gpu

MESHES = {
    "tri-r2": (lambda: W.shock_tube_2d(23, 7), 2),        # 322 cells: the last 8-cell tile has 2
    "tri-r3": (lambda: W.density_wave_2d(12), 3),
    "tri-r4": (lambda: W.density_wave_2d(18), 4),
    "tri-r5": (lambda: W.shock_tube_2d(21, 17), 5),
    "tri-r6": (lambda: W.density_wave_2d(21), 6),
    "tet-r2": (lambda: W.density_wave_3d(6), 2),
    "tet-r3": (lambda: _ragged(W.blast_3d(6), 5), 3),     # 1291 cells: the last 6-cell tile has 1
}


def _cond(o, n):
    return max(np.linalg.cond(o.lsq(i)[0]) for i in range(0, n, max(1, n // 60)))


def _states(wl, kind):
    rng = np.random.default_rng(7)
    d, n = wl.mesh.dim, wl.mesh.ncells
    if kind == "near-uniform":
        u = np.array([1.0] + [0.3, -0.2, 0.1][:d] + [2.5])
        return u[:, None] * (1 + 1e-12 * rng.uniform(-1, 1, (d + 2, n)))
    if kind == "wide":  # twelve decades between neighbours, both signs, exact zeros
        rho = 10.0 ** rng.uniform(-6, 6, n)
        mom = rho * rng.choice([0.0, 1.0, -1e-3], (d, n)) * 10.0 ** rng.uniform(-3, 0, (d, n))
        return np.concatenate([rho[None], mom, (rho * 10.0 ** rng.uniform(0.5, 2, n))[None]])
    return wl.U0 * {"small": 2.0 ** -200, "large": 2.0 ** 40}[kind]


@pytest.mark.parametrize("kind", ["near-uniform", "wide", "small", "large"])
@pytest.mark.parametrize("scheme", [0, 1, 2, 3], ids=["CTENO", "CTENOZ", "CWENO", "TENO"])
@pytest.mark.parametrize("name", list(MESHES))
def test_face_states_and_flags_at_the_limits(name, scheme, kind):
    native = _native()
    from oracle import Oracle
    if scheme == 2 and kind == "wide":
        pytest.skip("weights (eps + SI)^-4 of indicators that cancel over twelve decades: no 1e-12 in any order")
    make, degree = MESHES[name]
    wl = make()
    d, U = wl.mesh.dim, _states(wl, kind)
    o = Oracle(wl.mesh, degree=degree, scheme=scheme)
    tol = 1e-12 if degree <= 3 else max(1e-12, 50 * _cond(o, wl.mesh.ncells) * 2.0 ** -53)
    if kind == "near-uniform":
        tol = (o.nk + 2) * 2.0 ** -53
    o.set_state(U)
    o.residual()
    s = _solver(native, [wl.mesh], d, degree=degree, scheme=scheme)
    native.cteno_record_flags(s.ctx, True)
    s.set_state(U)
    s.stage(0, 0.0)
    got = native.cteno_get_face_states(s.ctx, 0).reshape(-1, d + 2)
    flags = native.cteno_get_flags(s.ctx, 0)
    s.close()
    ref = o.face_states().reshape(-1, d + 2)
    assert np.array_equal(flags, o.flags())
    st = np.array([np.append(o.stencil(i)[0], i) for i in range(wl.mesh.ncells)])
    scale = np.abs(U[:, st]).max(axis=2).T[:, None]
    assert np.all(np.abs(got - ref).reshape(len(st), -1, d + 2) <= tol * scale)


@pytest.mark.parametrize("name", list(MESHES))
def test_non_finite_mean_reaches_its_stencils_only(name):
    """A NaN in one cell's density: cells with it in their stencil fall back to their mean (the
    positivity guard), every other cell's face states stay the same bits."""
    native = _native()
    make, degree = MESHES[name]
    wl = make()
    d, n, bad = wl.mesh.dim, wl.mesh.ncells, wl.mesh.ncells // 2
    s = _solver(native, [wl.mesh], d, degree=degree)
    out = []
    for value in (wl.U0[0, bad], np.nan, np.inf):
        U = wl.U0.copy()
        U[0, bad] = value
        s.set_state(U)
        s.stage(0, 0.0)
        out.append(native.cteno_get_face_states(s.ctx, 0))
    hit = np.array([bad in native.cteno_get_stencil(s.ctx, 0, i)[0] for i in range(n)])
    s.close()
    hit[bad] = True
    for got in out[1:]:
        assert np.array_equal(got[~hit], out[0][~hit])
        rest = hit.copy()
        rest[bad] = False
        assert np.array_equal(got[rest], np.broadcast_to(wl.U0.T[rest][:, None, None], got[rest].shape))
