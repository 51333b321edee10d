"""The FP64 path at the limits of what it accepts, against the FP64 oracle: its reconstruction takes the central
inner products in integers and its flux compares wave speeds by their bits, and neither may show."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest

import workloads as W
from tests.test_gpu_parity import _native, _ragged, _relerr, _solver

pytestmark = pytest.mark.gpu

MESHES = {
    "tri-r2": (lambda: W.shock_tube_2d(23, 7), 2),
    "tri-r3": (lambda: W.density_wave_2d(12), 3),
    "tri-r4": (lambda: W.density_wave_2d(18), 4),
    "tri-r5": (lambda: W.shock_tube_2d(21, 17), 5),
    "tri-r6": (lambda: W.density_wave_2d(21), 6),
    "tet-r2": (lambda: W.density_wave_3d(6), 2),
    "tet-r3": (lambda: _ragged(W.blast_3d(6), 5), 3),
}


@pytest.mark.parametrize("jump", [1e2, 1e6, 1e10])
@pytest.mark.parametrize("scheme", [0, 1, 3], ids=["CTENO", "CTENOZ-wenoz", "TENO"])
@pytest.mark.parametrize("name", list(MESHES))
def test_low_side_of_a_jump(name, scheme, jump):
    """A jump of all variables between two smooth states: the cells beside it drop the stencils that cross it, and
    their face states are as accurate as products in FP64 give them, of the largest |U_v| over the members of the
    stencils that are kept (1e-12; max(1e-12, 50 cond(A) u) at degrees 4 to 6)."""
    native = _native()
    from oracle import Oracle
    make, degree = MESHES[name]
    wl = make()
    d, n = wl.mesh.dim, wl.mesh.ncells
    x = W.cell_centroids(wl.mesh)
    t = (x - x.min(0)) / np.ptp(x, axis=0).max()
    wave = 1 + 0.1 * np.sin(3 * t @ np.array([1.0, 0.7, 0.4])[:d] + np.arange(d + 2)[:, None])
    U = np.array([1.0] + [0.3, -0.2, 0.1][:d] + [2.5])[:, None] * wave * np.where(t[:, 0] > 0.5 * t[:, 0].max(), jump, 1.0)
    o = Oracle(wl.mesh, degree=degree, scheme=scheme, ctenoz_form=1)
    tol = 1e-12
    if degree >= 4:
        tol = max(tol, 50 * max(np.linalg.cond(o.lsq(i)[0]) for i in range(0, n, max(1, n // 60))) * 2.0 ** -53)
    o.set_state(U)
    o.residual()
    s = _solver(native, [wl.mesh], d, degree=degree, scheme=scheme, ctenoz_form=1)
    native.cteno_record_flags(s.ctx, True)
    s.set_state(U)
    s.stage(0, 0.0)
    got, flags = native.cteno_get_face_states(s.ctx, 0), native.cteno_get_flags(s.ctx, 0)
    s.close()
    assert np.array_equal(flags, o.flags())
    scale = np.abs(U)
    for i in range(n):
        central, directional, ok = o.stencil(i)
        for v in range(d + 2):
            kept = [central] if flags[i, v] & 1 else \
                [directional[f][directional[f] >= 0] for f in range(d + 1) if flags[i, v] >> (1 + f) & 1]
            scale[v, i] = max([scale[v, i]] + [np.abs(U[v, m]).max() for m in kept])
    low = t[:, 0] <= 0.5 * t[:, 0].max()
    assert (scale[0, low] < 2).any() and (flags[low, 0] & 1 == 0).any()
    assert np.all(np.abs(got - o.face_states()).reshape(n, -1, d + 2) <= tol * scale.T[:, None])


@pytest.mark.parametrize("guard", [0, 1])
@pytest.mark.parametrize("dim", [2, 3])
def test_negative_pressure_on_one_side_of_a_face(dim, guard):
    """Means with a negative pressure (alone, among physical ones): one side of their faces has no speed of sound,
    and the wave speeds are those of the other side and of the Roe average, as fmin and fmax give them."""
    native = _native()
    from oracle import Oracle
    wl = W.density_wave_2d(14) if dim == 2 else W.density_wave_3d(6)
    U = wl.U0.copy()
    for c in range(5, wl.mesh.ncells, wl.mesh.ncells // 7):
        U[-1, c] = 0.9 * 0.5 * (U[1:-1, c] ** 2).sum() / U[0, c]
    o = Oracle(wl.mesh, degree=2, guard=guard)
    o.set_state(U)
    o.stage(0, 1e-4)
    ref = o.get_state()
    assert np.isfinite(ref).all()
    s = _solver(native, [wl.mesh], dim, degree=2, positivity_guard=guard)
    s.set_state(U)
    s.stage(0, 1e-4)
    assert _relerr(s.get_state(), ref) < 1e-12
    assert s.sync() == o.nguard()
    s.close()


@pytest.mark.parametrize("guard", [0, 1])
@pytest.mark.parametrize("name", list(MESHES))
def test_cut_off_that_drops_every_stencil(name, guard):
    """TENO with C_T = 0.5: in smooth flow every chi_s is about 1 / s_t, no stencil is kept, and the face states
    are the mean (p = 0 added to U_0), with no help of the positivity guard."""
    native = _native()
    from oracle import Oracle
    make, degree = MESHES[name]
    wl = make()
    d = wl.mesh.dim
    o = Oracle(wl.mesh, degree=degree, scheme=3, C_T=0.5, guard=guard)
    o.set_state(wl.U0)
    o.residual()
    s = _solver(native, [wl.mesh], d, degree=degree, scheme=3, C_T=0.5, positivity_guard=guard)
    native.cteno_record_flags(s.ctx, True)
    s.set_state(wl.U0)
    s.stage(0, 0.0)
    got, flags = native.cteno_get_face_states(s.ctx, 0), native.cteno_get_flags(s.ctx, 0)
    count = ctypes.c_int64(-1)  # filled also where two negative pressures meet at a face, without the guard
    native.load_library().cteno_sync(s.ctx, ctypes.byref(count))
    s.close()
    assert (o.flags() == 0).any()
    assert np.array_equal(flags, o.flags()) and count.value == o.nguard()
    assert _relerr(got.reshape(-1, d + 2).T, o.face_states().reshape(-1, d + 2).T) < 1e-12


@pytest.mark.parametrize("name", list(MESHES))
def test_face_states_do_not_depend_on_the_cells_of_the_warp(name):
    """A mesh alone and as the second of a batch, whose first cells share a warp with the last ones of the first: the
    same bits. The first mesh is uniform, so that the range of its stencils is taken again from the whole means. The
    momenta of the second reach from -1 to 1 - 2^-40 in most stencils: the bound of that range by the high words is
    in the next binade, and the unit of the differences would be another. C_T = 0 keeps the central stencil."""
    native = _native()
    make, degree = MESHES[name]
    wl = make()
    d, n = wl.mesh.dim, wl.mesh.ncells
    small = {"tri-r2": lambda: W.shock_tube_2d(5, 9), "tri-r5": lambda: W.shock_tube_2d(9, 5),
             "tet-r3": lambda: _ragged(W.blast_3d(4), 1), "tet-r2": lambda: _ragged(W.density_wave_3d(4), 1)}
    first = small.get(name, lambda: W.density_wave_2d(13))()
    assert first.mesh.ncells % (8 if d == 2 else 6)
    flat = np.repeat(np.array([1.0] + [0.5, -0.25, 0.125][:d] + [2.0])[:, None], first.mesh.ncells, axis=1)
    for seed in range(3):
        rng = np.random.default_rng(seed)
        U = rng.uniform(1, 2, (d + 2, n))
        U[1:-1] = rng.uniform(-0.9, 0.9, (d, n))
        pick = rng.integers(0, 4, (d, n))
        U[1:-1][pick == 0] = -1.0
        U[1:-1][pick == 1] = 1.0 - 2.0 ** -40
        out = []
        for meshes, states in (([wl.mesh], [U]), ([first.mesh, wl.mesh], [flat, U])):
            s = _solver(native, meshes, d, degree=degree, C_T=0.0, positivity_guard=0)
            for k, u in enumerate(states):
                s.set_state(u, k)
            s.stage(0, 0.0)
            out.append(native.cteno_get_face_states(s.ctx, len(meshes) - 1))
            s.close()
        assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("scheme", [0, 2], ids=["CTENO", "CWENO"])
@pytest.mark.parametrize("exponent", [-930, 1015, 1021])
@pytest.mark.parametrize("name", list(MESHES))
def test_means_near_the_ends_of_the_exponents(name, exponent, scheme):
    """Fluid at rest in units of 2^exponent: a cell has the face states of the same flow in units of 2^-800 or 2^900
    (the indicators vanish against eps or overflow there too: the same selection), or, where coefficients or face
    values do not fit the range of the numbers, it has its mean at every face, counted by the positivity guard."""
    native = _native()
    from oracle import Oracle
    make, degree = MESHES[name]
    wl = make()
    d, n = wl.mesh.dim, wl.mesh.ncells
    unit = -800 if exponent < 0 else 900
    U = wl.U0 / 10
    U[1:-1] = 0.0
    o = Oracle(wl.mesh, degree=degree, scheme=scheme)
    o.set_state(np.ldexp(U, unit))
    o.residual()
    tol = max(1e-12, 50 * max(np.linalg.cond(o.lsq(i)[0]) for i in range(0, n, max(1, n // 60))) * 2.0 ** -53)
    s = _solver(native, [wl.mesh], d, degree=degree, scheme=scheme)
    s.set_state(np.ldexp(U, exponent))
    s.stage(0, 0.0)
    got = native.cteno_get_face_states(s.ctx, 0).reshape(n, -1, d + 2)
    count = ctypes.c_int64(-1)
    native.load_library().cteno_sync(s.ctx, ctypes.byref(count))
    s.close()
    ref = o.face_states().reshape(n, -1, d + 2)
    same = (np.abs(np.ldexp(got, -exponent) - np.ldexp(ref, -unit)) <= tol * np.abs(U).max(axis=1)).all(axis=(1, 2))
    mean = (got == np.ldexp(U, exponent).T[:, None]).all(axis=(1, 2))
    assert np.all(same | mean)
    flat = (ref == np.ldexp(U, unit).T[:, None]).all(axis=(1, 2)) & ~o.guarded()
    assert count.value == np.count_nonzero(mean & ~flat)
    if exponent < 1015:
        assert np.all(same)
