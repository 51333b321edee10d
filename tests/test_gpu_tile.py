"""The tile-per-warp reconstruction (launch values 10240 + b: two variables per lane, 11264 + b: one) keeps the order of every
sum: face states, flags and guard counts equal those of the variable-per-lane schedule (1024 + 128) bit for
bit, at tile remainders (16 and 8 cells in 2D, 10 and 6 in 3D), with every weighting, where the guard's bounds
decide, where its points have to be tested, and where cells fall back to their mean."""
from __future__ import annotations

import numpy as np
import pytest

import workloads as W
from tests.test_gpu_parity import _native, _ragged, _solver

pytestmark = pytest.mark.gpu

MESHES = {
    "tri-r2": (lambda: W.shock_tube_2d(23, 7), 2),          # 322 cells: the last tile has 2
    "tri-r2-one": (lambda: _ragged(W.shock_tube_2d(24, 8), 15), 2),  # 369: 1
    "tri-r3": (lambda: W.density_wave_2d(12), 3),           # 288: whole tiles
    "tet-r2": (lambda: W.density_wave_3d(6), 2),            # 1296: 6
    "tet-r3": (lambda: _ragged(W.blast_3d(6), 5), 3),       # 1291: 1
}


@pytest.mark.parametrize("launch", [10240 + 32, 10240 + 128, 11264 + 32, 11264 + 128])
@pytest.mark.parametrize("scheme", [0, 1, 2, 3], ids=["CTENO", "CTENOZ", "CWENO", "TENO"])
@pytest.mark.parametrize("state", ["flow", "thin", "nan"])
@pytest.mark.parametrize("name", list(MESHES))
def test_equal_to_the_lane_schedule(name, state, scheme, launch):
    native = _native()
    make, degree = MESHES[name]
    wl = make()
    d, U = wl.mesh.dim, wl.U0.copy()
    rng = np.random.default_rng(3)
    if state == "thin":  # pressures within 1e-5 of nothing, and steep jumps: the points decide, some fail
        U[1] += U[0] * rng.choice([0.0, 3.0, 300.0], wl.mesh.ncells)
        U[-1] = 0.5 * (U[1:-1] ** 2).sum(0) / U[0] + 10.0 ** rng.uniform(-6, 0, wl.mesh.ncells)
    if state == "nan":
        U[0, wl.mesh.ncells // 3] = np.nan
    out = []
    for value in (1024 + 128, launch):
        s = _solver(native, [wl.mesh], d, degree=degree, scheme=scheme, precision=native.CTENO_MIXED)
        native.cteno_set_launch(s.ctx, value, 128)
        native.cteno_record_flags(s.ctx, True)
        s.set_state(U)
        s.stage(0, 0.0)
        try:
            guard = s.sync()
        except native.CtenoError:  # the update found a non-finite state (the NaN, or a flux of the thin one)
            guard = None
        out.append((native.cteno_get_face_states(s.ctx, 0), native.cteno_get_flags(s.ctx, 0), guard))
        s.close()
    assert np.array_equal(out[0][0], out[1][0], equal_nan=True)
    assert np.array_equal(out[0][1], out[1][1])
    assert out[0][2] == out[1][2]
    if state == "thin":
        assert out[0][2] is None or out[0][2] > 0


@pytest.mark.parametrize("degree", [2, 3])
def test_2d_results_do_not_depend_on_the_schedule(degree):
    """2D, mixed: the thread-per-cell and the tile-per-warp schedules, and with them any the
    library takes by default, give the same bits over several steps."""
    native = _native()
    wl = W.shock_tube_2d(37, 11)
    out = []
    for launch in ((128, 128), (10240 + 32, -128), (11264 + 128, 8192 + 128)):
        s = _solver(native, [wl.mesh], 2, degree=degree, scheme=1, precision=native.CTENO_MIXED)
        native.cteno_set_launch(s.ctx, *launch)
        s.set_state(wl.U0)
        s.run(5)
        out.append((s.get_state(), s.dt()))
        s.close()
    for o in out[1:]:
        assert np.array_equal(o[0], out[0][0]) and np.array_equal(o[1], out[0][1])
