"""The positivity guard's count of the tile-per-warp schedule where cells do fall back to their mean. A synchronising
call that reports a non-finite state raises in the Python wrapper and drops the count, so it is read from the library
call itself, which fills it either way."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest

import workloads as W
from tests.test_gpu_parity import _native, _solver
from tests.test_gpu_tile import MESHES

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("launch", [10240 + 32, 10240 + 128, 11264 + 32, 11264 + 128])
@pytest.mark.parametrize("name", list(MESHES))
def test_equal_and_positive(name, launch):
    native = _native()
    make, degree = MESHES[name]
    wl = make()
    d, U = wl.mesh.dim, wl.U0.copy()
    rng = np.random.default_rng(3)
    U[1] += U[0] * rng.choice([0.0, 3.0, 300.0], wl.mesh.ncells)
    U[-1] = 0.5 * (U[1:-1] ** 2).sum(0) / U[0] + 10.0 ** rng.uniform(-6, 0, wl.mesh.ncells)
    counts = []
    for value in (1024 + 128, launch):
        s = _solver(native, [wl.mesh], d, degree=degree, precision=native.CTENO_MIXED)
        native.cteno_set_launch(s.ctx, value, 128)
        s.set_state(U)
        s.stage(0, 0.0)
        n = ctypes.c_int64(-1)
        native.load_library().cteno_sync(s.ctx, ctypes.byref(n))
        counts.append(n.value)
        s.close()
    assert counts[0] == counts[1] > 0
