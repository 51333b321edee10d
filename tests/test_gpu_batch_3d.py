"""Batches of tetrahedral meshes, whose warps hold cells of two meshes and spare lanes: every mesh advances with its own
CFL step, bit for bit as alone."""
from __future__ import annotations

import numpy as np
import pytest

import workloads as W
from tests.test_gpu_parity import _native, _ragged, _solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("degree", [2, 3])
@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
def test_batch_equals_the_meshes_alone(precision, degree):
    native = _native()
    wls = [_ragged(W.blast_3d(n, seed=n), drop) for n, drop in ((5, 1), (4, 2), (6, 5), (4, 3))]
    states = [w.U0 * (1 + 0.5 * k) for k, w in enumerate(wls)]  # another time step for each
    launch = (0, 0) if precision == 0 else (11264 + 32, 8192 + 128)
    b = _solver(native, [w.mesh for w in wls], 3, degree=degree, precision=precision, cfl=0.3)
    native.cteno_set_launch(b.ctx, *launch)
    for k, u in enumerate(states):
        b.set_state(u, k)
    b.run(4)
    dts = b.dt()
    for k, (w, u) in enumerate(zip(wls, states)):
        s = _solver(native, [w.mesh], 3, degree=degree, precision=precision, cfl=0.3)
        native.cteno_set_launch(s.ctx, *launch)
        s.set_state(u)
        s.run(4)
        assert np.array_equal(s.get_state(), b.get_state(k)) and s.dt()[0] == dts[k]
        s.close()
    assert b.sync() >= 0 and len(set(dts)) > 1
    b.close()
