"""Every kernel that waits for its bulk copies gives up after a limit, reports it and lets the copies land: the test
hook's barrier, which nothing completes, in the kernels that the library takes by default (the FP64 reconstruction,
the streamed one at degrees 4 to 6, the tile-per-warp one with one and two variables per lane)."""
from __future__ import annotations

import pytest

import workloads as W
from tests.test_gpu_failures import CTENO_ERR_DEVICE, _fresh_context_works
from tests.test_gpu_parity import _native, _ragged, _solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,degree,precision,launch", [
    (2, 2, 0, 0), (2, 3, 0, 64), (2, 4, 0, 0), (2, 6, 0, 0), (3, 2, 0, 128), (3, 3, 0, 0),
    (2, 4, 1, 0), (2, 5, 1, 1024 + 128), (2, 6, 1, 1536 + 64),
    (2, 2, 1, 0), (2, 3, 1, 11264 + 128), (2, 2, 1, 10240 + 64), (3, 2, 1, 11264 + 32), (3, 3, 1, 10240 + 32)])
def test_a_wait_that_runs_out_is_reported(dim, degree, precision, launch):
    native = _native()
    wl = W.shock_tube_2d(63, 17) if dim == 2 else _ragged(W.blast_3d(6), 5)  # the last tile is not whole
    s = _solver(native, [wl.mesh], dim, degree=degree, precision=precision, cfl=0.3)
    native.cteno_set_launch(s.ctx, launch, 0)
    s.set_state(wl.U0)
    s.run(1)
    assert s.sync() >= 0                # the schedule runs cleanly without the hook
    native.cteno_test_wait_timeout(s.ctx, 1_000_000)   # 1 ms
    s.run(1)
    with pytest.raises(native.CtenoError) as e:
        s.sync()
    assert e.value.code == CTENO_ERR_DEVICE
    assert "timed out" in str(e.value)
    s.close()
    _fresh_context_works(native)
