"""cteno_autotune times a Runge-Kutta stage before the context has taken a step: what memory held before must
not reach the check for non-finite states."""
from __future__ import annotations

import pytest

import workloads as W
from tests.test_gpu_parity import _native, _solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rk", [3, 4])
@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
def test_autotune_on_memory_that_held_nan(precision, rk):
    import torch
    native = _native()
    wl = W.shock_tube_2d(64, 16)
    for _ in range(3):
        for n in (1 << 10, 1 << 14, 1 << 16, 1 << 18, 1 << 20):
            x = [torch.full((n,), float("nan"), dtype=torch.float64, device="cuda") for _ in range(8)]
            del x
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        s = _solver(native, [wl.mesh], 2, degree=2, precision=precision, rk=rk)
        s.set_state(wl.U0)
        native.cteno_autotune(s.ctx)
        s.run(1)
        assert s.sync() >= 0
        s.close()
