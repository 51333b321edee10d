"""Programmatic dependent launch: a stage kernel may start before the previous one has ended, so every load of
what that one writes (the state, the face states, the face fluxes) comes after the wait for it. A read-only load
counts as a load of constants, which the compiler may move above the wait, unless its address is taken behind it
(after_wait): checked in the sources here, and on the GPU by equal bits with and without the dependent launch.
"""
from __future__ import annotations

import os
import re

import numpy as np
import pytest

import paper_2312_17042_gb300 as package
import workloads as W
from tests.test_gpu_parity import _native, _ragged, _solver

CSRC = os.path.join(os.path.dirname(package.__file__), "csrc")
WRITTEN = r"\ba\.(U|U32|Uf|Ff)\b"  # fields of the kernel arguments that stage kernels write


def _read_only_loads(text):
    """Arguments of __ldg and of the record loads that start with read-only loads."""
    for m in re.finditer(r"\b(__ldg|load16|load16_stream)\s*(<[^()]*>)?\(", text):
        if m.group(1) == "load16" and m.group(2) and m.group(2).rstrip(">").split(",")[-1].strip() == "true":
            continue  # a shared-memory copy
        depth, k = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[k], 0)
            k += 1
        yield text[m.end():k - 1]


@pytest.mark.parametrize("name", sorted(n for n in os.listdir(CSRC) if n.endswith((".cu", ".cuh"))))
def test_read_only_loads_of_written_data_start_behind_the_wait(name):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    for load in _read_only_loads(text):
        assert not re.search(WRITTEN, load), load
    # a pointer kept for such loads (no alias, to constants) comes from after_wait
    for line in re.findall(r"const [^;\n]*\*\s*__restrict__ \w+ = [^;]*;", text):
        assert not re.search(WRITTEN, line) or "after_wait(" in line, line


# every reconstruction schedule of the mixed path at degrees 2 and 3, with each of the flux schedules
MIXED = [(128, 128), (-128, -128), (1024 + 128, 1024 + 128), (2048 + 32, 128), (3072 + 64, 8192 + 128), (4096, 128),
         (4097, 128), (5120 + 4, 128), (5152 + 4, -128), (6144 + 2, 128), (7168 + 2, 128), (10240 + 32, 128),
         (11264 + 32, 8192 + 128)]
CASES = ([(d, 2, 1, 0, 0, launch) for d in (2, 3) for launch in MIXED] +
         [(d, 3, 1, 0, 1, launch) for d in (2, 3) for launch in ((128, -128), (1024 + 256, 128), (6144 + 1, 128), (11264 + 128, 128))] +
         [(d, deg, 0, 0, 0, (128, 64)) for d, deg in ((2, 2), (2, 3), (2, 5), (3, 2), (3, 3))] +
         [(2, deg, 1, 0, 0, (1024 + 32, 128)) for deg in (4, 6)] +
         [(d, deg, p, 1, 0, (1024 + 128, 128)) for d, deg in ((2, 2), (2, 3), (2, 4), (3, 2), (3, 3)) for p in (0, 1)])


@pytest.mark.gpu
@pytest.mark.parametrize("dim,degree,precision,characteristic,scheme,launch", CASES)
def test_dependent_launch_keeps_every_bit(monkeypatch, dim, degree, precision, characteristic, scheme, launch):
    native = _native()
    wl = W.shock_tube_2d(61, 17) if dim == 2 else _ragged(W.blast_3d(7), 5)
    out = []
    for pdl in ("1", "0"):
        monkeypatch.setenv("CTENO_PDL", pdl)
        s = _solver(native, [wl.mesh], dim, degree=degree, precision=precision, characteristic=characteristic,
                    scheme=scheme, cfl=0.3)
        try:
            native.cteno_set_launch(s.ctx, *launch)
        except native.CtenoError:  # a staged schedule whose stages do not fit at this degree
            s.close()
            pytest.skip("refused at this degree")
        s.set_state(wl.U0)
        s.run(4)
        out.append((s.get_state(), s.dt(), s.sync()))
        s.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    assert out[0][2] == out[1][2]
