"""The steps that the validation cuts rows plus entries into, on the host: the
arithmetic of csrc/gc_steps.h, compiled with g++.  Every step begins in
exactly one row, in both widths of the division; a row whose start lies before
the first one (malformed offsets: off[0] above later offsets) begins none."""
import ctypes
import subprocess
from pathlib import Path

import numpy as np
import pytest

ROOT = Path(__file__).resolve().parents[1]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = tmp_path_factory.mktemp("row_steps") / "row_steps.so"
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC",
                           f"-I{ROOT / 'paper_1407_6745_gb300' / 'csrc'}",
                           str(ROOT / "tests" / "helpers" / "row_steps.cpp"), "-o", str(so)])
    lib = ctypes.CDLL(str(so))
    lib.row_steps.argtypes = [ctypes.c_int64, ctypes.c_int32, ctypes.c_int64, ctypes.c_int, ctypes.c_void_p]
    return lib


def _steps(lib, d, deg, steps, narrow):
    k = (ctypes.c_int64 * 2)()
    lib.row_steps(d, deg, steps, narrow, k)
    return range(k[0], k[1] + 1)


@pytest.mark.parametrize("narrow", [0, 1])
@pytest.mark.parametrize("degrees", [[0], [0] * 1000, [251], [252], [253], [100_000], [0, 251, 0, 252, 1, 504, 0, 0],
                                     list(np.random.default_rng(1).integers(0, 700, 500))])
def test_every_step_begins_in_one_row(lib, degrees, narrow):
    places = lib.step_places()
    n, nnz = len(degrees), int(sum(degrees))
    steps = (n + nnz) // places + 1
    first = [None] * steps
    at = 0  # row v covers the places [at, at + deg + 1)
    starts = []
    for v, deg in enumerate(degrees):
        starts.append(at)
        for k in _steps(lib, at, int(deg), steps, narrow):
            assert first[k] is None
            first[k] = v
        at += int(deg) + 1
    for k in range((n + nnz + places - 1) // places):
        assert first[k] == int(np.searchsorted(starts, k * places, side="right")) - 1


@pytest.mark.parametrize("narrow", [0, 1])
@pytest.mark.parametrize("d", [-1, -7, -251, -252, -(1 << 31), -(1 << 40)])
def test_a_row_before_the_first_begins_no_step(lib, d, narrow):
    assert len(_steps(lib, d, 0, 8_500_000, narrow)) == 0
    assert len(_steps(lib, d, 1000, 8_500_000, narrow)) == 0
