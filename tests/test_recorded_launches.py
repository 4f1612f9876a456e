"""What the library's host side asks of the device, on the CPU: gp_api.cu is
compiled with stand-ins for the CUDA runtime and the kernel launchers
(recorded_launches.cpp), which write down every allocation and every launch's
arguments."""
from __future__ import annotations

import ctypes as C
import os
import shutil
import subprocess

import pytest

from paper_2110_11226_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
MSE, PEARSON, SPEARMAN = 1, 4, 5


@pytest.fixture
def lib(tmp_path):
    """a library of its own, with nothing allocated yet"""
    cuda = os.path.join(os.path.dirname(os.path.dirname(build._nvcc())) or "/usr/local/cuda", "include")
    if shutil.which("g++") is None or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("g++ and the CUDA headers are needed")
    so = str(tmp_path / "recorded.so")
    # (-Bsymbolic: its own stand-ins, whatever else the process has loaded)
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-I" + build.INCLUDE,
                    "-I" + build.CSRC, "-I" + cuda, os.path.join(HERE, "recorded_launches.cpp"), "-o", so], check=True)
    lib = C.CDLL(so)
    lib.recorded.restype = C.c_char_p
    lib.memory_limit.argtypes = [C.c_size_t]
    return lib


P = C.c_void_p(1 << 20)  # a device pointer that nothing reads, 16-byte aligned


def _lines(lib, *kinds):
    """the recorded lines of these kinds as dicts, and forgets all"""
    out = []
    for line in lib.recorded().decode().splitlines():
        kind, *fields = line.split()
        if kind in kinds:
            out.append(dict({k: int(v) for k, v in (f.split("=") for f in fields)}, kind=kind))
    lib.record_anew()
    return out


def _evaluate(lib, n_progs, n_rows, n_feat, metric, w=None):
    return lib.gp_evaluate(P, P, n_progs, P, C.c_int64(n_rows), n_feat, P, w, metric, P, None)


@pytest.mark.parametrize("n_feat", [1, 2, 3])
@pytest.mark.parametrize("n_rows", [999, 4096])
def test_column_stride_of_every_evaluator_launch(lib, n_feat, n_rows):
    """Feature mode 2 reads n_rows floats at X + ld: inside the table only when
    ld is 0 (one column) or n_rows (two)."""
    calls = [lambda: _evaluate(lib, 100, n_rows, n_feat, m) for m in (MSE, PEARSON, SPEARMAN)]
    calls.append(lambda: lib.gp_predict(P, P, 100, P, C.c_int64(n_rows), n_feat, P, None))
    calls.append(lambda: lib.gp_const_grad(P, P, 100, P, C.c_int64(n_rows), n_feat, P, None, MSE, P, P, None))
    for call in calls:
        assert call() == 0
        launches = _lines(lib, "eval", "predict")
        assert launches
        for a in launches:
            assert a["fmode"] == (2 if n_feat <= 2 else 0) and a["rows"] == n_rows
            assert a["ld"] == (0 if n_feat == 1 else n_rows), a
