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


@pytest.fixture(scope="module")
def recorded(tmp_path_factory):
    cuda = os.path.join(os.path.dirname(os.path.dirname(build._nvcc())) or "/usr/local/cuda", "include")
    if shutil.which("g++") is None or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("g++ and the CUDA headers are needed")
    so = str(tmp_path_factory.mktemp("recorded") / "recorded.so")
    # (-Bsymbolic: its own stand-ins, whatever else the process has loaded)
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-I" + build.INCLUDE,
                    "-I" + build.CSRC, "-I" + cuda, os.path.join(HERE, "recorded_launches.cpp"), "-o", so], check=True)
    return so


@pytest.fixture
def lib(recorded, tmp_path):
    """a copy of its own, with nothing allocated yet"""
    lib = C.CDLL(shutil.copy(recorded, tmp_path / "copy.so"))
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


@pytest.mark.parametrize("limit", [1 << 40, 7 << 29], ids=["room", "3.5 GB"])
def test_rank_scratch_is_allocated_once(lib, limit):
    """A population of several batches: where the device gives no 4.5 GB the
    smaller batch runs, and the next call of the shape neither frees nor
    allocates (it may be captured in a graph)."""
    lib.memory_limit(limit)
    for call in range(3):
        assert _evaluate(lib, 512, 1_000_000, 2, SPEARMAN) == 0
        lines = _lines(lib, "malloc", "free", "rank")
        memory = [a for a in lines if a["kind"] != "rank"]
        batches = [a["segments"] for a in lines if a["kind"] == "rank"]
        assert sum(batches) == 512 and len(set(batches[:-1])) == 1
        if call == 0:
            big = [a for a in memory if a["bytes"] > 1 << 30]
            assert [a["ok"] for a in big] == ([1] if limit > 1 << 33 else [0, 1])
            first = batches
        else:
            assert memory == []
            assert batches == first


def test_refused_rank_scratch_leaves_what_is_held(lib):
    """The larger batch is asked for beside the buffer that is there: when it
    is refused and the buffer serves the smaller batch, nothing moves."""
    lib.memory_limit(7 << 29)
    assert _evaluate(lib, 512, 1_000_000, 2, SPEARMAN) == 0
    small = max(a["segments"] for a in _lines(lib, "rank"))
    lib.gp_shutdown()
    lib.record_anew()
    assert _evaluate(lib, small, 1_000_000, 2, SPEARMAN) == 0   # one batch, within the smaller budget
    assert [a["ok"] for a in _lines(lib, "malloc") if a["bytes"] > 1 << 30] == [1]
    assert _evaluate(lib, 512, 1_000_000, 2, SPEARMAN) == 0
    lines = _lines(lib, "malloc", "free")
    assert [(a["kind"], a.get("ok")) for a in lines if a["bytes"] > 1 << 30] == [("malloc", 0)]


@pytest.mark.parametrize("w", [None, P], ids=["unweighted", "weighted"])
@pytest.mark.parametrize("n_rows", [1, 500, 2000, 3000])
def test_rank_batch_fits_a_grid(lib, w, n_rows):
    """A segment is a row of the sort's grid: at most 65535 of them."""
    assert _evaluate(lib, 200_000, n_rows, 2, SPEARMAN, w) == 0
    batches = [a["segments"] for a in _lines(lib, "rank")]
    assert sum(batches) == 200_000 and max(batches) <= 65535
