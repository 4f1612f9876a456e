"""The sample that splits the rank fitness's values into buckets: it must not be
misled by rows that follow one another by a rule.  Where it is (a column made to
defeat it), the sort takes over with the same results."""
from __future__ import annotations

import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle
from paper_2110_11226_gb300 import build, synth

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ is needed")
    so = str(tmp_path_factory.mktemp("sample") / "sample.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-I" + build.CSRC,
                    os.path.join(HERE, "rank_sample.cpp"), "-o", so], check=True)
    lib = C.CDLL(so)
    for f in (lib.buckets, lib.samples):
        f.argtypes = [C.c_int64]
    lib.row.argtypes, lib.row.restype = [C.c_int, C.c_int64], C.c_int64
    return lib


def _rows(lib, n):
    return np.array([lib.row(i, n) for i in range(lib.samples(n))], dtype=np.int64)


SIZES = [6145, 8192, 16384, 65536, 200_003, 1 << 18, 1_000_000, 1 << 20, 1 << 22]


@pytest.mark.parametrize("n", SIZES)
def test_one_row_of_each_stratum(lib, n):
    rows, s = _rows(lib, n), lib.samples(n)
    i = np.arange(s, dtype=np.int64)
    assert np.all(rows >= i * n // s) and np.all(rows < (i + 1) * n // s)


@pytest.mark.parametrize("n", SIZES)
def test_no_bucket_overflows_on_structured_rows(lib, n):
    r = np.arange(n)
    side = int(round(n ** 0.5))
    rng = np.random.default_rng(1)
    noise = rng.random(n)
    columns = dict(fast_axis=r % side, slow_axis=r // side, rising=r, falling=-r, iid=rng.standard_normal(n),
                   sine256=np.sin(2 * np.pi * r / 256) + 1e-3 * noise,
                   sine100=np.sin(2 * np.pi * r / 100) + 1e-6 * noise,
                   period128=r % 128 + 1e-3 * noise, period64=r % 64 + 1e-3 * noise,
                   interleaved=(r % 64) * 1e6 + r // 64, two_rows=r % (2 * side) + 1e-6 * (r // side),
                   surface=np.sin((r % side) * 10.0 / side) * np.cos((r // side) * 10.0 / side))
    nb, rows = lib.buckets(n), _rows(lib, n)
    for name, v in columns.items():
        v = v.astype(np.float32)
        sample = np.sort(v[rows])
        split = sample[np.arange(1, nb, dtype=np.int64) * len(sample) // nb]
        j = np.searchsorted(split, v, side="left")   # splitters below
        equal = (j < nb - 1) & (split[np.minimum(j, nb - 2)] == v)  # these need no place
        fullest = np.bincount(j[~equal], minlength=nb).max()
        assert fullest <= lib.capacity(), name


@pytest.mark.parametrize("n_seg", [1, 3, 600, 65535])
@pytest.mark.parametrize("x", [1, 2, 4, 32, 245, 1024])
def test_listed_segments_fill_the_device(lib, n_seg, x):
    """blocks for every SM, or for every segment, and few that read a zero"""
    rows = lib.listed_rows(C.c_int64(n_seg), C.c_int64(x))
    assert 1 <= rows <= n_seg
    assert rows * x >= min(n_seg * x, 4 * 152)
    assert rows * x < max(4 * x, 4 * 152 + x) + 1


@pytest.mark.gpu
@pytest.mark.parametrize("n,n_progs", [(8192, 700), (16384, 600), (200_003, 12), (1_000_000, 9)])
def test_every_program_misjudged(lib, n, n_progs):
    """Values far below at the sampled rows and close together elsewhere: the
    buckets of every program overflow and the sort ranks them.  Powers of two
    times the column, so each has the column's ranks."""
    import torch

    from paper_2110_11226_gb300 import gp
    rng = np.random.default_rng(n)
    x = rng.random(n).astype(np.float32) + 1.0
    rows = _rows(lib, n)
    x[rows] = rng.random(len(rows)).astype(np.float32) * 1e-3
    y = np.round(rng.standard_normal(n) + 0.5 * (x - 1.0), 3).astype(np.float32)
    V, M, K = synth.OP["var"], synth.OP["mul"], synth.OP["const"]
    progs = [[(M, 0, 0.0), (K, 0, (-1.0) ** p * 2.0 ** (p % 41 - 20)), (V, 0, 0.0)] for p in range(n_progs)]
    progs[n_progs // 2] = [(V, 1, 0.0)]                # one that is not
    nodes, off = synth.pack(progs)
    X = np.stack([x, rng.standard_normal(n).astype(np.float32)])
    got = gp.gp_evaluate(gp.nodes_to_device(nodes), torch.from_numpy(off).cuda(), torch.from_numpy(X).cuda(),
                         torch.from_numpy(y).cuda(), None, "spearman").cpu().numpy()
    want = [oracle.spearman_of(c.astype(np.float64), y.astype(np.float64)) for c in X]
    want = np.where(np.arange(n_progs) == n_progs // 2, want[1], want[0])
    # the rounding of the FP32 result and of two FP64 evaluations
    np.testing.assert_allclose(got, want, rtol=1e-6, atol=1e-9)


@pytest.mark.gpu
@pytest.mark.parametrize("n", [100, 4096, 6144, 16384, 200_003, 1_000_000])
def test_repeated_values(n):
    """Values that repeat (integers, decimals, a grid's axes), alone and among
    others so close that they fall into the same bin; in each the ranks are
    the definition's."""
    import torch

    from paper_2110_11226_gb300 import gp
    rng = np.random.default_rng(n)
    r, side = np.arange(n), int(n ** 0.5)
    z = rng.standard_normal(n)
    near = 1.0 + rng.integers(0, 40, n) * 2.0 ** -23
    cols = [np.round(z, 2), rng.integers(0, 10000, n), rng.integers(0, 30, n), r % side, r // side,
            np.where(rng.random(n) < 0.9, 0.0, z), np.where(rng.random(n) < 0.5, near, 1000.0 * z),
            np.where(rng.random(n) < 0.02, 1.0 + 1e-5 * rng.random(n), np.round(1000.0 * z, 0)),
            np.round(rng.standard_normal(n) ** 5, 1)]
    X = np.stack(cols).astype(np.float32)
    y = np.round(rng.standard_normal(n) + 0.2 * X[0], 2).astype(np.float32)
    nodes, off = synth.pack([[(synth.OP["var"], f, 0.0)] for f in range(len(X))])
    got = gp.gp_evaluate(gp.nodes_to_device(nodes), torch.from_numpy(off).cuda(), torch.from_numpy(X).cuda(),
                         torch.from_numpy(y).cuda(), None, "spearman").cpu().numpy()
    want = [oracle.spearman_of(c.astype(np.float64), y.astype(np.float64)) for c in X]
    # the rounding of the FP32 result and of two FP64 evaluations
    np.testing.assert_allclose(got, want, rtol=1e-6, atol=1e-9)
