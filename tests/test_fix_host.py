"""Rules, tables and arithmetic of the fixed-point FP64 passes (csrc/fix.h, csrc/fix_band.h), which
compile for the host: no GPU needed."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2311_06926_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    if cxx is None or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("no host compiler or CUDA headers")
    so = str(tmp_path_factory.mktemp("fix") / "host_fix.so")
    subprocess.run([cxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-isystem", cuda,
                    os.path.join(ROOT, "tests", "host_fix.cpp"),
                    os.path.join(CSRC, "host_setup.cpp"), "-o", so], check=True)
    so = ctypes.CDLL(so)
    so.along_smem.restype = ctypes.c_longlong
    return so


@pytest.mark.parametrize("H", [1, 2, 3, 4, 5, 6])
def test_banded_passes_that_do_not_fit_are_not_offered(lib, H):
    """The passes along x1 stage the tables of whole operators: every launch that the set-up and its
    tuner can ask for (up to three operators and four lines per thread group, blocks of 128 and 256
    threads and of one line) fits a block wherever the rule offers the passes, and the rule refuses
    the sizes whose largest launch does not fit."""
    limit = 227 * 1024
    seen = set()
    for b in range(1, 2200):
        segs = (b + 7) // 8
        offered = bool(lib.fits(b, H))
        seen.add(offered)
        largest = 0
        for threads in (128, 256):
            threads = max(threads, (segs + 31) // 32 * 32)
            if threads > 256:
                largest = limit + 1
                continue
            lines = threads // segs
            for nterms, results in ((1, 1), (1, 2), (2, 2)):
                largest = max(largest, lib.along_smem(nterms + results - 1,
                                                      lines * (nterms + results), segs, H))
        assert offered == (largest <= limit), (b, H, largest)
    assert seen == {True, False}
    # the sizes that a set-up used to fail at
    for b, half in ((489, 6), (585, 5), (673, 4), (881, 3), (1265, 2)):
        assert not lib.fits(b, half)


def _ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


@pytest.mark.parametrize("zeros", ["leading", "trailing", "none"])
def test_rectangular_tables_of_a_pair_share_their_windows(lib, zeros):
    """A pass with two results loads one window: exact zeros at one end of one band must not move
    its table against the other's."""
    rng = np.random.default_rng(3)
    rows, cols, width = 21, 12, 4
    first = np.arange(rows) // 3                      # the inputs of the values
    second = first + {"leading": 1, "trailing": -1, "none": 0}[zeros]
    second = np.clip(second, 0, cols - width).astype(np.int32)
    first = np.clip(first, 0, cols - width).astype(np.int32)
    val = [rng.uniform(0.5, 1.0, (rows, width)) for _ in range(2)]
    w0 = np.zeros((2, 3), np.int32)
    dense = np.zeros((2, rows, cols))
    assert lib.rect_pair(rows, cols, width, _ptr(first), _ptr(val[0]), _ptr(second), _ptr(val[1]),
                         _ptr(w0), _ptr(dense)) == 1
    assert np.array_equal(w0[0], w0[1])
    for o, start in enumerate((first, second)):
        ref = np.zeros((rows, cols))
        for i in range(rows):
            ref[i, start[i]:start[i] + width] = val[o][i]
        assert np.abs(dense[o] - ref).max() <= 2.0 ** -53


def test_rectangular_tables_need_windows_of_eight(lib):
    """A pair whose segments read nine inputs together has no tables, though each band alone would."""
    rows, cols, width = 8, 16, 4
    a, b = np.full(rows, 0, np.int32), np.full(rows, 5, np.int32)
    val = np.ones((rows, width))
    w0, dense = np.zeros((2, 1), np.int32), np.zeros((2, rows, cols))
    args = [_ptr(val), _ptr(w0), _ptr(dense)]
    assert lib.rect_pair(rows, cols, width, _ptr(a), args[0], _ptr(b), *args) == 0
    assert lib.rect_pair(rows, cols, width, _ptr(a), args[0], _ptr(a + 4), *args) == 1
