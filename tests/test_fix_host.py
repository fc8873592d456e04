"""Rules, tables and arithmetic of the fixed-point FP64 passes (csrc/fix.h, csrc/fix_band.h), which
compile for the host: no GPU needed."""
import ctypes
import os
import shutil
import subprocess

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
