"""Rules, tables and arithmetic of the fixed-point FP64 passes (csrc/fix.h, csrc/fix_band.h), which
compile for the host: no GPU needed."""
import ctypes
import math
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
    # far above the line
    for b, half in ((700, 6), (700, 5), (800, 4), (1000, 3), (1400, 2)):
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


M, K, MC, TC = range(4)


def _band_lines(lib, n, p, ops, x, results=1):
    """Results of the passes of the matrices `ops` for lines of x (one array per term), and the
    matrices."""
    nterms, (lines, m) = len(x), x[0].shape
    val = np.zeros((len(ops), m, m))
    y = [np.zeros((lines, m)) for _ in range(results)]
    x = [np.ascontiguousarray(t) for t in x]
    assert lib.band_lines(n, p, nterms, results, _ptr(np.array(ops, np.int32)), _ptr(val), lines,
                          _ptr(x[0]), _ptr(x[1]) if nterms > 1 else None, _ptr(y[0]),
                          _ptr(y[1]) if results > 1 else None) == p + 1
    return val, y


def _units(D, x, y, rows):
    """Error of y against sum_t D_t x_t in units of 2^-53 sum_t |D_t| |x_t|, for the given rows. The
    exact sums by math.fsum of exact products (each product as its rounding and fma remainder)."""
    worst = 0.0
    for l in range(y.shape[0]):
        for i in rows:
            terms, size = [], 0.0
            for Dt, xt in zip(D, x):
                for j in np.flatnonzero(Dt[i]):
                    terms += _product(float(Dt[i, j]), float(xt[l, j]))
                    size += abs(Dt[i, j] * xt[l, j])
            if size and not np.isnan(y[l, i]):
                worst = max(worst, abs(math.fsum(terms + [-float(y[l, i])])) / size * 2.0 ** 53)
    return worst


def _product(a, b):
    """a b as two doubles, by Dekker's splitting."""
    p = a * b
    ah = a * 134217729.0
    ah -= ah - a
    bh = b * 134217729.0
    bh -= bh - b
    al, bl = a - ah, b - bh
    return [p, ((ah * bh - p) + ah * bl + al * bh) + al * bl]


# the 1D matrices alone, then the forms of the operator's passes: two results of one input (K and M;
# T-check and M-check), two terms (M-check and T-check), two terms with two results
FORMS = [([M], 1), ([K], 1), ([MC], 1), ([TC], 1), ([K, M], 2), ([TC, MC], 2), ([MC, TC], 1),
         ([MC, TC, MC], 2)]


def _form(n, p, ops, results, rng, lines):
    nterms = len(ops) - results + 1
    m = n + p - (1 if ops[0] in (M, K) else 0)
    return [rng.uniform(0.5, 1.0, (lines, m)) * rng.choice([-1.0, 1.0], (lines, m))
            for _ in range(nterms)]


def _outputs(D, x, y):
    """(matrices, inputs, result) of each result of a pass."""
    nterms = len(x)
    out = [(D[:nterms], x, y[0])]
    if len(y) > 1:
        out.append((D[nterms:], x[-1:], y[1]))
    return out


@pytest.mark.parametrize("n,p", [(60, 1), (61, 2), (64, 3), (64, 4), (60, 5)])
@pytest.mark.parametrize("ops,results", FORMS)
def test_rows_beside_the_walls_keep_their_accuracy(lib, n, p, ops, results):
    """Every output of a pass, the small rows beside T-check's penalty row above all, is as close as
    an FMA chain is bound to be: 2^-53 per term, of sum |D| |x| over its own row. Entries of one
    magnitude, so that only the scales of the rows count."""
    x = _form(n, p, ops, results, np.random.default_rng(n + p), 40)
    D, y = _band_lines(lib, n, p, ops, x, results)
    m = D.shape[1]
    for Dt, xt, yt in _outputs(D, x, y):
        rows = [*range(16), m // 2, m // 2 + 1, *range(m - 16, m)]
        assert _units(Dt, xt, yt, rows) <= sum((np.count_nonzero(d, axis=1).max()) for d in Dt)


def _wide(name, rng, lines, m):
    x = rng.standard_normal((lines, m))
    if name == "spike":
        x[np.arange(lines), rng.integers(0, m, lines)] *= 1e6
    elif name == "falls by 4":
        x *= 4.0 ** -(np.arange(m) % 40)
    elif name == "rises by 10":
        x *= 10.0 ** (np.arange(m) % 13)
    elif name == "steps":
        x *= np.where(np.arange(m) // 5 % 2, 1.0, 1e-9)
    return x


@pytest.mark.parametrize("n,p", [(60, 1), (61, 2), (64, 3), (64, 4), (60, 5)])
@pytest.mark.parametrize("ops,results", FORMS)
@pytest.mark.parametrize("kind", ["normal", "spike", "falls by 4", "rises by 10", "steps"])
def test_entries_do_not_lose_bits_to_larger_neighbours(lib, n, p, ops, results, kind):
    """Lines of wide range: every output that the fixed-point form keeps is as close as an FMA chain
    is bound to be, 2^-53 per term of sum |D| |x| over its own row (the others it leaves to a
    chain). Of lines of one magnitude it keeps nearly all."""
    rng = np.random.default_rng(7 * n + p)
    x = [_wide(kind, rng, 12, t.shape[1]) for t in _form(n, p, ops, results, rng, 12)]
    D, y = _band_lines(lib, n, p, ops, x, results)
    for Dt, xt, yt in _outputs(D, x, y):
        bound = sum((np.count_nonzero(d, axis=1).max()) for d in Dt)
        assert _units(Dt, xt, yt, range(D.shape[1])) <= bound
        if kind == "normal":
            assert np.isnan(yt).mean() < 0.03


def _digits(v):
    """Balanced digits of ten bits, the leading one first (weight 2^50)."""
    out = []
    for _ in range(6):
        d = (v + 512) % 1024 - 512
        out.append(d)
        v = (v - d) >> 10
    return out[::-1]


@pytest.mark.parametrize("xbits", [56, 57, 58])
def test_level_sums_of_equal_entries_stay_exact(lib, xbits):
    """FP32 holds the integer sums of a level exactly up to 2^24. Lines and columns of equal entries
    (their digits too) reach the largest sums; the levels above the result's unit must be moved
    before, level 4 (the unit) may lose its last bit, and the last level's truncations stay below
    a unit."""
    rng = np.random.default_rng(xbits)
    pairs = [(int(rng.integers(2 ** (xbits - 1), 2 ** xbits)), int(rng.integers(2 ** 57, 2 ** 58)))
             for _ in range(2000)]
    # and the largest digits of one sign
    low = sum(511 << (10 * k) for k in range(5))
    pairs += [(2 ** xbits - 2 ** 50 + low, 2 ** 58 - 2 ** 50 + low)]
    for v, u in pairs:
        dv, du = _digits(v), _digits(u)
        for level in range(6):
            term = sum(dv[i] * du[level - i] for i in range(level + 1))
            peak = abs(term) * 16 * lib.level_every(level, xbits)
            if level < 5:
                assert peak <= 2 ** (24 if level < 4 else 25), (level, v, u)
            else:   # units of 2^50 against the result's 2^60
                assert 5 * 2 ** max(0, peak.bit_length() - 24) < 2 ** 10
