"""The integer sum of a float pair (dbl_of_pair in tt_df.h, compiled for the
host) is (double)hi + (double)lo to one unit in the last place (rounded to nearest
after dropping less than half a unit), and the same bits where the sum is below
2^-71, zero of either sign, infinite or NaN: over random pairs of every exponent
distance, at powers of two, halfway cases, FP32 subnormals (alone, as remainder,
as sum) and overflow."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2212_11973_gb300", "csrc")


@pytest.fixture(scope="module")
def pairs(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    inc = "/usr/local/cuda/include"
    if not cxx or not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("no C++ compiler or CUDA headers")
    out = str(tmp_path_factory.mktemp("pair") / "libpair.so")
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, "-I", inc,
                    os.path.join(ROOT, "tests", "host", "pair_harness.cpp"), "-o", out], check=True)
    lib = C.CDLL(out)

    def run(hi, lo):
        hi, lo = np.ascontiguousarray(hi, np.float32), np.ascontiguousarray(lo, np.float32)
        v = np.empty(hi.size)
        f, d = C.POINTER(C.c_float), C.POINTER(C.c_double)
        lib.h_pairs(hi.ctypes.data_as(f), lo.ctypes.data_as(f), v.ctypes.data_as(d), C.c_int64(hi.size))
        return v

    run.lib = lib
    return run


def _same(got, hi, lo):
    with np.errstate(all="ignore"):
        want = hi.astype(np.float64) + lo.astype(np.float64)
        s = hi + lo
    loose = np.isfinite(s) & (np.abs(s) >= 2.0 ** -71)
    off = np.abs(got.view(np.int64) - want.view(np.int64))
    bad = np.where(loose, off > 1, (off != 0) & ~(np.isnan(got) & np.isnan(want)))
    assert not bad.any(), [(float(a).hex(), float(b).hex(), float(g).hex()) for a, b, g in
                           zip(hi[bad][:5], lo[bad][:5], got[bad][:5])]


def test_random_pairs(pairs):
    rng = np.random.default_rng(1)
    n = 400000
    hi = np.ldexp(rng.uniform(1, 2, n) * rng.choice([-1, 1], n), rng.integers(-126, 127, n)).astype(np.float32)
    for spread in (0, 3, 24, 30, 45, 60, 80):
        d = rng.integers(max(0, spread - 30), spread + 1, n)
        lo = (hi.astype(np.float64) * np.ldexp(rng.uniform(-1, 1, n), -d)).astype(np.float32)
        _same(pairs(hi, lo), hi, lo)


def test_edges(pairs):
    rng = np.random.default_rng(2)
    tiny = np.float32(2.0) ** -149
    v = [0.0, -0.0, tiny, -tiny, 5 * tiny, np.float32(2.0) ** -126, np.float32(2.0) ** -126 - tiny, np.inf, -np.inf,
         np.nan, np.finfo(np.float32).max, -np.finfo(np.float32).max, 1.0, -1.0, np.float32(2.0) ** -100]
    v += [np.float32(2.0) ** e for e in range(-148, 128, 7)] + [np.float32(1 + 2.0 ** -23) * np.float32(2.0) ** e
                                                                for e in range(-120, 127, 9)]
    v = np.array(v + [-x for x in v], np.float32)
    hi, lo = (a.reshape(-1) for a in np.meshgrid(v, v))
    _same(pairs(hi, lo), hi, lo)
    # remainders of 30 and fewer bits beyond the 53 kept: halfway and next to it
    s = np.ldexp(rng.integers(2 ** 23, 2 ** 24, 200000).astype(np.float64), -23).astype(np.float32)
    s[::3] = 1.0
    t = (rng.integers(0, 64, s.size) - 32) * 2.0 ** -54
    t += rng.integers(-3, 4, s.size) * 2.0 ** -24
    lo = t.astype(np.float32)
    _same(pairs(s, lo), s, lo)
    sub = (rng.integers(-2 ** 23, 2 ** 23, 200000) * 2.0 ** -149).astype(np.float32)
    near = (rng.integers(-2 ** 27, 2 ** 27, sub.size) * 2.0 ** -149).astype(np.float32)
    _same(pairs(near, sub), near, sub)


def _f64(a):
    return a.ctypes.data_as(C.POINTER(C.c_double))


@pytest.fixture(scope="module")
def lib(pairs):
    return pairs.lib


def test_roots_of_pairs(lib):
    """1 / sqrt(d) and sqrt(d) of a pair from a float seed up to 2 ulp off: e = 1 - d
    y^2 is known to 2^-48 (three roundings of terms below 2^-24), half of it and the
    roundings of the last two sums (2^-48 each) and of d to a pair (2^-47, half of it
    in the root): 2^-46 in all."""
    n = 200000
    d = np.exp(np.random.default_rng(4).uniform(-20, 20, n))
    root = np.sqrt(d.astype(np.longdouble))
    for off in range(-2, 3):
        r, rl, s, sl = (np.empty(n) for _ in range(4))
        lib.h_roots(_f64(d), off, _f64(r), _f64(rl), _f64(s), _f64(sl), C.c_int64(n))
        assert np.abs((r.astype(np.longdouble) + rl) * root - 1).max() <= 2.0 ** -46
        assert np.abs((s.astype(np.longdouble) + sl) / root - 1).max() <= 2.0 ** -46


def test_rank8_update(lib):
    """a - sum of 8 products on pairs of exact 46-bit values, normalised after each
    term: the low part stays below 2^-24 of the partial sum and takes three roundings
    a term, each of rms 2^-24 2^-24 / sqrt(12) of the largest of them: sqrt(24) of
    them give 2^-48.5 of the largest, 2^-50 of the sum of the magnitudes (8 terms
    of like size); doubled for the seven partial sums above the mean.  Left
    unnormalised, the low part grows with the terms: 2^-48.8."""
    rng = np.random.default_rng(5)
    n = 200000
    a, b, c = (np.rint(rng.standard_normal(k) * 2.0 ** 42) * 2.0 ** -42 for k in (n, 8 * n, 8 * n))
    out = np.empty(n)
    lib.h_rank8(_f64(a), _f64(b), _f64(c), _f64(out), C.c_int64(n))
    x = np.longdouble
    want = a.astype(x) - (b.astype(x) * c.astype(x)).reshape(n, 8).sum(1)
    scale = np.abs(a) + np.abs(b * c).reshape(n, 8).sum(1)
    err = ((out - want) / scale).astype(float)
    assert np.sqrt((err ** 2).mean()) <= 2.0 ** -49
