"""The tabulated S_m(y) = (-1)^m F_m(y / 2) of the Hermite kernels
(csrc/herm.cuh), every order, both precisions, over the whole range of y: the
near rows, the change to the far rows at y = 120, and far rows scaled by powers
of four up to y = 1e8.  Built for the host by tests/herm_host_harness.cpp, with
the library's own tables, against 40-digit values.

Bounds, relative.  FP64: the table's value and the two additions are rounded
(half a unit in the last place each, at most 3 x 2^-53 together), the tail's
double-float arithmetic adds at most 2^-53, and the first term the tail leaves
out is |S_{m+7} / S_m| z^7 / 7!.  df64: the table, the last addition and the
tail, 4 x 2^-48, and the first term left out, of order 8 (order 5 for L = 0).
|z| is at most half a grid step: 2^-7 near and 2^-5 far in FP64 (rows of y in
1/32 and 1/8, z = (y - y_i) / 2), 2^-5 in df64 (2^-8 near, 2^-7 far for L = 0).
"""
import ctypes
import os
import re
import shutil
import subprocess
import sys

import numpy as np
import pytest

mp = pytest.importorskip("mpmath")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1303_4916_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx, inc = shutil.which("g++"), "/usr/local/cuda/include"
    if not cxx or not os.path.isdir(inc):
        pytest.skip("no host C++ compiler or CUDA headers")
    from paper_1303_4916_gb300 import build
    tables = ctypes.CDLL(build.build())
    d = str(tmp_path_factory.mktemp("herm"))
    with open(os.path.join(CSRC, "herm.cuh")) as fh:
        s = fh.read()
    for pat, new in ((r'asm\("ld\.global\.nc\.v8\.b32.*?"l"\(p\)\);', "for (int k = 0; k < 8; ++k) v[k] = p[k];"),
                     (r'asm\("rsqrt\.approx\.ftz\.f64.*?\);', "y = host_rsqrt_estimate(a);"),
                     (r'asm\("ld\.global\.nc\.v4\.f64.*?\);', "")):
        s, n = re.subn(pat, new, s, flags=re.S)
        assert n >= 1, pat
    with open(os.path.join(d, "herm_host.cuh"), "w") as fh:
        fh.write(s)
    out = os.path.join(d, "libherm.so")
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", d, "-I", CSRC, "-I", inc,
                    os.path.join(ROOT, "tests", "herm_host_harness.cpp"), "-o", out], check=True)
    h = ctypes.CDLL(out)
    h.path = out
    h.t64, h.tdf = np.zeros(h.words64(), np.uint32), np.zeros(h.wordsdf(), np.uint32)
    tables._Z13hf_boysy_fillPjS_(h.t64.ctypes.data_as(ctypes.c_void_p), h.tdf.ctypes.data_as(ctypes.c_void_p))
    return h


def _S(m, y):
    T = mp.mpf(y) / 2
    f = mp.mpf(1) / (2 * m + 1) if T == 0 else mp.gammainc(m + mp.mpf(1) / 2, 0, T) / (2 * T ** (m + mp.mpf(1) / 2))
    return (-1) ** m * f


RNG = np.random.default_rng(19)
RANGES = {
    "near": np.concatenate([[0.0, 1e-300, 1e-9, 1 / 64, 1 / 32, 119.98, np.nextafter(120.0, 0)], RNG.uniform(0, 120, 40)]),
    "change": 120 + np.concatenate([[0.0, 1e-9], RNG.uniform(0, 8, 20)]),
    "far": np.concatenate([[127.9999, 128.0, 511.99, 512.0, 2047.9, 2048.0], np.exp(RNG.uniform(np.log(120), np.log(1e8), 40))]),
}


@pytest.mark.parametrize("name", sorted(RANGES))
@pytest.mark.parametrize("L", range(9))
def test_s_m_of_every_order(lib, name, L):
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    with mp.workdps(40):
        for y in RANGES[name]:
            y = float(y)
            s, d = np.zeros(L + 1), np.zeros(2 * L + 2, np.float32)
            lib.s_all(L, p(lib.t64), p(lib.tdf), ctypes.c_double(y), p(s), p(d))
            yd = float(np.float32(y)) + float(np.float32(y - float(np.float32(y))))
            far = y >= 120
            # far rows: of the argument scaled into [32, 128), where the terms left out are relative to the row's
            base = y
            while far and base >= 128:
                base /= 4
            for m in range(L + 1):
                ratio = lambda k: abs(_S(m + k, base) / _S(m, base))  # noqa: E731
                want = _S(m, y)
                z = 2.0 ** -5 if far else 2.0 ** -7
                tol = 4 * 2.0 ** -53 + ratio(7) * z ** 7 / 5040
                assert abs(mp.mpf(float(s[m])) - want) <= tol * abs(want), (L, m, y)
                want = _S(m, yd)
                if L == 0:
                    tol = 4 * 2.0 ** -48 + ratio(5) * (2.0 ** -7 if far else 2.0 ** -8) ** 5 / 120
                else:
                    tol = 4 * 2.0 ** -48 + ratio(8) * 2.0 ** -40 / 40320
                got = mp.mpf(float(d[2 * m])) + mp.mpf(float(d[2 * m + 1]))
                # below the range of floats the value is a power of T that no sum can see
                assert abs(got - want) <= tol * abs(want) + mp.mpf(2) ** -120, (L, m, y, "df64")


def test_rsqrt_of_every_exponent(lib):
    """hf_rsqrt: the 21-bit estimate and a third-order correction, within 1.5 units of 2^-53."""
    lib.rsqrt64.restype = ctypes.c_double
    with mp.workdps(40):
        for a in np.concatenate([np.exp(RNG.uniform(np.log(1e-30), np.log(1e30), 300)), [1.0, 2.0, 4.0, 0.25, np.nextafter(1.0, 0)]]):
            got = lib.rsqrt64(ctypes.c_double(float(a)))
            assert abs(mp.mpf(got) * mp.sqrt(mp.mpf(float(a))) - 1) <= 1.5 * 2.0 ** -53


CHILD = """
import ctypes, sys
import numpy as np
h, t = ctypes.CDLL(sys.argv[1]), np.load(sys.argv[2])
p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
for L in range(9):
    for y in (1e38, 3.5e38, 1e200, float("inf"), float("nan")):
        s, d = np.zeros(L + 1), np.zeros(2 * L + 2, np.float32)
        h.s_all(L, p(t["t64"]), p(t["tdf"]), ctypes.c_double(y), p(s), p(d))
        assert not y <= 1e38 or np.all(np.abs(d[::2]) <= 2.0 ** -60), (L, y, d)
print("ok")
"""


def test_arguments_beyond_the_range_of_floats_stay_in_the_tables(lib, tmp_path):
    """Centres 1e16 bohr apart are accepted; y = 2T then overflows a float, and the row index with it.
    In a child process: an index out of range ends it."""
    np.savez(tmp_path / "t.npz", t64=lib.t64, tdf=lib.tdf)
    r = subprocess.run([sys.executable, "-c", CHILD, lib.path, str(tmp_path / "t.npz")], capture_output=True, text=True)
    assert r.returncode == 0 and "ok" in r.stdout, r.stderr[-500:]
