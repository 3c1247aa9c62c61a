"""The FP64 Box-Muller pairs of csrc/normal64.cuh, compiled for the host with the hardware
reciprocal square root replaced by its documented form (the upper 32 bits of the value), against
extended precision at chosen words: both ends of every table cell, uniforms next to 0 and 1, ties
of the 53-bit uniform and its carry to 1, every sector of the angle.  Bound: five roundings (2^-53
each) of the radius -- logarithm, square root, the two sums of the rotation, the last product."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2407_12149_gb300", "csrc")

SHIM = r"""
#include <cmath>
#include <cstdint>
#include <cstring>
using std::fma;
#define __device__
#define __forceinline__ inline
struct uint4 { unsigned x, y, z, w; };
struct double2 { double x, y; };
template <typename T> static T __ldg(const T* p) { return *p; }
static double __longlong_as_double(long long v) { double d; std::memcpy(&d, &v, 8); return d; }
static long long bits(double d) { long long v; std::memcpy(&v, &d, 8); return v; }
static double __hiloint2double(int hi, int lo) { return __longlong_as_double(((long long)hi << 32) | (unsigned)lo); }
static int __double2hiint(double d) { return (int)(bits(d) >> 32); }
static int __double2loint(double d) { return (int)bits(d); }
static int __clz(int v) { return v ? __builtin_clz((unsigned)v) : 32; }
static int __clzll(long long v) { return v ? __builtin_clzll((unsigned long long)v) : 64; }
static double estimate(double t) { return __hiloint2double(__double2hiint(1.0 / std::sqrt(t)), 0); }
#define asm(...) y = estimate(t)
#include "normal64.cuh"
extern "C" void pairs(int kind, long n, const unsigned* w, double* z)
{
    for (long i = 0; i < n; ++i) {
        if (kind == 32)
            mgmc::n64::pair32(w[2 * i], w[2 * i + 1], z[2 * i], z[2 * i + 1]);
        else
            mgmc::n64::pair53(uint4{w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]}, z[2 * i], z[2 * i + 1]);
    }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("no extended precision")
    d = tmp_path_factory.mktemp("n64")
    (d / "shim.cpp").write_text(SHIM)
    (d / "cuda_runtime.h").write_text("")
    so = d / "n64.so"
    subprocess.run([gxx, "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I", str(d), "-I", CSRC, str(d / "shim.cpp"),
                    "-o", str(so)], check=True)
    L = ctypes.CDLL(str(so))
    L.pairs.argtypes = [ctypes.c_int, ctypes.c_long, ctypes.c_void_p, ctypes.c_void_p]
    return L


def _pairs(lib, kind, words):
    words = np.ascontiguousarray(words, dtype=np.uint32)
    z = np.zeros((words.shape[0], 2))
    lib.pairs(kind, words.shape[0], words.ctypes.data, z.ctypes.data)
    return z


def _check(z, u1, k2, bits):
    """u1: the double the logarithm is taken of; angle 2 pi (k2 + 1/2) 2^-bits."""
    L = np.longdouble
    r = np.sqrt(L(-2) * np.log(u1.astype(L)))
    pi = L("3.14159265358979323846264338327950288")
    a = L(2) * pi * (k2.astype(L) + L(0.5)) * L(2) ** -bits
    ref = np.stack([r * np.cos(a), r * np.sin(a)], 1)
    err = np.abs(z.astype(L) - ref).max(1)
    bad = err > 5 * L(2) ** -53 * r
    assert not bad.any(), (u1[bad][:4], k2[bad][:4], (err[bad] / r[bad])[:4])


def _cell_ends(scale_bits):
    """Integers k whose uniform (k + 1/2) 2^-scale_bits lies at either end of a cell of the table."""
    out = []
    for e in (0, -1, -2, -7):
        for c in range(129):
            z = 0.6875 + c / 256 if c <= 80 else 1.0 + (c - 80) / 128     # cell borders of [0.6875, 1.375)
            k = int(np.ldexp(min(z, 1.0) if e == 0 else z, scale_bits + e))
            out += [k - 2, k - 1, k, k + 1]
    top = (1 << scale_bits) - 1
    out += [0, 1, 2, 3, top, top - 1, top - 2, top - 3, top - 1000]
    out += [(1 << b) + d for b in range(2, scale_bits) for d in (-1, 0, 1)]
    return np.array(sorted({k for k in out if 0 <= k <= top}), dtype=np.uint64)


def _angles(bits):
    cell = 1 << (bits - 7)
    k = [s * cell + d for s in range(128) for d in (0, 1, cell // 2 - 1, cell // 2, cell - 1)]
    return np.array(k, dtype=np.uint64)


def _cross(k1, k2, seed):
    rng = np.random.default_rng(seed)
    a = np.concatenate([k1, rng.choice(k1, k2.size), rng.choice(k1, 20_000)])
    b = np.concatenate([rng.choice(k2, k1.size), k2, rng.choice(k2, 20_000)])
    return a, b


def test_pair32(lib):
    k1, k2 = _cross(_cell_ends(32), _angles(32), 1)
    r = np.random.default_rng(2).integers(0, 1 << 32, size=(200_000, 2), dtype=np.uint64)
    k1, k2 = np.concatenate([k1, r[:, 0]]), np.concatenate([k2, r[:, 1]])
    z = _pairs(lib, 32, np.stack([k1, k2], 1))
    _check(z, (k1.astype(np.float64) + 0.5) * 2.0 ** -32, k2, 32)


def test_pair53(lib):
    k1, k2 = _cross(_cell_ends(53), _angles(53), 3)
    r = np.random.default_rng(4).integers(0, 1 << 53, size=(200_000, 2), dtype=np.uint64)
    k1, k2 = np.concatenate([k1, r[:, 0]]), np.concatenate([k2, r[:, 1]])

    def words(k):
        return k >> np.uint64(21), (k & np.uint64((1 << 21) - 1)) << np.uint64(11)

    z = _pairs(lib, 53, np.stack([*words(k1), *words(k2)], 1))
    # (k + 1/2) rounded to 53 bits, ties to even: half of all draws are ties
    _check(z, (k1.astype(np.float64) + 0.5) * 2.0 ** -53, k2, 53)
    # the largest k carries to u = 1: radius 0
    assert np.all(z[k1 == (1 << 53) - 1] == 0.0) and (k1 == (1 << 53) - 1).any()
