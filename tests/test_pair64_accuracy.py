"""Accuracy of the integer forms of the FP64 pair terms (csrc/pair64.cuh, host
side) against long double arithmetic, whose own roundings (2^-64 each, or less)
stay below 2^-59 here.

A force or an energy adds its terms at 2^-56 of the largest and is rounded once:
with a half unit of 2^-53 for that and at most two units of r^-12's error, two and
a half units of the terms' magnitudes.  A fixed-point difference becomes a
double by one rounding.
"""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include <cmath>
#include <cstdint>
#define __host__
#define __device__
#define __forceinline__ inline
#include "pair64.cuh"
using namespace ffm;
typedef long double ld;
static void up(double &m, ld e) { if (std::fabs((double)e) > m) m = std::fabs((double)e); }
// fixed-point differences as doubles: the number that is not rounded once
extern "C" int differences(const double *d, int n) {
    int bad = 0;
    for (int i = 0; i < n; i++) {
        const double *p = d + 3 * i;
        Inv64 v;
        long long f[3];
        u64 a[3];
        int s;
        for (int k = 0; k < 3; k++)
            if (!fix64(p[k], f[k])) return -1;
        if (!inv64_fix(f[0], f[1], f[2], v, a[0], a[1], a[2], s)) continue;
        for (int k = 0; k < 3; k++) {
            const ld x = std::ldexp((ld)f[k], -54);
            if (std::fabs((double)((ld)fix_to_double(a[k], s, f[k]) - x)) > std::ldexp(std::fabs((double)x), -53)) bad++;
        }
    }
    return bad;
}
// p: q, c6, c12 of both atoms; out: largest errors of the force over r and of six
// times the energy, in units of the sums of their terms' magnitudes
extern "C" int pair_terms(const double *d, const double *p, int n, double *out) {
    int used = 0;
    for (int i = 0; i < n; i++) {
        const double *x = d + 3 * i, *a = p + 6 * i, *b = a + 3;
        Inv64 v;
        if (!inv64(x[0], x[1], x[2], v)) continue;
        u64 m[6];
        int e[6];
        bool ok = true;
        for (int k = 0; k < 3; k++) ok = split64(a[k], m[k], e[k]) && split64(b[k], m[3 + k], e[3 + k]) && ok;
        if (!ok) return -1;
        const uint32_t neg = (a[0] < 0) != (b[0] < 0) ? 0x80000000u : 0u;
        double f, y;
        inv64_force(v, m[0], m[3], e[0] + e[3], neg, m[1], m[4], e[1] + e[4], m[2], m[5], e[2] + e[5], f, y);
        const ld r2 = 1.0L / ((ld)x[0] * x[0] + (ld)x[1] * x[1] + (ld)x[2] * x[2]), r6 = r2 * r2 * r2;
        const ld c = (ld)a[0] * b[0] * std::sqrt(r2), t6 = (ld)a[1] * b[1] * r6, t12 = (ld)a[2] * b[2] * r6 * r6;
        up(out[0], (f - (c + 2 * t12 - t6) * r2) / ((std::fabs(c) + 2 * t12 + t6) * r2));
        up(out[1], (y - (6 * c + t12 - t6)) / (6 * std::fabs(c) + t12 + t6));
        used++;
    }
    return used;
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("pair64")
    (d / "host.cpp").write_text(SOURCE)
    subprocess.run([gxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_1810_03358_gb300", "csrc"), "-o", str(d / "host.so"),
                    str(d / "host.cpp")], check=True, capture_output=True, text=True)
    return C.CDLL(str(d / "host.so"))


def ptr(a):
    return a.ctypes.data_as(C.POINTER(C.c_double))


def differences(kind, n, rng):
    u = rng.normal(size=(n, 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    if kind == "box":       # an ordinary system's
        return rng.uniform(-200.0, 200.0, size=(n, 3))
    if kind == "near":      # from bonded neighbours up to a few A
        return u * rng.uniform(0.3, 4.0, size=(n, 1))
    if kind == "axes":      # along an axis, or nearly
        d = u * 10.0 ** rng.uniform(-18, 0, size=(n, 3))
        d[np.arange(n), rng.integers(0, 3, size=n)] = 10.0 ** rng.uniform(-0.5, 2.2, size=n)
        return d
    # powers of two and their neighbours: the ends of the significands' ranges
    d = 2.0 ** rng.integers(-1, 7, size=(n, 3)) * (1.0 + rng.integers(-2, 3, size=(n, 3)) * 2.0 ** -52)
    return d * rng.choice([-1.0, 1.0], size=(n, 3))


@pytest.mark.parametrize("kind", ["box", "near", "axes", "powers"])
def test_fixed_point_differences_are_rounded_once(host, kind):
    n = 300000
    d = np.ascontiguousarray(differences(kind, n, np.random.default_rng(11)))
    assert host.differences(ptr(d), n) == 0


@pytest.mark.parametrize("kind", ["box", "near", "axes"])
@pytest.mark.parametrize("zero", [None, 0, 1, 2])
def test_forces_and_energies(host, kind, zero):
    n = 200000
    rng = np.random.default_rng(13)
    d = np.ascontiguousarray(differences(kind, n, rng))
    p = np.empty((n, 2, 3))
    p[:, :, 0] = rng.uniform(-15.0, 15.0, size=(n, 2))
    sigma, w = rng.uniform(2.0, 4.0, size=(n, 2)), np.sqrt(24.0 * rng.uniform(0.01, 0.3, size=(n, 2)))
    p[:, :, 1], p[:, :, 2] = w * sigma ** 3, w * sigma ** 6
    if zero is not None:
        p[:, 1, zero] = 0.0
    out = np.zeros(2)
    assert host.pair_terms(ptr(d), ptr(np.ascontiguousarray(p)), n, ptr(out)) > 0.9 * n
    assert np.all(out <= 2.5 * 2.0 ** -53), out * 2.0 ** 53
