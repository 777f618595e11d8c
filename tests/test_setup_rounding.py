"""The setup kernels' TTI coefficients and b (csrc/twofloat.cuh, built for the host) against the
same quantities in extended precision: n and sqrt(1 + 2 delta) are the FP64 values rounded once
to FP32, as far as FP64 itself decides the rounding (2^-50 of the value; its functions and one
product are within 2^-51), b to 2^-44."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1807_03032_gb300", "csrc")

WRAP = """
#include "twofloat.cuh"
using namespace fdsweep;
extern "C" void axis(const float *th, const float *ph, float *n, long count) {
    for (long i = 0; i < count; ++i) axis_of(th[i], ph[i], n + 3 * i, n + 3 * i + 1, n + 3 * i + 2);
}
extern "C" long undecided(const float *th, const float *ph, long count) {
    long k = 0;
    for (long i = 0; i < count; ++i) {
        TwoFloat st, ct, sp, cp;
        float f;
        bool ok = sincos_two_float(th[i], &st, &ct);
        ok &= sincos_two_float(ph[i], &sp, &cp);
        ok &= rounds_surely(tf_mul(st, cp), &f);
        ok &= rounds_surely(tf_mul(st, sp), &f);
        ok &= rounds_surely(ct, &f);
        k += !ok;
    }
    return k;
}
extern "C" void root(const float *d, float *s, long count) {
    for (long i = 0; i < count; ++i) s[i] = anellipticity_root(d[i]);
}
extern "C" void quotient(const float *m, double dt, float *b, long count) {
    const float A = (float)(dt * dt), a = (float)(dt * dt - (double)A);
    for (long i = 0; i < count; ++i) b[i] = div_two_float_rn(A, a, m[i], 0.f);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("twofloat")
    src, so = str(d / "tf.cpp"), str(d / "tf.so")
    with open(src, "w") as f:
        f.write(WRAP)
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-std=c++17", "-shared", "-fPIC", "-I",
                    CSRC, src, "-o", so], check=True)
    lib = ctypes.CDLL(so)
    lib.undecided.restype = ctypes.c_long
    return lib


P = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731


def assert_rounded(got, exact, slack):
    """got is exact (long double) rounded to FP32, or exact lies within slack of its size of
    the midpoint between got and the nearest float."""
    want = exact.astype(np.float32)
    off = np.flatnonzero(got != want)
    mid = (got[off].astype(np.longdouble) + want[off].astype(np.longdouble)) / 2
    far = np.abs(exact[off] - mid) > np.abs(exact[off]) * slack
    assert not far.any(), (got[off][far][:4], want[off][far][:4])


def axis(lib, th, ph):
    th, ph = np.ascontiguousarray(th, np.float32), np.ascontiguousarray(ph, np.float32)
    n = np.empty(th.shape + (3,), np.float32)
    lib.axis(P(th), P(ph), P(n), ctypes.c_long(th.size))
    t, p = th.astype(np.longdouble), ph.astype(np.longdouble)
    return n, (np.sin(t) * np.cos(p), np.sin(t) * np.sin(p), np.cos(t))


@pytest.mark.parametrize("reach", [1e-3, np.pi / 4, 2 * np.pi, 40.0, 1000.0, 3e5])
def test_axis_is_the_64_bit_value_rounded_once(lib, reach):
    rng = np.random.default_rng(int(reach * 1000))
    th, ph = rng.uniform(-reach, reach, (2, 1000000))
    n, exact = axis(lib, th, ph)
    for c in range(3):
        assert_rounded(n[:, c], exact[c], 2.0 ** -50)


def test_axis_at_special_angles(lib):
    k = np.arange(-636, 637)
    quarter = (k * np.pi / 2).astype(np.float32)
    near = [quarter]
    for _ in range(3):
        near += [np.nextafter(near[-1], np.float32(np.inf))]
    near += [np.nextafter(quarter, np.float32(-np.inf))]
    tiny = np.float32([0.0, 1e-45, 1e-40, 1e-38, 1e-30, 1e-20, 1e-10, 1e-5, 999.9999, 1000.0])
    a = np.concatenate(near + [tiny, -tiny])
    th, ph = (v.ravel() for v in np.meshgrid(a[::7], np.concatenate([a[::11], tiny])))
    n, exact = axis(lib, th, ph)
    for c in range(3):
        normal = np.abs(exact[c]) >= 2.0 ** -126
        assert_rounded(n[normal, c], exact[c][normal], 2.0 ** -50)
        # subnormal floats are 2^-149 apart
        assert np.all(np.abs(n[~normal, c] - exact[c][~normal]) <= 2.0 ** -150 * (1 + 2.0 ** -20))
    zero = np.zeros(4, np.float32)
    n, _ = axis(lib, zero, np.float32([0.0, 1.0, -2.0, 3.0]))
    assert np.array_equal(n, np.tile(np.float32([0, 0, 1]), (4, 1)))


def test_few_angles_need_64_bits(lib):
    th, ph = np.random.default_rng(5).uniform(-2 * np.pi, 2 * np.pi,
                                              (2, 1000000)).astype(np.float32)
    # three components, a window of 2^-41 of the size in a unit of at least 2^-24 of it
    assert lib.undecided(P(th), P(ph), ctypes.c_long(th.size)) <= 3 * 2.0 ** -17 * th.size * 1.5


def test_right_angles_do_not_need_64_bits(lib):
    """A horizontal axis (theta = 90 degrees) or one along a grid axis is a whole model's value."""
    for th in np.float32([0.0, np.pi / 2, np.pi, -np.pi / 2]):
        for ph in np.float32([0.0, np.pi / 2, np.pi, 1.5 * np.pi, 2 * np.pi, -np.pi / 2]):
            a, b = np.full(4, th, np.float32), np.full(4, ph, np.float32)
            assert lib.undecided(P(a), P(b), ctypes.c_long(4)) == 0, (th, ph)
    k = (np.arange(-4, 5) * np.pi / 2).astype(np.float32)
    near = np.concatenate([k] + [k + s * np.spacing(np.abs(k)) for s in range(-40, 41)])
    n, exact = axis(lib, *(v.ravel() for v in np.meshgrid(near, near)))
    for c in range(3):
        normal = np.abs(exact[c]) >= 2.0 ** -126
        assert_rounded(n[normal, c], exact[c][normal], 2.0 ** -50)


def test_root_is_the_64_bit_value_rounded_once(lib):
    rng = np.random.default_rng(9)
    d = np.concatenate([rng.uniform(-0.5, 0.5, 2000000), rng.uniform(-0.5, -0.49, 200000),
                        10.0 ** rng.uniform(-30, 38, 200000), np.arange(-64, 200) / 128.0,
                        [-0.5, np.nextafter(np.float32(-0.5), np.float32(0)), 0.0, 3e38]])
    d = d.astype(np.float32)
    s = np.empty_like(d)
    lib.root(P(d), P(s), ctypes.c_long(d.size))
    assert_rounded(s, np.sqrt(1 + 2 * d.astype(np.longdouble)), 2.0 ** -50)


def test_b_without_damping_is_rounded_once(lib):
    rng = np.random.default_rng(11)
    for dt in (0.123456789, 1.0, 1.604987, 3.9):
        m = (rng.uniform(1.0, 6.0, 1000000) ** -2).astype(np.float32)
        b = np.empty_like(m)
        lib.quotient(P(m), ctypes.c_double(dt), P(b), ctypes.c_long(m.size))
        assert_rounded(b, np.longdouble(dt * dt) / m.astype(np.longdouble), 2.0 ** -44)
