"""Single components of the plain form's integer pair term (csrc/hh_pair64.cuh), compiled for the host.

A pair seen from its other end gives the negative of every component, to the last bit; every digit has its negative."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1602_02832_gb300", "csrc")
SRC = r"""
#include "hh_pair64.cuh"
extern "C" int pair_sums(long n, const double *d, const double *w, const double *m, double eps2, int smin, double *out)
{
    hh::AccI64 A;
    A.zero();
    const hh::Soft64 S = hh::soft_of(eps2);
    for (long i = 0; i < n; i++) hh::pair_add(d + 3 * i, w + 3 * i, m[i], hh::mass_bits(m[i]), false, S, smin, A);
    for (int k = 0; k < 3; k++) {
        out[k] = hh::sum_get(A.a.u[k], A.a.o[k], A.a.e);
        out[3 + k] = hh::sum_get(A.j.u[k], A.j.o[k], A.j.e);
    }
    out[6] = hh::sum_get(A.p.u[0], A.p.o[0], A.p.e);
    return A.bad || !S.ok;
}
"""


@pytest.fixture(scope="module")
def pair_sums(tmp_path_factory):
    d = tmp_path_factory.mktemp("pair64")
    (d / "p.cpp").write_text(SRC)
    so = str(d / "p.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "p.cpp"), "-o", so], check=True)
    f = C.CDLL(so).pair_sums
    P = C.POINTER(C.c_double)
    f.argtypes = [C.c_long, P, P, P, C.c_double, C.c_int, P]

    def call(d, w, m, eps2):
        d, w, m = (np.ascontiguousarray(u, dtype=np.float64) for u in (d, w, m))
        out = np.zeros(7)
        p = lambda u: u.ctypes.data_as(P)  # noqa: E731
        left = f(len(m), p(d), p(w), p(m), eps2, max(2, int(len(m)).bit_length()), p(out))
        return out, left

    return call


@pytest.mark.parametrize("eps2", [0.0, 1e-8, 0.3, 1e4])
@pytest.mark.parametrize("kind", ["any", "lattice", "thin", "at rest"])
def test_a_pair_from_its_other_end(pair_sums, eps2, kind):
    rng = np.random.default_rng(17)
    n = 3000
    d, w = (rng.normal(size=(n, 3)) * np.exp(3 * rng.normal(size=(n, 3))) for _ in range(2))
    if kind == "lattice":  # few significant bits, zeros, negative zeros
        d, w = np.round(8 * d) / 8, np.round(8 * w) / 8
        d[(d == 0).all(1)] = 0.125
    elif kind == "thin":
        d[:, 2] *= 1e-9
        w[:, 1] *= 1e-7
    elif kind == "at rest":
        w[:] = 0.0
        w[::2] = -0.0
    m = np.exp(rng.normal(size=n))
    for i in range(n):
        a, left = pair_sums(d[i:i + 1], w[i:i + 1], m[i:i + 1], eps2)
        b, _ = pair_sums(-d[i:i + 1], -w[i:i + 1], m[i:i + 1], eps2)
        assert not left
        assert np.array_equal(a[:6], -b[:6]) and a[6] == b[6], (i, a, b)
        if kind == "at rest":
            assert not a[3:6].any()


def test_a_digit_without_a_negative(pair_sums):
    # found by search (one pair in 2^32): the jerk's factor of the separation has the low digit -2^31
    h = [float.fromhex(s) for s in ("0x1.821fa0ffd6076p-1", "0x1.6f6334dacc0ap-4", "-0x1.f74ed4f41876p-5",
                                    "0x1.e940d71cb38b8p-1", "-0x1.e8e0238142a64p-1", "-0x1.fc7cb8a0e6c4cp-2")]
    d, w = np.array(h[:3], dtype=np.longdouble), np.array(h[3:], dtype=np.longdouble)
    r2 = (d * d).sum()
    u = 1 / (r2 * np.sqrt(r2))
    jerk = u * (w - 3 * (d * w).sum() / r2 * d)
    got, left = pair_sums(d[None], w[None], np.ones(1), 0.0)
    assert not left
    # as in every pair: 2^-51 of |u w|
    assert (np.abs(got[3:6] - jerk) <= 2.0 ** -51 * u * np.sqrt((w * w).sum())).all()


@pytest.mark.parametrize("scale", [-250, -306, -312, -320, -330, -334, -345, -380, -386, -420])
def test_results_near_the_end_of_the_range(pair_sums, scale):
    # the jerk of a light pair far away and nearly at rest, down to subnormal numbers and zero
    d, w, m = np.array([[1.5, -0.75, 0.3]]) * 2.0 ** 170, np.array([[0.3, 0.2, -1.1]]) * 2.0 ** scale, np.array([1.25 * 2.0 ** -180])
    e = 2.0 ** -1074
    L = np.longdouble
    D, W = d[0].astype(L), w[0].astype(L)
    r2 = (D * D).sum()
    u = L(m[0]) / (r2 * np.sqrt(r2))
    ref = np.concatenate([u * D, u * (W - 3 * (D * W).sum() / r2 * D)])
    size = np.array([u * np.sqrt(r2)] * 3 + [u * np.sqrt((W * W).sum())] * 3)
    got, left = pair_sums(d, w, m, 0.0)
    assert not left
    # 2^-51 of the sizes, or the spacing of subnormal numbers (two roundings)
    assert (np.abs(got[:6] - ref) <= 2.0 ** -51 * size + 2 * e).all()
