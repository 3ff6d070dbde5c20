"""Single components of the plain form's integer pair term (csrc/hh_pair64.cuh), compiled for the host.

A pair seen from its other end gives the negative of every component, to the last bit."""
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
