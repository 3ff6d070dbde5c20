"""The plain form's integer pair term (csrc/hh_pair64.cuh) compiled for the host, against long double.

Softening, separation, velocity and mass each over a wide range: no error above the FP64 expression's bound, sums of
terms of very different sizes, exact zeros, and the terms that are left to FP64 (out of range, a mass that is not
positive, coincident points without softening)."""
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


def _reference(d, w, m, eps2):
    """Terms [n, 7] in long double, and the sizes that their errors are measured by."""
    L = np.longdouble
    d, w, m = d.astype(L), w.astype(L), m.astype(L)
    r2 = (d * d).sum(1) + L(eps2)
    rw = (d * w).sum(1)
    p = m / np.sqrt(r2)
    u = p / r2
    t = np.concatenate([u[:, None] * d, u[:, None] * (w - 3 * (rw / r2)[:, None] * d), p[:, None]], axis=1)
    nd, nw = np.sqrt((d * d).sum(1)), np.sqrt((w * w).sum(1))
    return t, np.stack([u * nd] * 3 + [u * nw] * 3 + [p], axis=1)


@pytest.mark.parametrize("eps2", [0.0, 1e-20, 1e-8, 0.05, 0.3, 1.0, 3.0, 1e6])
@pytest.mark.parametrize("spread", [0.0, 3.0, 12.0])
def test_each_pair_within_fp64_rounding(pair_sums, eps2, spread):
    rng = np.random.default_rng(int(spread) + 7)
    n = 400
    d = rng.normal(size=(n, 3)) * np.exp(spread * rng.uniform(-1, 1, (n, 1)))
    w = rng.normal(size=(n, 3)) * np.exp(spread * rng.uniform(-1, 1, (n, 1)))
    d[::17, 1] = 0.0
    d[5] = 0.0 if eps2 else d[5]
    w[3::19] = 0.0
    m = np.exp(rng.uniform(-8, 8, n))
    ref, size = _reference(d, w, m, eps2)
    for i in range(n):
        got, left = pair_sums(d[i:i + 1], w[i:i + 1], m[i:i + 1], eps2)
        assert not left
        # the last rounding (2^-53 of the value) and units in 2^-55 of the force and of |u w|: 2^-51 in all
        assert (np.abs(got - ref[i]) <= 2.0 ** -51 * size[i]).all(), (i, got, ref[i])


@pytest.mark.parametrize("n", [1, 2, 63, 1000, 5000])
@pytest.mark.parametrize("spread", [0.0, 10.0])
def test_sums_of_terms_of_many_sizes(pair_sums, n, spread):
    rng = np.random.default_rng(n)
    d = rng.normal(size=(n, 3)) * np.exp(spread * rng.uniform(-1, 1, (n, 1)))
    w, m = rng.normal(size=(n, 3)), np.exp(rng.uniform(-3, 3, n))
    for order in (np.arange(n), np.argsort((d * d).sum(1)), np.argsort(-(d * d).sum(1))):
        ref, size = _reference(d[order], w[order], m[order], 1e-8)
        got, left = pair_sums(d[order], w[order], m[order], 1e-8)
        assert not left
        # each term's own error plus one unit below the largest term's 2^-62 per term
        assert (np.abs(got - ref.sum(0)) <= 2.0 ** -51 * size.sum(0)).all()


@pytest.mark.parametrize("what", ["far", "fast", "zero mass", "negative mass", "large mass", "coincident", "nan", "inf",
                                  "eps inf", "eps tiny"])
def test_what_is_left_to_fp64(pair_sums, what):
    d, w, m, eps2 = np.ones((1, 3)), np.ones((1, 3)), np.ones(1), 1e-8
    if what == "far":
        d[0, 1] = 1e70
    elif what == "fast":
        w[0, 2] = -1e70
    elif what == "zero mass":
        m[0] = 0.0
    elif what == "negative mass":
        m[0] = -1.0
    elif what == "large mass":
        m[0] = 1e70
    elif what == "coincident":
        d[:], eps2 = 0.0, 0.0
    elif what == "nan":
        d[0, 0] = np.nan
    elif what == "inf":
        w[0, 0] = np.inf
    elif what == "eps inf":
        eps2 = np.inf
    elif what == "eps tiny":
        eps2 = 1e-200
    assert pair_sums(d, w, m, eps2)[1]
