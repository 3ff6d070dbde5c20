"""Single components of the plain form's integer pair term (csrc/hh_pair64.cuh), compiled for the host.

A pair seen from its other end gives the negative of every component, to the last bit; every digit has its negative;
results keep their value down to subnormal numbers; a component that is small in every term is as good as in FP64, or
its sums are left to FP64."""
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
    return (A.bad || !S.ok) + 2 * hh::thin(A.span);
}
extern "C" void scalars(long n, const double *d, const double *m, double eps2, double *out)
{
    const hh::Soft64 S = hh::soft_of(eps2);
    for (long i = 0; i < n; i++)
        hh::pair_scalars_f64(d + 3 * i, m[i], hh::mass_bits(m[i]), S, out[3 * i], out[3 * i + 1], out[3 * i + 2]);
}
"""


@pytest.fixture(scope="module")
def pair_sums(tmp_path_factory):
    d = tmp_path_factory.mktemp("pair64")
    (d / "p.cpp").write_text(SRC)
    so = str(d / "p.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "p.cpp"), "-o", so], check=True)
    lib = C.CDLL(so)
    f = lib.pair_sums
    P = C.POINTER(C.c_double)
    lib.scalars.argtypes = [C.c_long, P, P, C.c_double, P]
    lib.scalars.restype = None
    f.argtypes = [C.c_long, P, P, P, C.c_double, C.c_int, P]

    def call(d, w, m, eps2, with_thin=False):
        d, w, m = (np.ascontiguousarray(u, dtype=np.float64) for u in (d, w, m))
        out = np.zeros(7)
        p = lambda u: u.ctypes.data_as(P)  # noqa: E731
        left = f(len(m), p(d), p(w), p(m), eps2, max(2, int(len(m)).bit_length()), p(out))
        return (out, left & 1, left >> 1) if with_thin else (out, left & 1)

    def scalars(d, m, eps2):
        d, m = np.ascontiguousarray(d), np.ascontiguousarray(m)
        out = np.zeros((len(m), 3))
        p = lambda u: u.ctypes.data_as(P)  # noqa: E731
        lib.scalars(len(m), p(d), p(m), eps2, p(out))
        return out

    call.scalars = scalars
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


def _sheet(rng, n, thick, v_thick, one_side):
    d, w = rng.normal(size=(n, 3)), rng.normal(size=(n, 3))
    d[:, 2] *= thick
    w[:, 2] *= v_thick
    if one_side:
        d[:, 2], w[:, 2] = np.abs(d[:, 2]), np.abs(w[:, 2])
    return d, w, np.exp(rng.normal(size=n))


def _component_reference(d, w, m, eps2):
    """Sums [6] in long double and the sums of the sizes of each component's own terms."""
    L = np.longdouble
    d, w, m = d.astype(L), w.astype(L), m.astype(L)
    r2 = (d * d).sum(1) + L(eps2)
    u = m / (r2 * np.sqrt(r2))
    f, v, q = u[:, None] * d, u[:, None] * w, (u * 3 * (d * w).sum(1) / r2)[:, None] * d
    return np.concatenate([f.sum(0), (v - q).sum(0)]), np.concatenate([np.abs(f).sum(0), (np.abs(v) + np.abs(q)).sum(0)])


@pytest.mark.parametrize("n", [30, 300, 2000])
@pytest.mark.parametrize("one_side", [False, True])
@pytest.mark.parametrize("places", [0, 1, 3, 5, 6, 7, 8, 9, 10, 12, 16, 24, 40, 60, 300])
def test_small_components(pair_sums, n, one_side, places):
    for seed in range(20):
        rng = np.random.default_rng([seed, n, places])
        for v in (1.0, 2.0 ** -places):
            d, w, m = _sheet(rng, n, 2.0 ** -places, v, one_side)
            got, left, thin = pair_sums(d, w, m, 1e-8, with_thin=True)
            assert not left
            ref, size = _component_reference(d, w, m, 1e-8)
            if not thin:
                # a term: about one unit in 2^58 of the vector's largest (rounding, dropped products of low digits, the
                # cut of the components); the component's largest term at most 9 places lower, its sum of sizes at
                # most two places below that ratio
                assert (np.abs(got[:6] - ref) <= 2.0 ** -46 * size).all(), (places, v, (got[:6] - ref) / size)
            # (a pair close in the sheet's plane is less thin than the sheet, and the heavier for it: not far below
            # the line among 2000 terms)
            assert thin or places < 24
            assert not thin or places > 1 or n < 300


def test_components_of_zero_are_exact(pair_sums):
    # motion in a plane, along a line, and from rest
    rng = np.random.default_rng(3)
    for zero in ([2], [0, 2]):
        d, w, m = _sheet(rng, 200, 1.0, 1.0, False)
        d[:, zero] = w[:, zero] = 0.0
        got, left, thin = pair_sums(d, w, m, 0.0, with_thin=True)
        ref, size = _component_reference(d, w, m, 0.0)
        assert not left and not thin and not got[zero].any() and not got[[3 + k for k in zero]].any()
        assert (np.abs(got[:6] - ref) <= 2.0 ** -49 * size).all()
        got, left, thin = pair_sums(d, np.zeros_like(w), m, 0.0, with_thin=True)
        assert not left and not thin and not got[3:6].any()


@pytest.mark.parametrize("eps2", [0.0, 1e-60, 1e-8, 0.3, 1e4, 1e60])
@pytest.mark.parametrize("spread", [0.0, 8.0, 40.0])
def test_scalars_alone(pair_sums, eps2, spread):
    # m / r, m / r^3 and 3 / r^2 as the thin parts' sums take them
    rng = np.random.default_rng(int(spread))
    n = 20000
    d = rng.normal(size=(n, 3)) * np.exp(spread * rng.uniform(-1, 1, (n, 1)))
    d[::7, 2] *= 1e-9
    d[::11, 1] = 0.0
    d[5] = [1.0, 0.0, 0.0]
    m = np.exp(rng.uniform(-1, 1, n) * (1.0 + spread))
    got = pair_sums.scalars(d, m, eps2)
    L = np.longdouble
    r2 = (d.astype(L) ** 2).sum(1) + L(eps2)
    p = m.astype(L) / np.sqrt(r2)
    ref = np.stack([p, p / r2, 3 / r2], axis=1)
    # the last rounding, and for m / r^3 the two units in 2^56 or more that its last product may lack (the others: in 2^60)
    assert (np.abs(got - ref) <= (2.0 ** -53 + np.array([2.0 ** -58, 2.0 ** -55 + 2.0 ** -57, 2.0 ** -58])) * ref).all()
