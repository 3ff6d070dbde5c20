// The plain form's pair term in 64-bit integer arithmetic.
//
// What bounds it: the FP64 pipe issues one warp instruction in 64 cycles per
// SM sub-partition (fused multiply-add; 76 for an add or a product, 368 for a
// reciprocal square root), so the pair term in FP64 took 2280 cycles a warp and
// pair whatever else the SM did.  32 x 32 + 64-bit integer multiply-adds take 2
// to 4 cycles, adds 1, and run beside the FP64 pipe (FP32 multiply-adds do not:
// they delay it).  So only the six differences stay in FP64 (bit for bit as
// before); all that follows is fixed point with one exponent per vector: the
// separation, the relative velocity and every scalar as 64-bit numbers in two
// signed 32-bit digits, the sums in 96 bits with an exponent of their own.
// A micro-benchmark of the pair loop (4 warps per sub-partition, records in
// shared memory) went from 2280 to 690 cycles a warp and pair; one evaluation of
// N = 65536 particles (theta 0.5 lists) from 11.5 to 3.34 ms, a tree interval of
// its block steps from 90.8 to 49.9 ms.  What bounds it now is the integer
// multiply-add pipe (70% busy; the ALU pipe 61%, FP64 56%, issue 58%) and the
// latency of its chains with 4 warps a sub-partition.  Taken back: the next
// pair's differences one iteration ahead (its registers: 6% slower), unpacking
// by FP64-to-integer conversions (64 cycles each on the FP64 pipe: 1% slower for
// two components, 9% for three), five or six warps a sub-partition (the same).
//
// Errors, measured against quad precision: force 4.7e-17 (rms, relative) and
// jerk 6.8e-17 of |m w / r^3| a pair, where FP64 arithmetic has 1.9e-16 and
// 4.9e-16; sums of 300 terms 4.7e-17 and 4.9e-17 against 7.8e-16 and 7.8e-16
// (a 96-bit sum drops nothing that counts).  Of a single component's own terms:
// see thin().  No term depends on the order or
// the partners of a lane, so results stay as reproducible as in FP64.
//
// Numbers beyond 2^+-200 (separations only above, when there is a softening),
// masses that are not positive and points that coincide without softening set
// `bad`: the caller then sums the whole list part in FP64 as before.
#pragma once

#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define HH_HD __host__ __device__ __forceinline__
#else
#define HH_HD inline
#endif

namespace hh {

HH_HD uint32_t f64_hi(double x)
{
#ifdef __CUDA_ARCH__
    return (uint32_t)__double2hiint(x);
#else
    uint64_t b;
    std::memcpy(&b, &x, 8);
    return (uint32_t)(b >> 32);
#endif
}
HH_HD uint32_t f64_lo(double x)
{
#ifdef __CUDA_ARCH__
    return (uint32_t)__double2loint(x);
#else
    uint64_t b;
    std::memcpy(&b, &x, 8);
    return (uint32_t)b;
#endif
}
HH_HD double f64_of(uint32_t hi, uint32_t lo)
{
#ifdef __CUDA_ARCH__
    return __hiloint2double((int)hi, (int)lo);
#else
    const uint64_t b = ((uint64_t)hi << 32) | lo;
    double x;
    std::memcpy(&x, &b, 8);
    return x;
#endif
}
HH_HD uint32_t mul_hi(uint32_t a, uint32_t b)
{
#ifdef __CUDA_ARCH__
    return __umulhi(a, b);
#else
    return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}
HH_HD int32_t mul_hi_s(int32_t a, int32_t b)
{
#ifdef __CUDA_ARCH__
    return __mulhi(a, b);
#else
    return (int32_t)(((int64_t)a * b) >> 32);
#endif
}
HH_HD int clz32(uint32_t a)
{
#ifdef __CUDA_ARCH__
    return __clz((int)a);
#else
    return a ? __builtin_clz(a) : 32;
#endif
}
HH_HD int imax(int a, int b) { return a > b ? a : b; }
HH_HD uint32_t umax(uint32_t a, uint32_t b) { return a > b ? a : b; }
HH_HD int64_t wide_s(int32_t a, int32_t b) { return (int64_t)a * b; }
// max(a + b, c) in both 16-bit halves.
HH_HD uint32_t addmax_u16x2(uint32_t a, uint32_t b, uint32_t c)
{
#ifdef __CUDA_ARCH__
    return __viaddmax_u16x2(a, b, c);
#else
    const uint32_t s = a + b, l = umax(s & 0xffffu, c & 0xffffu), h = umax(s >> 16, c >> 16);
    return h << 16 | l;
#endif
}
HH_HD uint64_t wide_u(uint32_t a, uint32_t b) { return (uint64_t)a * b; }
HH_HD uint32_t hi32(uint64_t x) { return (uint32_t)(x >> 32); }
HH_HD uint32_t lo32(uint64_t x) { return (uint32_t)x; }

// c + a b with a 64-bit c (one multiply-add instruction).
HH_HD int64_t mad_s(int32_t a, int32_t b, int64_t c)
{
#ifdef __CUDA_ARCH__
    int64_t r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
#else
    return c + (int64_t)a * b;
#endif
}
HH_HD uint64_t mad_u(uint32_t a, uint32_t b, uint64_t c)
{
#ifdef __CUDA_ARCH__
    uint64_t r;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
#else
    return c + (uint64_t)a * b;
#endif
}
// Logical shift to the right; 0 from 64 places on.
HH_HD uint64_t shr64(uint64_t x, int s)
{
#ifdef __CUDA_ARCH__
    uint64_t r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));
    return r;
#else
    return s >= 64 ? 0 : x >> s;
#endif
}
HH_HD int64_t sar64(int64_t x, int s)
{
#ifdef __CUDA_ARCH__
    int64_t r;
    asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));
    return r;
#else
    return x >> (s > 63 ? 63 : s);
#endif
}

// Two signed digits of a 64-bit number: x = h 2^32 + l (signed digits, so that
// every partial product is one signed multiply-add and the middle ones land 32
// bits up, where taking the high word is free).
struct Dig {
    int32_t h, l;
};
HH_HD Dig dig(int64_t x)
{
    Dig d;
    d.l = (int32_t)lo32((uint64_t)x);
    d.h = (int32_t)(hi32((uint64_t)x) + (lo32((uint64_t)x) >> 31));
    return d;
}

// Top 64 bits of a 64 x 64-bit product of values below 2^63 (within 2 units).
HH_HD uint64_t mul_top(uint64_t a, uint64_t b)
{
    const uint64_t mid = mad_u(lo32(a), hi32(b), wide_u(hi32(a), lo32(b)));
    return wide_u(hi32(a), hi32(b)) + hi32(mid);
}
// The same of signed numbers in digits, rounded.
HH_HD int64_t mul_dig(const Dig &a, const Dig &b)
{
    const int64_t mid = mad_s(a.l, b.h, mad_s(a.h, b.l, 0x80000000ll));
    return wide_s(a.h, b.h) + (int32_t)hi32((uint64_t)mid);
}

// Three components with one exponent.
struct Vec64 {
    Dig k[3];
    int32_t e;
    uint32_t x[3];  // each component's own (biased) exponent
};

constexpr int kMaxExp = 1223;  // 2^200: largest separation and velocity taken here
constexpr int kMinExp = 128;   // smallest block exponent: anything below counts as zero against it

// kDown = 2: component 2^(e - 1084), largest in [2^61, 2^62); each more place halves that.
// The last bit is always set: what the shift cut off is then wrong by at most one
// unit either way, without a bias, and the ones' complement with that bit set is
// exactly -x (with no carry to pay for), so that f(-d, -w) = -f(d, w).  (Ones'
// complement alone, -x - 1, leant every negative component and broke that in half
// of all pairs; a full negation costs 4% of an evaluation of N = 65536, the bit and
// the test for a vector of zeros 1.5%: 3.23 -> 3.28 ms.)
template <int kDown>
HH_HD void unpack_vec(const double *d, Vec64 &v)
{
    uint32_t a[3];
    for (int k = 0; k < 3; k++) a[k] = f64_hi(d[k]) & 0x7fffffffu;
    v.e = imax((int)(umax(umax(a[0], a[1]), a[2]) >> 20), kMinExp);
    const int base = v.e + kDown;
    for (int k = 0; k < 3; k++) {
        v.x[k] = a[k] >> 20;
        const uint32_t hi = f64_hi(d[k]), lo = f64_lo(d[k]);
        // 1.mantissa left-aligned in 64 bits, then down to its place
        const uint64_t m = ((((uint64_t)hi << 32) | lo) << 11) | 0x8000000000000000ull;
        const uint64_t x = shr64(m, base - (int)v.x[k]);
        const uint32_t neg = (uint32_t)((int32_t)hi >> 31);
        const uint32_t xl = (lo32(x) ^ neg) | 1u;
        v.k[k].l = (int32_t)xl;
        v.k[k].h = (int32_t)((hi32(x) ^ neg) + (xl >> 31));
    }
}

// A positive constant as q 2^x with even x and q in [2^58, 2^60) (0: q = 0).
struct Soft64 {
    uint64_t q;
    int32_t x;
    int32_t dmin;  // smallest block exponent of a separation
    int32_t ok;    // zero or a normal number of moderate size
};
HH_HD Soft64 soft_of(double eps2)
{
    Soft64 s;
    const uint32_t hi = f64_hi(eps2);
    const int e = (int)(hi >> 20);
    if (hi == 0 && f64_lo(eps2) == 0) {
        s.q = 0;
        s.x = -(1 << 20);
        s.dmin = 823;
        s.ok = 1;
        return s;
    }
    s.ok = e >= 623 && e <= 1423;
    s.dmin = 0;
    const uint64_t m = ((((uint64_t)hi << 32) | f64_lo(eps2)) & 0xfffffffffffffull) | 0x10000000000000ull;
    // eps2 = m 2^(e - 1075)
    const int odd = (e - 1075 - 6) & 1;
    s.q = m << (6 + odd);
    s.x = e - 1075 - 6 - odd;
    return s;
}

// Mass of a j entry: mantissa left-aligned below 2^63.  Zero for a mass that
// is not a positive number of moderate size (the pair is then left to FP64).
HH_HD uint64_t mass_bits(double m)
{
    const uint32_t hi = f64_hi(m), e = hi >> 20;
    if (e < 823u || e > 1223u) return 0ull;  // (a set sign bit makes e >= 2048)
    return (((((uint64_t)hi << 32) | f64_lo(m)) & 0xfffffffffffffull) | 0x10000000000000ull) << 10;
}

// Sums of N components with a common exponent: value = (o 2^32 + u) 2^(e - 32).
template <int N>
struct Sum64 {
    uint64_t u[N];
    int64_t o[N];
    int32_t e;
    HH_HD void zero()
    {
        for (int k = 0; k < N; k++) {
            u[k] = 0;
            o[k] = 0;
        }
        e = -(1 << 20);
    }
};

// Where a sum puts its first term (and one too large for it): 24 places below the
// top of the window leave room for terms 2^(24 - smin) larger, so that a thread's
// terms rarely move the scale (a move costs as much as a pair, and one lane's
// move holds up its warp; with 4 places of room instead of about 18 an
// evaluation of N = 65536 took 3.53 ms against 3.41 ms), and 8 bits below the first
// term's last one for smaller ones.  (smin is 5 for 256 entries of a tile of 14, 7
// for 1024: 2^19 and 2^17; the least room is 2^14, 2048 entries of a full tile.)
constexpr int kPlace = 24;

// sum += t 2^(e - s), smin <= s <= 32 (smin: the bits of the number of terms, at least 2)
template <int N>
HH_HD void sum_put(Sum64<N> &S, const int64_t *t, int s)
{
    const uint32_t m = 1u << (32 - s);
    for (int k = 0; k < N; k++) {
        S.u[k] = mad_u(lo32((uint64_t)t[k]), m, S.u[k]);
        S.o[k] = mad_s((int32_t)hi32((uint64_t)t[k]), (int32_t)m, S.o[k]);
    }
}

// The same for any s: makes room for a term larger than any before, drops the
// lowest bits of a much smaller one.
template <int N>
HH_HD void sum_any(Sum64<N> &S, int64_t *t, int s, int smin)
{
    if (s < smin) {
        const int ns = imax(smin, kPlace), d = ns - s;
        if (d < 128) {
            for (int k = 0; k < N; k++) {
                __int128 x = ((__int128)S.o[k] << 32) + (__int128)S.u[k];
                x >>= d;
                S.u[k] = (uint64_t)(uint32_t)x;
                S.o[k] = (int64_t)(x >> 32);
            }
        } else {
            for (int k = 0; k < N; k++) {
                S.u[k] = 0;
                S.o[k] = 0;
            }
        }
        S.e += d;
        s = ns;
    } else if (s > 32) {
        for (int k = 0; k < N; k++) t[k] = sar64(t[k], s - 32);
        s = 32;
    }
    sum_put<N>(S, t, s);
}

// The sum as a double (to nearest on its top 64 bits).
HH_HD double sum_get(uint64_t u, int64_t o, int e)
{
    // 96 bits: c w0, then the magnitude
    uint64_t c = (uint64_t)o + hi32(u);
    uint32_t w0 = lo32(u);
    const bool neg = (int64_t)c < 0;
    if (neg) {
        c = ~c + (w0 == 0u ? 1u : 0u);
        w0 = 0u - w0;
    }
    e -= 32;
    for (int q = 0; q < 2; q++)
        if (hi32(c) == 0u) {  // 32 places up
            c = (c << 32) | w0;
            w0 = 0u;
            e -= 32;
        }
    if (hi32(c) == 0u) return 0.0;
    const int z = clz32(hi32(c));
    uint64_t m = (c << z) | (z ? w0 >> (32 - z) : 0u);
    e += 96 - z;  // value = m 2^(e - 64) with the top bit of m set
    const bool small = e < -1021;  // below the normal range: 2^128 times the value, scaled down by one product
    if (small) e += 128;
    if (e < -1021) return 0.0;
    if (e > 1024) return f64_of(neg ? 0xfff00000u : 0x7ff00000u, 0u);  // beyond it
    // round to 53 bits, ties to even (bits below the 64 kept ones are dropped)
    const uint64_t lsb = (m >> 11) & 1ull;
    m = (m >> 11) + ((((m & 0x7ffull) + lsb) > 0x400ull) ? 1ull : 0ull);
    // m in [2^52, 2^53]; the exponent field carries a round-up to 2^53
    const uint64_t b = ((uint64_t)(e - 1 + 1022) << 52) + m;
    const double x = f64_of(hi32(b) | (neg ? 0x80000000u : 0u), lo32(b));
    return small ? x * 0x1p-128 : x;
}

// Component k's largest term of the force (low half) and of the velocity's part of
// the jerk (high half), as the exponent of u = m / r^3 plus the component's own.
struct Span64 {
    uint32_t k[3];
};

// The integers hold a vector to a unit of its largest component, so a component
// that is small in every term (of a disc, a ring, a nearly planar or collinear
// set) loses what FP64 would keep of it.  True if the largest term of a component is more
// than kThinForce or kThinJerk places below the vector's: the caller then sums in
// FP64.  At that line both are about as good: sheets of 30, 100 and 1000 terms of
// thickness 2^-9 have rms errors of 1.7e-16, 2.2e-16 and 5.0e-16 of the component's own sizes
// in the force and 2.9e-16, 3.5e-16 and 8.2e-16 in the jerk, all in FP64 1.9e-16, 2.3e-16,
// 6.4e-16 and 3.0e-16, 3.6e-16, 8.7e-16; thicker ones are better in integers, thinner ones came
// out worse by 2^-9 over the thickness.  Places less would make more parts of a
// round cluster take FP64 for one close pair's direction (with 5 instead of 8
// places in the jerk one in fourteen: N = 65536 4.22 against 3.42 ms).  A
// component of zeros, which the integers hold exactly, has no exponent to speak
// of: it comes out kThinEnd places or more below the others.
constexpr uint32_t kThinForce = 8, kThinJerk = 8, kThinEnd = 600;
HH_HD bool thin(const Span64 &s)
{
    bool t = false;
    for (int half = 0; half < 2; half++) {
        uint32_t e[3];
        for (int k = 0; k < 3; k++) e[k] = half ? s.k[k] >> 16 : s.k[k] & 0xffffu;
        const uint32_t most = umax(umax(e[0], e[1]), e[2]), lim = half ? kThinJerk : kThinForce;
        for (int k = 0; k < 3; k++) t |= most - e[k] - lim - 1u < kThinEnd - lim - 1u;
    }
    return t;
}

struct AccI64 {
    Sum64<3> a, j;
    Sum64<1> p;
    Span64 span;
    bool bad;
    HH_HD void zero()
    {
        a.zero();
        j.zero();
        p.zero();
        for (int k = 0; k < 3; k++) span.k[k] = 0u;
        bad = false;
    }
};

HH_HD float seed_rsqrt(float f)
{
#ifdef __CUDA_ARCH__
    return rsqrtf(f);
#else
    return 1.0f / __builtin_sqrtf(f);
#endif
}

// y = m / r^3 and the rest follow with scales that keep each product's leading
// bit at 2^55 or above and every middle sum (up to six partial products) below
// 2^63:
//   separation D 2^(D.e - 1084), largest component in [2^61, 2^62); velocity
//   W 2^(W.e - 1081), in [2^58, 2^59); R = r^2 in [2^60, 2^62) 2^(X - n);
//   y = 2^93 / sqrt(R); Z = 2^122 / R; mr = m y 2^-64; u in [2^61, 2^62).
// The jerk uses u w - rho (u d) with rho = 3 (d.w) / r^2: |rho d| <= 3 |w|, so
// rho has a fixed scale against w whatever the sizes.
struct Scal64 {
    uint64_t Z, mr, u;
    int sh, n, h, em, eu;
};
HH_HD Scal64 pair_scalars(const Vec64 &D, double m, uint64_t mb, const Soft64 &eps)
{
    // r^2 = R 2^X
    int64_t hh = wide_s(D.k[0].h, D.k[0].h), hl = wide_s(D.k[0].h, D.k[0].l);
    hh = mad_s(D.k[1].h, D.k[1].h, hh);
    hl = mad_s(D.k[1].h, D.k[1].l, hl);
    hh = mad_s(D.k[2].h, D.k[2].h, hh);
    hl = mad_s(D.k[2].h, D.k[2].l, hl);
    uint64_t R = (uint64_t)(hh + (hl >> 31));
    int X = 2 * D.e - 2104;
    const int sh = imax(eps.x - X, 0);
    R = shr64(R, sh) + shr64(eps.q, imax(X - eps.x, 0));
    X += sh;
    const bool low = hi32(R) < (1u << 28);
    const int n = low ? 2 : 0;
    if (low) R <<= 2;  // [2^60, 2^62)
    const int h = (X - n) >> 1;  // X and n are even
    // y = 2^93 / sqrt(R): FP32 seed, one step of third order on the exact residual
    const float yf = seed_rsqrt((float)hi32(R));
#ifdef __CUDA_ARCH__
    const uint32_t Y = (uint32_t)__float_as_int(__fmaf_rn(yf, 68719476736.0f, 12582912.0f)) - 0x4B400000u;
#else
    const uint32_t Y = (uint32_t)__builtin_rintf(yf * 68719476736.0f);
#endif
    const uint64_t T = wide_u(Y, Y);
    uint64_t P = mad_u(lo32(R), hi32(T), mul_hi(lo32(R), lo32(T)));
    P = mad_u(hi32(R), lo32(T), P);
    P += (uint64_t)(hi32(R) * hi32(T)) << 32;
    const int64_t e = -(int64_t)P;  // 1 - R Y^2 2^-104 in units of 2^-72
    const int32_t e32 = (int32_t)(e >> 21);
    const uint64_t H = mad_u((uint32_t)mul_hi_s(e32, e32), 3u, (uint64_t)e);
    uint64_t y = (uint64_t)mad_s((int32_t)Y, (int32_t)hi32(H), (int64_t)mul_hi(Y, lo32(H)));
    y += (uint64_t)(Y << 9) << 32;
    // 2^122 / R
    const uint64_t Z = wide_u(hi32(y), hi32(y)) + (wide_u(hi32(y), lo32(y)) >> 31);
    const uint64_t mr = mul_top(mb, y);  // m / r
    uint64_t u = mul_top(mr, Z);         // m / r^3
    const int lz = clz32(hi32(u)) - 2;
    u <<= (lz & 31);  // [2^61, 2^62)
    const int em = (int)(f64_hi(m) >> 20);
    return Scal64{Z, mr, u, sh, n, h, em, em - 3 * h - lz};
}

// Adds the pair term of separation d, relative velocity w, mass m (mb its
// mass_bits); a term that has to be left to FP64 sets A.bad.
HH_HD void pair_add(const double *d, const double *w, double m, uint64_t mb, bool self, const Soft64 &eps, int smin,
                    AccI64 &A)
{
    Vec64 D, W;
    unpack_vec<2>(d, D);
    unpack_vec<5>(w, W);
    const Scal64 q = pair_scalars(D, m, mb, eps);
    const uint64_t Z = q.Z, mr = q.mr;
    const int sh = q.sh, n = q.n, h = q.h, em = q.em, eu = q.eu;
    const Dig U = dig((int64_t)q.u);
    // places below the sums' scales
    int sa = A.a.e - (eu + D.e - 2192), sj = A.j.e - (eu + W.e - 2189);
    const int sp = A.p.e - (em - h - 1114);
    int64_t ta[3], tj[3], tp[1] = {(int64_t)mr};
    for (int k = 0; k < 3; k++) ta[k] = mul_dig(U, D.k[k]);
    // jerk: u w - rho (u d) with rho = 3 (d.w) / r^2
    int64_t gh = wide_s(D.k[0].h, W.k[0].h), gl = wide_s(D.k[0].h, W.k[0].l);
    gl = mad_s(D.k[0].l, W.k[0].h, gl);
    gh = mad_s(D.k[1].h, W.k[1].h, gh);
    gl = mad_s(D.k[1].h, W.k[1].l, gl);
    gl = mad_s(D.k[1].l, W.k[1].h, gl);
    gh = mad_s(D.k[2].h, W.k[2].h, gh);
    gl = mad_s(D.k[2].h, W.k[2].l, gl);
    gl = mad_s(D.k[2].l, W.k[2].h, gl);
    const int64_t RW = (int64_t)((uint64_t)gh << (2 + n)) + (gl >> (30 - n));
    // rho in units of the components, times 2^64
    int64_t G = mul_dig(dig(RW), dig((int64_t)Z));
    G = sar64(G, sh);
    G = -(int64_t)((uint64_t)G * 12ull);  // (negated here: a digit of -2^31 has no negative)
    const Dig N = dig(G);
    for (int k = 0; k < 3; k++) {
        const Dig t = dig((int64_t)((uint64_t)ta[k] << 2));
        int64_t mid = mad_s(U.h, W.k[k].l, 0x80000000ll);
        mid = mad_s(U.l, W.k[k].h, mid);
        mid = mad_s(N.h, t.l, mid);
        mid = mad_s(N.l, t.h, mid);
        tj[k] = (int32_t)hi32((uint64_t)mid) + mad_s(N.h, t.h, wide_s(U.h, W.k[k].h));
    }
    // terms more than 32 places down lose their lowest bits
    const int da = imax(sa - 32, 0), dj = imax(sj - 32, 0);
    for (int k = 0; k < 3; k++) ta[k] = sar64(ta[k], da);
    for (int k = 0; k < 3; k++) tj[k] = sar64(tj[k], dj);
    sa -= da;
    sj -= dj;
    const uint32_t out = umax(umax((uint32_t)(sa - smin), (uint32_t)(sj - smin)), (uint32_t)(sp - smin));
    const bool far = (uint32_t)(D.e - eps.dmin) > (uint32_t)(kMaxExp - eps.dmin);
    // (W.e above kMinExp: the last bits of a vector of zeros are no velocity)
    if (out <= (uint32_t)(32 - smin) && !self && !far && (uint32_t)(W.e - kMinExp - 1) < (uint32_t)(kMaxExp - kMinExp) &&
        hi32(mb) != 0u) {
        sum_put<3>(A.a, ta, sa);
        sum_put<3>(A.j, tj, sj);
        sum_put<1>(A.p, tp, sp);
        for (int k = 0; k < 3; k++) A.span.k[k] = addmax_u16x2(D.x[k] | W.x[k] << 16, (uint32_t)eu * 0x10001u, A.span.k[k]);
    } else if (!self) {
        if (far || W.e > kMaxExp || hi32(mb) == 0u) {
            A.bad = true;
        } else {
            sum_any<3>(A.a, ta, sa, smin);
            if (W.e > kMinExp) sum_any<3>(A.j, tj, sj, smin);
            sum_any<1>(A.p, tp, sp, smin);
            for (int k = 0; k < 3; k++)
                A.span.k[k] = addmax_u16x2(D.x[k] | W.x[k] << 16, (uint32_t)eu * 0x10001u, A.span.k[k]);
        }
    }
}

// q 2^x as a double, q in [2^52, 2^64), to nearest.
HH_HD double f64_scaled(uint64_t q, int x)
{
    const int z = clz32(hi32(q));
    uint64_t m = q << z;
    m = (m >> 11) + ((((m & 0x7ffull) + ((m >> 11) & 1ull)) > 0x400ull) ? 1ull : 0ull);
    const uint64_t b = ((uint64_t)(x - z + 1085) << 52) + m;
    return f64_of(hi32(b), lo32(b));
}

// The scalars of a pair alone, as doubles: m / r, m / r^3 and 3 / r^2.
HH_HD void pair_scalars_f64(const double *d, double m, uint64_t mb, const Soft64 &eps, double &mr, double &u, double &z3)
{
    Vec64 D;
    unpack_vec<2>(d, D);
    const Scal64 q = pair_scalars(D, m, mb, eps);
    mr = f64_scaled(q.mr, q.em - q.h - 1114);
    u = f64_scaled(q.u, q.eu - 1172);
    z3 = f64_scaled(3 * q.Z, -2 * q.h - 122);
}

}  // namespace hh
