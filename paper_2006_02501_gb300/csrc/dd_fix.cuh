// Pair derivatives with 112-bit mantissas on the integer pipes: the
// double-double form's arithmetic.
//
// A double-double product is 7 FP64 instructions and a sum 20, of 64 cycles each
// per warp and sub-partition on GB300; the pair terms of pair_fix.cuh with
// mantissas twice as long are 13 integer products of 4 cycles where a double-double
// product is needed, and sums of products need one carry pass for all of them.
//
// Numbers.  A mantissa M, normally 2^110 <= |M| < 2^111, is four limbs of 28 bits,
// M = l3 2^84 + l2 2^56 + l1 2^28 + l0 with l0 .. l2 in [0, 2^28) and l3 signed;
// value M 2^(e-111) with an exponent e per vector or scalar.  28 bits leave
// column sums of products far from 64 bits, so products are added column by
// column without carries:
//   M N / 2^112 from columns 2 .. 6 (13 of the 16 limb products); the dropped
//   ones are below one unit of the result, which is up to 2^110.
// A result is good to 2^-108 of its operands' range; double-double operations are
// good to 2^-104 .. 2^-106.
//
// Inputs.  The components of a body's x, v, a, a-dot are 160-bit two's complement
// integers on units of 2^(e-155) with an exponent e per vector and group of
// components (a and a-dot of the bodies of a planetary system span 2^100).  Of two
// bodies the smaller vector is shifted to the larger's unit, and the difference takes
// its exponent from its leading bit: bits are lost only below 2^-153 of a difference
// that did not cancel.  The formulas are those of pair_fix.cuh, and so are the groups:
// the flattest axis of a system, its third component, has exponents of its own.
#pragma once

#include "pair_fix.cuh"

namespace mh {

constexpr int kLb = 28;
constexpr int kLmask = (1 << kLb) - 1;

struct Lx {
    int l[4];
};

MH_HD long long mulw(int a, int b)
{
#ifdef __CUDA_ARCH__
    long long d;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
    return d;
#else
    return (long long)a * b;
#endif
}

// Columns 2 .. 6 of a sum of products.
struct LxSum {
    long long c[5];
};

MH_HD LxSum lx_zero() { return LxSum{{0, 0, 0, 0, 0}}; }

MH_HD void lx_add(LxSum &s, const Lx &a, const Lx &b)
{
    s.c[0] += mulw(a.l[0], b.l[2]) + mulw(a.l[1], b.l[1]) + mulw(a.l[2], b.l[0]);
    s.c[1] += mulw(a.l[0], b.l[3]) + mulw(a.l[1], b.l[2]) + mulw(a.l[2], b.l[1]) + mulw(a.l[3], b.l[0]);
    s.c[2] += mulw(a.l[1], b.l[3]) + mulw(a.l[2], b.l[2]) + mulw(a.l[3], b.l[1]);
    s.c[3] += mulw(a.l[2], b.l[3]) + mulw(a.l[3], b.l[2]);
    s.c[4] += mulw(a.l[3], b.l[3]);
}

MH_HD void lx_add_sqr(LxSum &s, const Lx &a)
{
    const int d1 = a.l[1] + a.l[1], d2 = a.l[2] + a.l[2], d3 = a.l[3] + a.l[3];
    s.c[0] += mulw(a.l[0], d2) + mulw(a.l[1], a.l[1]);
    s.c[1] += mulw(a.l[0], d3) + mulw(d1, a.l[2]);
    s.c[2] += mulw(a.l[1], d3) + mulw(a.l[2], a.l[2]);
    s.c[3] += mulw(d2, a.l[3]);
    s.c[4] += mulw(a.l[3], a.l[3]);
}

// The sum / 2^112, rounded.
MH_HD Lx lx_get(const LxSum &s)
{
    Lx r;
    long long t = s.c[1] + (s.c[0] >> kLb) + (1 << (kLb - 1));
    t = s.c[2] + (t >> kLb);
    r.l[0] = (int)t & kLmask;
    t = s.c[3] + (t >> kLb);
    r.l[1] = (int)t & kLmask;
    t = s.c[4] + (t >> kLb);
    r.l[2] = (int)t & kLmask;
    r.l[3] = (int)(t >> kLb);
    return r;
}

MH_HD Lx lx_mul(const Lx &a, const Lx &b)
{
    LxSum s = lx_zero();
    lx_add(s, a, b);
    return lx_get(s);
}

MH_HD Lx lx_sqr(const Lx &a)
{
    LxSum s = lx_zero();
    lx_add_sqr(s, a);
    return lx_get(s);
}

// Limbs of any sign and up to 31 bits to their ranges.
MH_HD Lx lx_carry(Lx a)
{
    a.l[1] += a.l[0] >> kLb;
    a.l[0] &= kLmask;
    a.l[2] += a.l[1] >> kLb;
    a.l[1] &= kLmask;
    a.l[3] += a.l[2] >> kLb;
    a.l[2] &= kLmask;
    return a;
}

// ka a + kb b for small integers (|ka| + |kb| <= 14).
MH_HD Lx lx_comb(int ka, const Lx &a, int kb, const Lx &b)
{
    // limbs below 2^28 times 14 pass 2^31: the top half of the sum goes through 64 bits
    Lx r;
    long long t = 0;
    for (int k = 0; k < 4; ++k) {
        t = mulw(ka, a.l[k]) + mulw(kb, b.l[k]) + t;
        if (k < 3) {
            r.l[k] = (int)t & kLmask;
            t >>= kLb;
        } else {
            r.l[k] = (int)t;
        }
    }
    return r;
}

MH_HD Lx lx_scale(int ka, const Lx &a)
{
    Lx r;
    long long t = 0;
    for (int k = 0; k < 4; ++k) {
        t = mulw(ka, a.l[k]) + t;
        if (k < 3) {
            r.l[k] = (int)t & kLmask;
            t >>= kLb;
        } else {
            r.l[k] = (int)t;
        }
    }
    return r;
}

// 2a limb by limb, no carries: an operand of lx_mul, whose result keeps a bit more.
MH_HD Lx lx_twice(const Lx &a)
{
    return Lx{{a.l[0] + a.l[0], a.l[1] + a.l[1], a.l[2] + a.l[2], a.l[3] + a.l[3]}};
}

MH_HD Lx lx_plus(const Lx &a, const Lx &b)
{
    return lx_carry(Lx{{a.l[0] + b.l[0], a.l[1] + b.l[1], a.l[2] + b.l[2], a.l[3] + b.l[3]}});
}

// a >> n with sign, any n >= 0.
MH_HD Lx lx_sar(Lx a, int n)
{
    n = imin(n, 5 * kLb - 1);
    while (n >= kLb) {
        a.l[0] = a.l[1];
        a.l[1] = a.l[2];
        a.l[2] = a.l[3] & kLmask;
        a.l[3] >>= kLb;
        n -= kLb;
    }
    Lx r;
    r.l[0] = (int)(((unsigned)a.l[0] >> n) | ((unsigned)a.l[1] << (kLb - n))) & kLmask;
    r.l[1] = (int)(((unsigned)a.l[1] >> n) | ((unsigned)a.l[2] << (kLb - n))) & kLmask;
    r.l[2] = (int)(((unsigned)a.l[2] >> n) | ((unsigned)a.l[3] << (kLb - n))) & kLmask;
    r.l[3] = a.l[3] >> n;
    return r;
}

// a >> n to the nearest (down where n is a multiple of 28; l0 may be 2^28): for
// scalars that small integers multiply next.
MH_HD Lx lx_sar_near(Lx a, int n)
{
    Lx r = lx_sar(a, n);
    if (n > 0 && n < kLb) r.l[0] += a.l[0] >> (n - 1) & 1;
    return r;
}

// a << n, 0 <= n < 28 (the top limb must hold it).
MH_HD Lx lx_shl(const Lx &a, int n)
{
    Lx r;
    r.l[0] = (int)((unsigned)a.l[0] << n) & kLmask;
    r.l[1] = (int)((unsigned)a.l[1] << n | (unsigned)a.l[0] >> (kLb - n)) & kLmask;
    r.l[2] = (int)((unsigned)a.l[2] << n | (unsigned)a.l[1] >> (kLb - n)) & kLmask;
    r.l[3] = (int)((unsigned)a.l[3] << n | (unsigned)a.l[2] >> (kLb - n));
    return r;
}

// Redundant-sign measure of a top limb: leading bit one above |l|'s.
MH_HD unsigned lx_top(int l) { return (unsigned)l ^ ((unsigned)l + (unsigned)l); }

// To 2^110 <= |M| < 2^111 (zero stays); returns the left shift (negative: right).
MH_HD int lx_norm(Lx &a)
{
    int n = 0;
    for (int k = 0; k < 3 && lx_top(a.l[3]) < 2; ++k) {    // pure sign: a whole limb
        a.l[3] = (int)((unsigned)a.l[3] << kLb) | a.l[2];
        a.l[2] = a.l[1];
        a.l[1] = a.l[0];
        a.l[0] = 0;
        n += kLb;
    }
    const int b = imin(clz32(lx_top(a.l[3])), 31) - 4;     // |l3| to [2^26, 2^27)
    if (b >= 0) {
        a = lx_shl(a, b);
    } else {
        a = lx_sar(a, -b);
    }
    return n + b;
}

struct Lx3 {
    Lx c[3];
    int e[2];          // of the first two components together and of the third
};

MH_HD unsigned shr32(unsigned lo, unsigned hi, int n)     // low word of (hi:lo) >> n, 0 <= n < 32
{
#ifdef __CUDA_ARCH__
    return __funnelshift_r(lo, hi, n);
#else
    return n ? lo >> n | hi << (32 - n) : lo;
#endif
}

// Five-word differences, |a - b| < 2^157, unit 2^(E-155).
MH_HD void sub160(const unsigned (&a)[5], const unsigned (&b)[5], unsigned (&d)[5])
{
#ifdef __CUDA_ARCH__
    asm("sub.cc.u32 %0, %5, %10;\n\tsubc.cc.u32 %1, %6, %11;\n\tsubc.cc.u32 %2, %7, %12;\n\t"
        "subc.cc.u32 %3, %8, %13;\n\tsubc.u32 %4, %9, %14;"
        : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3]), "=r"(d[4])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]));
#else
    unsigned long long br = 0;
    for (int k = 0; k < 5; ++k) {
        const unsigned long long q = (unsigned long long)a[k] - b[k] - br;
        d[k] = (unsigned)q;
        br = q >> 63;
    }
#endif
}

// Words of group g of a vector, w >> n with sign, n >= 0.
template <int g>
MH_HD void lx_shift_words(unsigned (&w)[3][5], int n)
{
    n = imin(n, 159);
    while (n >= 32) {
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int c = fx_first(g); c < fx_first(g + 1); ++c) {
            w[c][0] = w[c][1];
            w[c][1] = w[c][2];
            w[c][2] = w[c][3];
            w[c][3] = w[c][4];
            w[c][4] = (unsigned)((int)w[c][4] >> 31);
        }
        n -= 32;
    }
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int c = fx_first(g); c < fx_first(g + 1); ++c) {
        for (int k = 0; k < 4; ++k) w[c][k] = shr32(w[c][k], w[c][k + 1], n);
        w[c][4] = (unsigned)((int)w[c][4] >> n);
    }
}

// Group g of b - a: words of unit 2^(eb-155) and 2^(ea-155).
template <int g>
MH_HD void lx_diff_group(unsigned (&b)[3][5], int eb, unsigned (&a)[3][5], int ea, Lx3 &r)
{
    unsigned d[3][5];
    if (ea < eb) lx_shift_words<g>(a, eb - ea);
    if (eb < ea) lx_shift_words<g>(b, ea - eb);
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int c = fx_first(g); c < fx_first(g + 1); ++c) sub160(b[c], a[c], d[c]);
    auto fold = [&]() { return g ? fold1(d[2][4]) : fold1(d[0][4]) | fold1(d[1][4]); };
    unsigned t = fold();
    int e = imax(ea, eb) + 2;
    for (int k = 0; k < 5 && t < 2; ++k) {
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int c = fx_first(g); c < fx_first(g + 1); ++c) {
            d[c][4] = shl32(d[c][3], d[c][4], 29);
            d[c][3] = shl32(d[c][2], d[c][3], 29);
            d[c][2] = shl32(d[c][1], d[c][2], 29);
            d[c][1] = shl32(d[c][0], d[c][1], 29);
            d[c][0] <<= 29;
        }
        e -= 29;
        t = fold();
    }
    const int n = imin(clz32(t), 31) - 2;              // top word's magnitude to [2^28, 2^29)
    r.e[g] = e - n;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int c = fx_first(g); c < fx_first(g + 1); ++c) {
        const unsigned w4 = shl32(d[c][3], d[c][4], n), w3 = shl32(d[c][2], d[c][3], n);
        const unsigned w2 = shl32(d[c][1], d[c][2], n), w1 = shl32(d[c][0], d[c][1], n);
        // mantissa = bits 46 .. 157
        r.c[c].l[0] = (int)((w1 >> 14 | w2 << 18) & (unsigned)kLmask);
        r.c[c].l[1] = (int)((w2 >> 10 | w3 << 22) & (unsigned)kLmask);
        r.c[c].l[2] = (int)((w3 >> 6 | w4 << 26) & (unsigned)kLmask);
        r.c[c].l[3] = (int)w4 >> 2;
    }
}

MH_HD Lx3 lx_diff(const unsigned (&bw)[3][5], const int (&eb)[2], const unsigned (&aw)[3][5], const int (&ea)[2])
{
    unsigned a[3][5], b[3][5];
    for (int c = 0; c < 3; ++c)
        for (int k = 0; k < 5; ++k) {
            a[c][k] = aw[c][k];
            b[c][k] = bw[c][k];
        }
    Lx3 r;
    lx_diff_group<0>(b, eb[0], a, ea[0], r);
    lx_diff_group<1>(b, eb[1], a, ea[1], r);
    return r;
}

// a.b as v[0] 2^(e[0]-110) + v[1] 2^(e[1]-110), |v[0]| <= 2^111, |v[1]| <= 2^110.
struct LxDot {
    Lx v[2];
    int e[2];
};

MH_HD LxDot lx_dot(const Lx3 &a, const Lx3 &b)
{
    LxSum s = lx_zero(), z = lx_zero();
    lx_add(s, a.c[0], b.c[0]);
    lx_add(s, a.c[1], b.c[1]);
    lx_add(z, a.c[2], b.c[2]);
    return LxDot{{lx_get(s), lx_get(z)}, {a.e[0] + b.e[0], a.e[1] + b.e[1]}};
}

MH_HD LxDot lx_dot_self(const Lx3 &a)
{
    LxSum s = lx_zero(), z = lx_zero();
    lx_add_sqr(s, a.c[0]);
    lx_add_sqr(s, a.c[1]);
    lx_add_sqr(z, a.c[2]);
    return LxDot{{lx_get(s), lx_get(z)}, {2 * a.e[0], 2 * a.e[1]}};
}

MH_HD int lx_upper(const LxDot &d) { return imax(d.e[0], d.e[1]); }

// Its value in units of 2^(e-110), e >= lx_upper.
MH_HD Lx lx_at(const LxDot &d, int e) { return lx_plus(lx_sar(d.v[0], e - d.e[0]), lx_sar(d.v[1], e - d.e[1])); }

// Group g of the components v 2^(e-110), normalised.
template <int g>
MH_HD void lx_norm_group(const Lx (&v)[3], int e, Lx3 &r)
{
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int c = fx_first(g); c < fx_first(g + 1); ++c) r.c[c] = v[c];
    e += 1;
    auto fold = [&]() { return g ? lx_top(r.c[2].l[3]) : lx_top(r.c[0].l[3]) | lx_top(r.c[1].l[3]); };
    unsigned t = fold();
    for (int k = 0; k < 3 && t < 2; ++k) {
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int c = fx_first(g); c < fx_first(g + 1); ++c) {
            Lx &a = r.c[c];
            a.l[3] = (int)((unsigned)a.l[3] << kLb) | a.l[2];
            a.l[2] = a.l[1];
            a.l[1] = a.l[0];
            a.l[0] = 0;
        }
        e -= kLb;
        t = fold();
    }
    const int b = imin(clz32(t), 31) - 4;
    r.e[g] = e - b;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int c = fx_first(g); c < fx_first(g + 1); ++c) r.c[c] = b >= 0 ? lx_shl(r.c[c], b) : lx_sar(r.c[c], -b);
}

MH_HD Lx3 lx_norm3(const Lx (&v)[3], const int (&e)[2])
{
    Lx3 r;
    lx_norm_group<0>(v, e[0], r);
    lx_norm_group<1>(v, e[1], r);
    return r;
}

// A positive scalar M 2^(e-111), normalised.
struct LxNum {
    Lx m;
    int e;
};

constexpr int kLxZero = -20000;        // exponent of the representation of zero
constexpr int kLxBad = 1 << 24;        // exponent of S for s = 0

// s = r.r + eps^2; s^-1 and s^(-3/2).
// rsqrt(f): 1/sqrt(f) in FP64, f in [0.5, 2).  One third-order step from it:
// y = y0 (1 + d/2 + 3 d^2/8), d = 1 - f y0^2 ~ 2^-52, f y0^2 to 2^-111.
template <typename Rsqrt>
MH_HD void lx_inverse(const LxDot &rr, const LxNum &eps2, Rsqrt &&rsqrt, LxNum &sinv, LxNum &S)
{
    int es = lx_upper(rr);
    Lx s = lx_at(rr, es);
    es += 1;
    es -= lx_norm(s);                                  // s 2^(es-111)
    if ((s.l[1] | s.l[2] | s.l[3]) == 0) es = kLxZero;  // (l0 may hold the rounding of a zero sum)
    if (eps2.e > kLxZero) {
        const int E = imax(es, eps2.e) + 1;
        s = lx_plus(lx_sar(s, E - es), lx_sar(eps2.m, E - eps2.e));
        es = E - lx_norm(s);
    }
    if (es <= kLxZero / 2) {                           // bodies at one point without softening
        sinv = S = LxNum{Lx{{0, 0, 0, 1 << 26}}, 0};
        S.e = kLxBad;
        return;
    }
    const int odd = es & 1, h = (es - odd) / 2;        // s = f 2^(2h), f = M 2^(odd-111) in [0.5, 2)
    // top 56 bits of M to a double
    const double f = ((double)s.l[3] * 268435456.0 + (double)s.l[2]) * (odd ? 2.0 : 1.0) * (1.0 / 36028797018963968.0);
    const double y0 = rsqrt(f);
    const long long Y0 = (long long)(y0 * 72057594037927936.0);   // 2^56 y0, exact (53 bits)
    const int a0 = (int)Y0 & kLmask, a1 = (int)(Y0 >> kLb);
    Lx Yq;                                             // 2^112 y0^2
    {
        long long t = mulw(a0, a0);
        Yq.l[0] = (int)t & kLmask;
        t = (t >> kLb) + mulw(a0 + a0, a1);
        Yq.l[1] = (int)t & kLmask;
        t = (t >> kLb) + mulw(a1, a1);
        Yq.l[2] = (int)t & kLmask;
        Yq.l[3] = (int)(t >> kLb);
    }
    Lx p = lx_mul(lx_shl(s, odd), Yq);                 // 2^111 f y0^2
    // d 2^111 = 2^111 - p, below 2^61: 64 bits of it are enough
    const long long D = -(long long)(((unsigned long long)p.l[2] << 56) + ((unsigned long long)p.l[1] << kLb) +
                                     (unsigned long long)p.l[0]);
    const long long dh = D >> 31;
    const long long del = D + ((3 * (dh * dh)) >> 51);  // (d/2 + 3 d^2/8) 2^112
#ifdef __CUDA_ARCH__
    const long long C = __mul64hi(Y0 << 6, del << 2);
#else
    const long long C = (long long)(((__int128)(Y0 << 6) * (del << 2)) >> 64);
#endif
    Lx y{{(int)C & kLmask, (int)(C >> kLb) & kLmask, a0 + (int)(C >> (2 * kLb)), a1}};   // y 2^(112+h)
    y = lx_carry(y);
    const int ey = -h - 1 - lx_norm(y);                // y 2^(ey-111)
    Lx si = lx_sqr(y);
    sinv.e = 2 * ey + 1 - lx_norm(si);
    sinv.m = si;
    Lx s3 = lx_mul(si, y);
    S.e = sinv.e + ey + 1 - lx_norm(s3);
    S.m = s3;
}

template <int P>
struct LxBody {
    unsigned w[P + 1][3][5];
    int e[P + 1][2];
};

// One pair: r^(k) = b^(k) - a^(k), as pair_fix.  weight(S) once, then sink(k, A) for
// k = 0 .. P: A^(k)/(G m S) = A.c[c] 2^(A.e-111).
template <int P, typename Rsqrt, typename Weight, typename Sink>
MH_HD void pair_wide(const LxBody<P> &a, const LxBody<P> &b, const LxNum &eps2, Rsqrt &&rsqrt,
                     Weight &&weight, Sink &&sink)
{
    const Lx3 r = lx_diff(b.w[0], b.e[0], a.w[0], a.e[0]);
    LxNum sinv, S;
    lx_inverse(lx_dot_self(r), eps2, rsqrt, sinv, S);
    const int q = sinv.e;
    weight(S);
    sink(0, r);

    const Lx3 v = lx_diff(b.w[1], b.e[1], a.w[1], a.e[1]);
    // products of scalars carry a factor of 2: their rounding reaches a^(3) times 7 and 5
    const Lx sv = lx_twice(sinv.m);
    Lx an;
    int ea_;
    {
        const LxDot rv = lx_dot(r, v);
        const int erv = lx_upper(rv);
        an = lx_mul(lx_at(rv, erv), sv);                       // alpha 2^(110-erv-q)
        ea_ = erv + q + 1 - lx_norm(an);                       // alpha = an 2^(ea_-111)
    }
    const Lx m3a = lx_scale(-3, an);
    {
        Lx A[3];
        int e[2];
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int g = 0; g < 2; ++g) {
            e[g] = imax(v.e[g], ea_ + 2 + r.e[g]);
            const Lx k1 = lx_sar(m3a, e[g] - r.e[g] - ea_);
#ifdef __CUDACC__
#pragma unroll
#endif
            for (int c = fx_first(g); c < fx_first(g + 1); ++c)
                A[c] = lx_plus(lx_mul(k1, r.c[c]), lx_sar(v.c[c], 1 + e[g] - v.e[g]));
        }
        sink(1, lx_norm3(A, e));
    }
    if constexpr (P >= 2) {
        const Lx3 w = lx_diff(b.w[2], b.e[2], a.w[2], a.e[2]);
        int eq;
        Lx vv;
        {
            const LxDot v2 = lx_dot_self(v), rw = lx_dot(r, w);
            eq = imax(lx_upper(v2), lx_upper(rw));
            vv = lx_plus(lx_at(v2, eq), lx_at(rw, eq));
        }
        const Lx a2 = lx_twice(an);
        const Lx u0 = lx_mul(vv, sv);                          // u 2^(110-eq-q), below 3 2^111
        const Lx p0 = lx_mul(an, a2);                          // alpha^2 2^(111-2 ea_), below 2^111
        const int pu = eq + q - 110, pa = 2 * ea_ - 111;
        const int eu = imax(pu, pa);
        const Lx u = lx_sar_near(u0, eu - pu), p = lx_sar_near(p0, eu - pa);
        Lx m2 = lx_comb(5, p, -1, u);
        const int ec2 = eu + 111 - lx_norm(m2);
        {
            Lx A[3];
            int e[2];
#ifdef __CUDACC__
#pragma unroll
#endif
            for (int g = 0; g < 2; ++g) {
                e[g] = imax(w.e[g], imax(ea_ + 3 + v.e[g], ec2 + 2 + r.e[g]));
                const Lx k1 = lx_sar(m3a, e[g] - v.e[g] - ea_ - 1);
                const Lx k2 = lx_sar(lx_scale(3, m2), e[g] - r.e[g] - ec2);
#ifdef __CUDACC__
#pragma unroll
#endif
                for (int c = fx_first(g); c < fx_first(g + 1); ++c) {
                    LxSum t = lx_zero();
                    lx_add(t, k1, v.c[c]);
                    lx_add(t, k2, r.c[c]);
                    A[c] = lx_plus(lx_get(t), lx_sar(w.c[c], 1 + e[g] - w.e[g]));
                }
            }
            sink(2, lx_norm3(A, e));
        }
        if constexpr (P >= 3) {
            const Lx3 y = lx_diff(b.w[3], b.e[3], a.w[3], a.e[3]);
            int ez;
            Lx zz;
            {
                const LxDot vw = lx_dot(v, w), ry = lx_dot(r, y);
                ez = imax(lx_upper(vw), lx_upper(ry));
                zz = lx_comb(3, lx_at(vw, ez), 1, lx_at(ry, ez));
            }
            const Lx z0 = lx_mul(zz, sv);                      // z 2^(110-ez-q), below 3 2^112
            Lx h = lx_comb(3, u, -7, p);
            const int eh = eu + 111 - lx_norm(h);
            const Lx t0 = lx_mul(h, a2);                       // alpha h 2^(111-eh-ea_)
            const int pt = eh + ea_ - 111, pz = ez + q - 110;
            const int et = imax(pt, pz);
            Lx m3 = lx_comb(5, lx_sar_near(t0, et - pt), -1, lx_sar_near(z0, et - pz));
            const int ec3 = et + 111 - lx_norm(m3);
            Lx A[3];
            int e[2];
#ifdef __CUDACC__
#pragma unroll
#endif
            for (int g = 0; g < 2; ++g) {
                e[g] = imax(imax(y.e[g], ea_ + 4 + w.e[g]), imax(ec2 + 4 + v.e[g], ec3 + 2 + r.e[g]));
                const Lx k1 = lx_sar(lx_scale(-9, an), e[g] - w.e[g] - ea_);
                const Lx k2 = lx_sar(lx_scale(9, m2), e[g] - v.e[g] - ec2);
                const Lx k3 = lx_sar(lx_scale(3, m3), e[g] - r.e[g] - ec3);
#ifdef __CUDACC__
#pragma unroll
#endif
                for (int c = fx_first(g); c < fx_first(g + 1); ++c) {
                    LxSum t = lx_zero();
                    lx_add(t, k1, w.c[c]);
                    lx_add(t, k2, v.c[c]);
                    lx_add(t, k3, r.c[c]);
                    A[c] = lx_plus(lx_get(t), lx_sar(y.c[c], 1 + e[g] - y.e[g]));
                }
            }
            sink(3, lx_norm3(A, e));
        }
    }
}

}  // namespace mh
