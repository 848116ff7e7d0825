// Pair derivatives in 64-bit fixed point: the FP64 form's arithmetic on the
// integer pipes.
//
// GB300 issues one FP64 instruction of a warp per sub-partition every 64
// cycles, a 32 x 32 -> 64 bit integer multiply-add every ~4.5 and a 64-bit
// addition every ~2.5 (measured, 4 warps per sub-partition).  A product of two
// 62-bit fixed-point numbers is three such multiply-adds, so one FP64 multiply-add
// costs as much as four or five products of higher accuracy.  This header
// evaluates a pair that way: only 1/sqrt(s) and its powers (8 instructions)
// stay on the FP64 pipe.
//
// Numbers.  A vector or scalar is an integer mantissa M, |M| <= 2^61, with an
// exponent e of its own per pair: value = M 2^(e-61).  M is held as two 32-bit
// limbs h 2^32 + l with l signed ("balanced"), so that all partial products are
// signed 32 x 32 -> 64 bit ones:
//   M N / 2^64 = h h' + (h l' + l h') / 2^32 + l l' / 2^64;
// the last term (below 1/4 unit of a result of up to 2^58) is dropped.
//
// Inputs.  Every component of x, v, a, a-dot of a body is a 96-bit two's
// complement integer on a grid per row (x, v, a or a-dot) for the whole
// system: unit 2^(E-91), E the exponent of the largest component.  An FP64 value
// down to 2^-38 of the largest is on the grid exactly; systems with a wider
// range of magnitudes are evaluated in FP64 (the caller's rule).  Differences
// are then exact.
//
// The components of a vector share an exponent, from the leading bit of the largest,
// so a small one keeps fewer bits than it would in FP64.  The flattest axis of a
// system (a disc's), which the caller makes the third component, therefore has grids,
// exponents and sums of its own (Fx3::e[1]): only dot products meet both.  What the
// other two lack between them is the caller's rule again.
//
// Pair derivatives (Dittmann 2020, Section 3, intro), with S = s^(-3/2),
// s = r.r + eps^2, in Leibniz form A^(k) / (G m S) = sum C(k, n) c_n r^(k-n),
// c_n = S^(n) / S:
//   alpha = (r.v)/s,  u = (v.v + r.a)/s,  z = (3 v.a + r.adot)/s,
//   c1 = -3 alpha,  c2 = 3 (5 alpha^2 - u),  c3 = 3 (5 alpha (3 u - 7 alpha^2) - z).
// Every scalar is normalised to its own exponent; in the sums for A^(k) the
// scalars are shifted to the exponent of the largest product, so an A^(k) is
// accurate to about 2^-57 of its largest term (FP64: 2^-53).
#pragma once

#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define MH_HD __host__ __device__ __forceinline__
#else
#include <math.h>
#define MH_HD inline
#endif

namespace mh {

// value h 2^32 + l, l in [-2^31, 2^31)
struct Fx {
    int h, l;
};

MH_HD Fx fx(long long v)
{
    const int l = (int)(unsigned)v;
    return Fx{(int)(v >> 32) + (int)((unsigned)l >> 31), l};
}

// 32 x 32 -> 64 bit product plus c.  By name on the device: written as C the
// compiler widens both factors first and multiplies 64 x 64 bits.
MH_HD long long madw(int a, int b, long long c)
{
#ifdef __CUDA_ARCH__
    long long d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
#else
    return (long long)a * b + c;
#endif
}

// A sum of products in two 64-bit parts: hi 2^64 + mid 2^32.  mid carries an
// offset of 2^63, so that its high word is unsigned and adds to hi without a
// sign extension (hi starts 2^31 lower), and half a unit of hi, which rounds fx_get.
struct FxSum {
    long long hi, mid;
};
constexpr long long kMidOffset = (long long)0x8000000080000000ull;
constexpr long long kHiOffset = -0x80000000ll;

MH_HD FxSum fx_mul(Fx a, Fx b)
{
    return FxSum{madw(a.h, b.h, kHiOffset), madw(a.l, b.h, madw(a.h, b.l, kMidOffset))};
}

MH_HD FxSum fx_sqr(Fx a)
{
    return FxSum{madw(a.h, a.h, kHiOffset), madw(a.h + a.h, a.l, kMidOffset)};
}

MH_HD void fx_add(FxSum &s, Fx a, Fx b)
{
    s.hi = madw(a.h, b.h, s.hi);
    s.mid = madw(a.l, b.h, madw(a.h, b.l, s.mid));
}

MH_HD void fx_add_sqr(FxSum &s, Fx a)
{
    s.hi = madw(a.h, a.h, s.hi);
    s.mid = madw(a.h + a.h, a.l, s.mid);
}

// The sum / 2^64, rounded.
MH_HD long long fx_get(FxSum s) { return s.hi + (long long)(unsigned)((unsigned long long)s.mid >> 32); }

// The same times 2^n.
MH_HD long long fx_get_shl(FxSum s, int n) { return (long long)((unsigned long long)fx_get(s) << n); }

MH_HD int clz32(unsigned x)
{
#ifdef __CUDA_ARCH__
    return __clz((int)x);
#else
    return x ? __builtin_clz(x) : 32;
#endif
}

MH_HD unsigned shl32(unsigned lo, unsigned hi, int n)     // top word of (hi:lo) << n, 0 <= n < 32
{
#ifdef __CUDA_ARCH__
    return __funnelshift_l(lo, hi, n);
#else
    return n ? hi << n | lo >> (32 - n) : hi;
#endif
}

MH_HD int imax(int a, int b) { return a > b ? a : b; }
MH_HD int imin(int a, int b) { return a < b ? a : b; }

// v >> n with sign, any n >= 0.
MH_HD long long sar(long long v, int n)
{
#ifdef __CUDA_ARCH__
    long long r;
    asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));   // clamps n
    return r;
#else
    return v >> imin(n, 63);
#endif
}

// v to 2^60 <= |M| <= 2^61 (fewer bits if |v| < 2^32); returns the left shift.
MH_HD int fx_norm(long long &v)
{
    const int h = (int)(v >> 32);
    const int n = clz32((unsigned)(h ^ (h >> 31))) - 3;
    v = n >= 0 ? (long long)((unsigned long long)v << n) : v >> -n;
    return n;
}

// A vector: mantissas, and exponents of the first two components together and of the
// third, value = M 2^(e-61).
struct Fx3 {
    Fx c[3];
    int e[2];
};
MH_HD constexpr int fx_group(int c) { return c == 2; }
// components of group g: [fx_first(g), fx_first(g + 1))
MH_HD constexpr int fx_first(int g) { return g == 0 ? 0 : g + 1; }

MH_HD void sub96(const unsigned (&a)[3], const unsigned (&b)[3], unsigned (&d)[3])
{
#ifdef __CUDA_ARCH__
    asm("sub.cc.u32 %0, %3, %6;\n\tsubc.cc.u32 %1, %4, %7;\n\tsubc.u32 %2, %5, %8;"
        : "=r"(d[0]), "=r"(d[1]), "=r"(d[2])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(b[0]), "r"(b[1]), "r"(b[2]));
#else
    const unsigned long long q0 = (unsigned long long)a[0] - b[0];
    const unsigned long long q1 = (unsigned long long)a[1] - b[1] - (q0 >> 63);
    d[0] = (unsigned)q0;
    d[1] = (unsigned)q1;
    d[2] = a[2] - b[2] - (unsigned)(q1 >> 63);
#endif
}

// Bits above 1 mark changes between neighbouring bits of a high word: the leading one
// of the two components' (or the one's) is one above the largest's leading bit.
MH_HD unsigned fold1(unsigned h) { return h ^ (h + h); }

// A difference of 96-bit two's complement components (w[c] = low, middle, high word,
// |value| < 2^93), units 2^(E-91) of the first two and 2^(Ez-91) of the third.
MH_HD Fx3 fx_diff(const unsigned (&a)[3][3], const unsigned (&b)[3][3], int E, int Ez)
{
    unsigned d[3][3];
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int c = 0; c < 3; ++c) sub96(a[c], b[c], d[c]);
    Fx3 r;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int g = 0; g < 2; ++g) {
        auto fold = [&] { return g ? fold1(d[2][2]) : fold1(d[0][2]) | fold1(d[1][2]); };
        unsigned t = fold();
        int e = (g ? Ez : E) + 2;
        // a difference far below the largest component: 29 bits at a time (the high
        // words are pure sign, so 29 more bits fit)
        for (int k = 0; k < 3 && t < 2; ++k) {
#ifdef __CUDACC__
#pragma unroll
#endif
            for (int c = fx_first(g); c < fx_first(g + 1); ++c) {
                d[c][2] = shl32(d[c][1], d[c][2], 29);
                d[c][1] = shl32(d[c][0], d[c][1], 29);
                d[c][0] <<= 29;
            }
            e -= 29;
            t = fold();
        }
        const int n = imin(clz32(t), 31) - 2;
        r.e[g] = e - n;
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int c = fx_first(g); c < fx_first(g + 1); ++c) {
            const unsigned h = shl32(d[c][1], d[c][2], n), l = shl32(d[c][0], d[c][1], n);
            r.c[c] = Fx{(int)h + (int)(l >> 31), (int)l};
        }
    }
    return r;
}

// Components v 2^(e-58) to 2^60 <= |M| <= 2^61 of the group's largest (or |v| < 2^32
// shifted by 29).
MH_HD Fx3 fx_norm3(const long long (&v)[3], const int (&e)[2])
{
    Fx3 r;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int g = 0; g < 2; ++g) {
        const unsigned t = g ? fold1((unsigned)(v[2] >> 32))
                             : fold1((unsigned)(v[0] >> 32)) | fold1((unsigned)(v[1] >> 32));
        const int n = imin(clz32(t), 31) - 2;
        r.e[g] = e[g] + 3 - n;
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int c = fx_first(g); c < fx_first(g + 1); ++c) r.c[c] = fx((long long)((unsigned long long)v[c] << n));
    }
    return r;
}

MH_HD long long fx_val(Fx a)
{
    return (long long)((unsigned long long)(unsigned)(a.h + (a.l >> 31)) << 32 | (unsigned)a.l);
}

// a.b as v[0] 2^(e[0]-58) + v[1] 2^(e[1]-58), |v[0]| <= 2^59, |v[1]| <= 2^58.
struct FxDot {
    long long v[2];
    int e[2];
};

MH_HD FxDot fx_dot(const Fx3 &a, const Fx3 &b)
{
    FxSum s = fx_mul(a.c[0], b.c[0]);
    fx_add(s, a.c[1], b.c[1]);
    return FxDot{{fx_get(s), fx_get(fx_mul(a.c[2], b.c[2]))}, {a.e[0] + b.e[0], a.e[1] + b.e[1]}};
}

MH_HD FxDot fx_dot_self(const Fx3 &a)
{
    FxSum s = fx_sqr(a.c[0]);
    fx_add_sqr(s, a.c[1]);
    return FxDot{{fx_get(s), fx_get(fx_sqr(a.c[2]))}, {2 * a.e[0], 2 * a.e[1]}};
}

MH_HD int fx_top(const FxDot &d) { return imax(d.e[0], d.e[1]); }

// Its value in units of 2^(e-58), e >= fx_top.
MH_HD long long fx_at(const FxDot &d, int e) { return sar(d.v[0], e - d.e[0]) + sar(d.v[1], e - d.e[1]); }

// r.r as a double: rounded to nearest.
MH_HD double fx_square_to_double(const FxDot &rr)
{
    const int e = fx_top(rr);
    unsigned long long u = (unsigned long long)fx_at(rr, e) << 4;       // r^2 2^(62-e), below 2^64
    const int c = clz32((unsigned)(u >> 32));                           // 0 .. 3 unless r = 0
    u <<= c;
    unsigned long long b = (u >> 11) + ((unsigned)u >> 10 & 1u);
    b += (unsigned long long)(unsigned)(1023 + e - c) << 52;            // the leading bit adds 1 to the exponent
    if (c > 3) b = 0;
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double d;
    memcpy(&d, &b, 8);
    return d;
#endif
}

// Mantissa M in [2^60, 2^61) and exponent q of a positive normal double, value M 2^(q-60).
MH_HD Fx fx_from_double(double d, int &q)
{
    long long b;
#ifdef __CUDA_ARCH__
    b = __double_as_longlong(d);
#else
    memcpy(&b, &d, 8);
#endif
    const unsigned hi = (unsigned)(b >> 32), lo = (unsigned)b;
    q = (int)(hi >> 20) - 1023;
    const unsigned h = ((hi << 8 | lo >> 24) & 0x0fffffffu) | 0x10000000u, l = lo << 8;
    return Fx{(int)h + (int)(l >> 31), (int)l};
}

// Fixed-point record of one body: P + 1 rows of three 96-bit components.
template <int P>
struct FxBody {
    unsigned w[P + 1][3][3];
};

// The powers s^-1 and s^(-3/2) and the terms of one pair with the differences
// r^(k) = diff(k) = b^(k) - a^(k) (components c[c] 2^(e-61), each group's largest normalised).
// inverse(r, sinv, S): the FP64 powers of s = r.r + eps^2.  Calls weight(S) once, then
// sink(k, A) for k = 0 .. P in order: A^(k)/(G m S) has components A.c[c] 2^(A.e-61),
// each group's largest normalised.
template <int P, typename Diff, typename Inverse, typename Weight, typename Sink>
MH_HD void pair_terms(Diff &&diff, Inverse &&inverse, Weight &&weight, Sink &&sink)
{
    const Fx3 r = diff(0);
    double sinv_d, S_d;
    inverse(r, sinv_d, S_d);
    int q;
    const Fx sinv = fx_from_double(sinv_d, q);                  // s^-1 = sinv 2^(q-60)
    weight(S_d);
    sink(0, r);

    const Fx3 v = diff(1);
    const FxDot rvd = fx_dot(r, v);
    const int erv = fx_top(rvd);
    const Fx rv = fx((long long)((unsigned long long)fx_at(rvd, erv) << 1));   // r.v 2^(59-erv)
    long long an = fx_get_shl(fx_mul(rv, sinv), 3);             // alpha 2^(58-erv-q)
    const int ea_ = erv + q + 3 - fx_norm(an);                  // alpha = an 2^(ea_-61)
    const long long m3a = -(an + 2 * an);
    const Fx al = fx(an);
    {
        long long A[3];
        int e[2];
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int g = 0; g < 2; ++g) {
            e[g] = imax(v.e[g], ea_ + 2 + r.e[g]);
            const Fx k1 = fx(sar(m3a, e[g] - r.e[g] - ea_));
            const int nv = 3 + e[g] - v.e[g];
#ifdef __CUDACC__
#pragma unroll
#endif
            for (int c = fx_first(g); c < fx_first(g + 1); ++c)
                A[c] = fx_get(fx_mul(k1, r.c[c])) + sar(fx_val(v.c[c]), nv);
        }
        sink(1, fx_norm3(A, e));
    }
    if constexpr (P >= 2) {
        const Fx3 w = diff(2);
        // v.v + r.a on the larger exponent of the two, times 1/s
        const FxDot vv = fx_dot_self(v), rw = fx_dot(r, w);
        const int eq = imax(fx_top(vv), fx_top(rw));
        const Fx vq = fx(fx_at(vv, eq) + fx_at(rw, eq));
        const long long u0 = fx_get_shl(fx_mul(vq, sinv), 3);   // u 2^(57-eq-q)
        const long long p0 = fx_get_shl(fx_sqr(al), 2);         // alpha^2 2^(60-2 ea_)
        const int pu = eq + q - 57, pa = 2 * ea_ - 60;
        const int eu = imax(pu + 2, pa + 1);                    // |u|, |p| < 2^59
        const long long u = sar(u0, eu - pu), p = sar(p0, eu - pa);
        long long m2 = p + 4 * p - u;                           // (5 alpha^2 - u) 2^-eu
        const int ec2 = eu + 61 - fx_norm(m2);
        const long long m2x3 = m2 + 2 * m2;
        {
            long long A[3];
            int e[2];
#ifdef __CUDACC__
#pragma unroll
#endif
            for (int g = 0; g < 2; ++g) {
                e[g] = imax(w.e[g], imax(ea_ + 3 + v.e[g], ec2 + 2 + r.e[g]));
                const Fx k1 = fx(sar(m3a, e[g] - v.e[g] - ea_ - 1));
                const Fx k2 = fx(sar(m2x3, e[g] - r.e[g] - ec2));
                const int nw = 3 + e[g] - w.e[g];
#ifdef __CUDACC__
#pragma unroll
#endif
                for (int c = fx_first(g); c < fx_first(g + 1); ++c) {
                    FxSum t = fx_mul(k1, v.c[c]);
                    fx_add(t, k2, r.c[c]);
                    A[c] = fx_get(t) + sar(fx_val(w.c[c]), nw);
                }
            }
            sink(2, fx_norm3(A, e));
        }
        if constexpr (P >= 3) {
            const Fx3 y = diff(3);
            const FxDot vw = fx_dot(v, w), ry = fx_dot(r, y);
            const int ez = imax(fx_top(vw), fx_top(ry));
            const long long va = fx_at(vw, ez);
            const Fx zz = fx(va + 2 * va + fx_at(ry, ez));
            const long long z0 = fx_get_shl(fx_mul(zz, sinv), 2);      // z 2^(56-ez-q)
            long long h = u + 2 * u - (8 * p - p);                     // (3 u - 7 alpha^2) 2^-eu
            const int eh = eu + 61 - fx_norm(h);
            const long long t0 = fx_get(fx_mul(fx(h), al));            // alpha h 2^(58-eh-ea_)
            const int pt = eh + ea_ - 58, pz = ez + q - 56;
            const int et = imax(pt, pz + 1);
            const long long t = sar(t0, et - pt);
            long long m3 = t + 4 * t - sar(z0, et - pz);               // (5 alpha h - z) 2^-et
            const int ec3 = et + 61 - fx_norm(m3);
            long long A[3];
            int e[2];
#ifdef __CUDACC__
#pragma unroll
#endif
            for (int g = 0; g < 2; ++g) {
                e[g] = imax(imax(y.e[g], ea_ + 4 + w.e[g]), imax(ec2 + 4 + v.e[g], ec3 + 2 + r.e[g]));
                const Fx k1 = fx(sar(3 * (m3a >> 2), e[g] - w.e[g] - ea_ - 2));
                const Fx k2 = fx(sar(3 * (m2x3 >> 2), e[g] - v.e[g] - ec2 - 2));
                const Fx k3 = fx(sar(m3 + 2 * m3, e[g] - r.e[g] - ec3));
                const int ny = 3 + e[g] - y.e[g];
#ifdef __CUDACC__
#pragma unroll
#endif
                for (int c = fx_first(g); c < fx_first(g + 1); ++c) {
                    FxSum s = fx_mul(k1, w.c[c]);
                    fx_add(s, k2, v.c[c]);
                    fx_add(s, k3, r.c[c]);
                    A[c] = fx_get(s) + sar(fx_val(y.c[c]), ny);
                }
            }
            sink(3, fx_norm3(A, e));
        }
    }
}

// One pair of two bodies on the rows' grids, E for the first two components and E + dz
// for the third.  weight(MS, qS): S = MS 2^(qS-60); rinv3(s, sinv, S): the FP64 powers of s.
template <int P, typename Rsqrt, typename Weight, typename Sink>
MH_HD void pair_fix(const FxBody<P> &a, const FxBody<P> &b, const int (&E)[4], int dz, double eps2, Rsqrt &&rinv3,
                    Weight &&weight, Sink &&sink)
{
    pair_terms<P>([&](int k) { return fx_diff(b.w[k], a.w[k], E[k], E[k] + dz); },
                  [&](const Fx3 &r, double &sinv, double &S) {
                      rinv3(fx_square_to_double(fx_dot_self(r)) + eps2, sinv, S);
                  },
                  [&](double S) {
                      int qS;
                      const Fx MS = fx_from_double(S, qS);
                      weight(MS, qS);
                  },
                  sink);
}

}  // namespace mh
