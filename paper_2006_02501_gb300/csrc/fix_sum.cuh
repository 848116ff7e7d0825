// Sums of fixed-point pair terms (pair_fix.cuh): 64-bit integer accumulators on an
// exponent per body and order that rises with the largest term met; a stage of up to
// 32 terms then goes to FP64 sums.  Shared by pair_fix.cu and batch.cu.
#pragma once

#include "pair_fix.cuh"

namespace mh {

constexpr int kFixExp = 100;           // largest |exponent| of a row
constexpr int kNoMass = -8000;         // exponent of a zero mass: its terms shift out
constexpr int kNoBase = -30000;        // exponent of an accumulator that holds nothing

// Exponent field of a double, |x| < 2^(field - 1022): 0 only for x = 0 (a
// subnormal counts as the smallest normal), 0x7ff for non-finite x.
__device__ __forceinline__ int exponent_field(double x)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int f = (int)(hi >> 20 & 0x7ff);
    return f == 0 && (hi << 1 | lo) != 0 ? 1 : f;
}

// How flat a system is, axis by axis and row by row (x, v, a, a-dot): the mean over its
// bodies of the gap, in bits, of the axis' component below the largest in the difference
// to another body of the system, taken at pseudo-random (fix_partner) so that the order
// of the bodies does not matter.  A gap is at most kGapMax, the gap of a component that
// agrees exactly; axes on which a row is zero throughout don't count.  An isotropic system
// has means of 1.0 to 1.25, a disc of inclinations ~0.025 has 5.8 on its axis and 0.9 in
// its plane.  The means stand for the bulk of the pairs: one inclined body in a thin disc,
// or one thick population among others, leaves the gaps of the rest in them.
//
// The flattest axis, by the smallest of its rows' means, takes the separate exponent of
// Fx3.  Where the other two have a mean above gap_limit between them (a bit more than a
// plane's own, and a margin for the spread of n bodies' mean), what is smaller would be less
// exact than in FP64, which it then takes.
constexpr int kGapMax = 15;

__device__ __forceinline__ float gap_limit(int64_t n) { return 2.0f + 6.0f * rsqrtf((float)n); }

// The other body of the difference: i plus a step that spreads over the system
// (multiplicative hashing by the golden ratio).
__device__ __forceinline__ int64_t fix_partner(int64_t i, int64_t N)
{
    const int64_t j = i + 1 + (int64_t)__umulhi((unsigned)i * 2654435761u, (unsigned)(N - 1));
    return j < N ? j : j - N;
}

// Gaps of a difference's components below the largest, axis `skip` left out.
__device__ __forceinline__ void component_gaps(const double (&d)[3], int skip, int (&g)[3])
{
    int e[3], top = 0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        e[c] = exponent_field(d[c]);
        if (c != skip) top = max(top, e[c]);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) g[c] = top == 0 || c == skip ? 0 : e[c] ? min(top - e[c], kGapMax) : kGapMax;
}

// The flattest axis: gap(k, c) is the mean gap of row k and axis c, negative where the
// axis does not count.
template <int P, typename Gap>
__device__ __forceinline__ int flattest_axis(Gap &&gap)
{
    float best = -1.0f;
    int f = 2;
#pragma unroll
    for (int c = 2; c >= 0; --c) {
        float low = 1e9f;
#pragma unroll
        for (int k = 0; k <= P; ++k) {
            const float q = gap(k, c);
            if (q >= 0.0f) low = fminf(low, q);
        }
        if (low > best) {                      // an axis without motion is flattest of all
            best = low;
            f = c;
        }
    }
    return f;
}

// Vectors hold the flattest axis f last: position of axis c, and axis of position c.
__device__ __forceinline__ int swap_axis(int c, int f) { return c == f ? 2 : c == 2 ? f : c; }

// v 2^e: added to the exponent where the result is normal.
__device__ __forceinline__ double scaled(long long v, int e)
{
    const double d = (double)v;
    const int f = (__double2hiint(d) >> 20 & 0x7ff) + e;
    if (f > 0 && f < 0x7ff && v != 0) return __hiloint2double(__double2hiint(d) + (e << 20), __double2loint(d));
    const int e1 = max(-1000, min(1000, e >> 1)), e2 = max(-1000, min(1000, e - (e >> 1)));
    return d * __hiloint2double((1023 + e1) << 20, 0) * __hiloint2double((1023 + e2) << 20, 0);
}

// The accumulators count units of 2^(base-56).
constexpr int kUnit = 56;

constexpr int kPoison = 1 << 28;       // exponent of an accumulator that is NaN

// acc += a b / 2^64, rounded, plus 2^31: an accumulator of n terms holds its sum
// plus n 2^31 (the offset of FxSum::mid), which raise and the end of the stage take off.
__device__ __forceinline__ void fx_accumulate(long long &acc, Fx a, Fx b)
{
    const long long mid = madw(a.l, b.h, madw(a.h, b.l, kMidOffset));
    acc = fx_get(FxSum{madw(a.h, b.h, acc), mid});
}

// The weight W / 2^n of an accumulator n bits coarser.  Setting the last bit
// makes its truncation error even-handed (an odd integer is the centre of what
// truncates to it or to the even one below): a one-sided error of half a unit
// would add up over the sources on one side of a body.
__device__ __forceinline__ Fx weight(long long W, int n) { return fx(sar(W, n) | 1); }

// Raise the exponent of group g's accumulators to hold terms of exponent `need`: one
// bit more, so that a slowly growing term does not come here each time.
template <int g>
__device__ __forceinline__ void raise(int &base, int need, int terms, long long (&a)[3])
{
    const int to = need + 1, n = to - base;
    const long long off = (long long)terms << 31;
#pragma unroll
    for (int c = fx_first(g); c < fx_first(g + 1); ++c) a[c] = sar(a[c] - off, n) + off;
    base = to;
}

// One order of a pair into a body's accumulators: a[c] += the weight, of mantissa W and
// exponent ew, times A.c[c]; base(g) is the exponent of group g's, `terms` their number so far.
template <typename Base>
__device__ __forceinline__ void fx_take(long long (&a)[3], Base &&base, long long W, int ew, const Fx3 &A, int terms)
{
#pragma unroll
    for (int g = 0; g < 2; ++g) {
        const int need = ew + A.e[g] + 1;
        int b = base(g);
        if (need > b) {
            g ? raise<1>(b, need, terms, a) : raise<0>(b, need, terms, a);
            base(g) = b;
        }
        const Fx w = weight(W, b - need + 1);
#pragma unroll
        for (int c = fx_first(g); c < fx_first(g + 1); ++c) fx_accumulate(a[c], w, A.c[c]);
    }
}

// End of a stage of n terms: group g's accumulators of an order to FP64.  Sums
// that came out far below the unit's range (the largest body was in an earlier
// stage) lower the exponent for the next stage to leave six bits of room, so the
// rounding of small terms does not stay at the largest one's unit.
template <int g, typename Add>
__device__ __forceinline__ void drain(int &base, int n, const long long (&a)[3], Add &&add)
{
    const long long off = (long long)n << 31;
    unsigned top = 0;
    bool any = false;
#pragma unroll
    for (int c = fx_first(g); c < fx_first(g + 1); ++c) {
        const long long v = a[c] - off;
        const double s = scaled(v, base - kUnit);
        add(c, base >= kPoison ? __longlong_as_double(0x7ff8000000000000ll) : s);
        top |= (unsigned)((int)(v >> 32) ^ (int)(v >> 63));
        any |= v != 0;
    }
    const int spare = __clz((int)top) - 16;          // the sums are below 2^(48 - spare)
    if (spare > 0 && any && base < kPoison) base -= spare + 3;
}

}  // namespace mh
