// FP64 states as zone-scaled 64-bit integers.
//
// Most FP64 instructions of the predictor and face kernels were linear algebra: node states are fixed linear
// combinations of a zone's modes.  GB300 executes 1.7 FP64 additions per clock and SM, but 58 64-bit integer
// additions (measured, independent chains on every SM), so these combinations run on integers: a zone's modes
// of one variable share the exponent of the largest of them, q = mode * 2^s, and sums and differences of q are
// exact.  Only the products and quotients of the fluxes stay FP64.
//
// Precision.  The largest value of a frame keeps all its 53 bits and LSH more below them; the others are cut at the same
// unit, 2^-(53 + LSH) of the largest.  A sum then carries an error of a few such units before it is rounded once to
// FP64, where an FP64 sum rounds at every operation to 2^-53 of its partial sums.  With the frame's largest value among
// a sum's terms the integers' error is the smaller one.  A sum of terms that are all small beside the largest value of
// the frame keeps that absolute error, where FP64 would keep a relative one.  Frames therefore hold values that enter
// the same sums: the modes of one variable of a zone (every node state has the mean in it), the fluxes of one variable
// in one direction (the pressure sets the size of one direction's momentum flux and is absent from the others'), and
// the differences of one WENO stencil.  What is left: a variable whose mean is far below its variation along one axis
// holds its variation along another to 2^-58 of the larger one (order 4: 2^-56) instead of to its own last place.
//
// Measured (FP64): face states alone took the third-order predictor of 64 x 128 x 128 zones, one thread a zone, from
// 6.28 to 4.71 ms (3224 -> 2116 FP64 instructions a zone); with the sums of flux modes, teams of warps (team.cuh) and
// the reciprocals (common.cuh) it takes 2.6 ms and 1053.  The nodal fourth-order step of 56^3 zones fell from 5.60 to
// 3.0 ms when its tables moved here.  A frame per direction instead of one for all costs 2% of a third-order and 4% of a
// fourth-order step (256^3 nodal 68.2 -> 69.6 ms, 96^3 modal 14.4 -> 14.9 ms).
//
// Range.  HEADROOM = 10 - LSH bits are left above the largest mode for sums; intermediate sums may wrap (the
// arithmetic is modulo 2^64) as long as no wrapped value is shifted or scaled by a fraction.  Modes of magnitude
// below 2^-767 count as zero; a variable with a mode that is not finite, or within 2^16 of the largest FP64
// number, leaves as NaN at every node.
#pragma once
#include "common.cuh"

namespace ader {

struct Fix {
    long long q;
};

ADER_DEV Fix fix_wrap(unsigned long long q) {
    Fix r;
    r.q = (long long)q;
    return r;
}
ADER_DEV Fix operator+(Fix a, Fix b) { return fix_wrap((unsigned long long)a.q + (unsigned long long)b.q); }
ADER_DEV Fix operator-(Fix a, Fix b) { return fix_wrap((unsigned long long)a.q - (unsigned long long)b.q); }
ADER_DEV Fix operator-(Fix a) { return fix_wrap(0ull - (unsigned long long)a.q); }

// the upper 64 bits of the 128-bit product
ADER_DEV long long fix_mulhi(long long a, long long b) {
#ifdef __CUDA_ARCH__
    return __mul64hi(a, b);
#else
    return (long long)(((__int128)a * b) >> 64);
#endif
}

// c a for a literal c (folded at compile time): the nearest integer by a multiplication, a fractional power of
// two by a shift, any other fraction by the upper half of a product with it (c's FP64 value less the integer, at
// most 53 bits)
ADER_DEV Fix fix_times(double c, Fix a) {          // c >= 0
    const long long i = (long long)(c + 0.49999999);
    const double f = c - (double)i;                 // in (-1/2, 1/2]
    const double g = f < 0.0 ? -f : f;
    Fix r = fix_wrap((unsigned long long)a.q * (unsigned long long)i);
    if (g == 0.0) return r;
    Fix p;
    if (g == 0.5) p.q = a.q >> 1;
    else if (g == 0.25) p.q = a.q >> 2;
    else if (g == 0.125) p.q = a.q >> 3;
    else if (g == 0.0625) p.q = a.q >> 4;
    else if (g == 0.03125) p.q = a.q >> 5;
    else if (g == 0.015625) p.q = a.q >> 6;
    else p.q = fix_mulhi(a.q, (long long)(g * 18446744073709551616.0));
    return f < 0.0 ? r - p : r + p;
}
ADER_DEV Fix operator*(double c, Fix a) { return c < 0.0 ? -fix_times(-c, a) : fix_times(c, a); }

template <int NV>
ADER_DEV Vec<NV, Fix> operator*(double s, const Vec<NV, Fix>& a) {
    Vec<NV, Fix> r;
#pragma unroll
    for (int i = 0; i < NV; ++i) r.v[i] = s * a.v[i];
    return r;
}

ADER_DEV long long bits_of(double x) {
#ifdef __CUDA_ARCH__
    return __double_as_longlong(x);
#else
    long long b;
    __builtin_memcpy(&b, &x, 8);
    return b;
#endif
}
ADER_DEV double of_bits(long long b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double(b);
#else
    double x;
    __builtin_memcpy(&x, &b, 8);
    return x;
#endif
}

// What a zone's node states are built in: the scalar S, and the way in and out.  In general S is the bulk
// precision R itself and both ways are the identity; FP64 takes Fix with one exponent per variable.
// Use: include() every mode, close(), then enter() the modes and leave() with the states.
template <int NV, class R>
struct PlainFrame {
    using S = R;
    ADER_DEV void include(const Vec<NV, R>&) {}
    ADER_DEV void close() {}
    ADER_DEV Vec<NV, S> enter(const Vec<NV, R>& m) const { return m; }
    ADER_DEV PlainFrame extended(const Vec<NV, R>*, int) const { return *this; }
    ADER_DEV void join(const PlainFrame&) {}
    ADER_DEV Vec<NV, S> from(const PlainFrame&, const Vec<NV, S>& u) const { return u; }
    ADER_DEV Vec<NV, R> leave(const Vec<NV, S>& u) const { return u; }
};

template <int NV, int LSH>
struct FixFrame {
    using S = Fix;
    unsigned e[NV];       // biased exponent of the largest mode
    unsigned bad[NV];     // bits that make a value NaN, or none

    ADER_DEV FixFrame() {
#pragma unroll
        for (int v = 0; v < NV; ++v) e[v] = 0;
    }
    ADER_DEV void include(const Vec<NV, double>& m) {
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const unsigned h = (unsigned)((unsigned long long)bits_of(m[v]) >> 32) & 0x7ff00000u;
            e[v] = h > e[v] ? h : e[v];
        }
    }
    ADER_DEV void close() {
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            e[v] >>= 20;
            bad[v] = e[v] > 2046u - 16u ? 0x7ff80000u : 0u;
            e[v] = e[v] < 256u ? 256u : e[v];
        }
    }
    ADER_DEV Vec<NV, Fix> enter(const Vec<NV, double>& m) const {
        Vec<NV, Fix> r;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const long long b = bits_of(m[v]);
            const unsigned long long mant = ((unsigned long long)b & 0xfffffffffffffull) | 0x10000000000000ull;
            const unsigned d = e[v] - ((unsigned)((unsigned long long)b >> 52) & 0x7ffu);
            const unsigned long long q = (mant << LSH) >> (d < 63u ? d : 63u);
            const unsigned long long s = (unsigned long long)(b >> 63);
            r[v] = fix_wrap((q ^ s) - s);
        }
        return r;
    }
    // this frame, wide enough for the n modes m too; from() brings a state of the narrower frame into it
    ADER_DEV FixFrame extended(const Vec<NV, double>* m, int n) const {
        FixFrame r;
#pragma unroll
        for (int k = 0; k < n; ++k) r.include(m[k]);
        r.close();
        r.join(*this);
        return r;
    }
    // after close(): wide enough for the values of o too
    ADER_DEV void join(const FixFrame& o) {
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            e[v] = e[v] > o.e[v] ? e[v] : o.e[v];
            bad[v] |= o.bad[v];
        }
    }
    ADER_DEV Vec<NV, Fix> from(const FixFrame& o, const Vec<NV, Fix>& u) const {
        Vec<NV, Fix> r;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const unsigned d = e[v] - o.e[v];
            r[v].q = u[v].q >> (d < 63u ? d : 63u);
        }
        return r;
    }
    // the nearest FP64 value (ties away from zero)
    ADER_DEV double leave_one(int v, Fix u) const {
        const unsigned long long s = (unsigned long long)(u.q >> 63);
        const unsigned long long a = ((unsigned long long)u.q ^ s) - s;
        const unsigned hi = (unsigned)(a >> 32), lo = (unsigned)a;
        const unsigned top = hi ? hi : lo;
#ifdef __CUDA_ARCH__
        const unsigned lz = (unsigned)__clz((int)top) + (hi ? 0u : 32u);
#else
        const unsigned lz = (top ? (unsigned)__builtin_clz(top) : 32u) + (hi ? 0u : 32u);
#endif
        const unsigned long long n = ((a << (lz - 1u & 63u)) + 0x200ull) >> 10;       // bit 52 is the leading one
        const unsigned ex = e[v] + (unsigned)(11 - LSH) - lz - 1u;                     // its place adds one
        unsigned h = (unsigned)(n >> 32) + (ex << 20);
        h = a ? h : 0u;
        h |= ((unsigned)s & 0x80000000u) | bad[v];
        return of_bits((long long)(((unsigned long long)h << 32) | (unsigned)n));
    }
    ADER_DEV Vec<NV, double> leave(const Vec<NV, Fix>& u) const {
        Vec<NV, double> r;
#pragma unroll
        for (int v = 0; v < NV; ++v) r[v] = leave_one(v, u[v]);
        return r;
    }
};

// Multiplication of integers by c_d = dt / dx_d inside a frame: c_d is a 63-bit integer with the exponent of the largest
// of the three, the product the upper half of 128 bits; out() is the frame of the products.  The bits of an axis are cut
// at the unit of the largest c (an axis 2^10 times wider loses one and more), so the predictors scale in FP64, behind a
// direction's sum; the host check of the frames holds this form.
template <class FR> struct AxisScale;
template <int NV, int LSH>
struct AxisScale<FixFrame<NV, LSH>> {
    long long c[3];
    int k;
    ADER_DEV AxisScale(double cx, double cy, double cz) {
        const long long b[3] = {bits_of(cx), bits_of(cy), bits_of(cz)};
        int e[3];
        k = 0;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            e[d] = (int)((unsigned)((unsigned long long)b[d] >> 52) & 0x7ffu);
            k = e[d] > k ? e[d] : k;
        }
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const unsigned long long m = (((unsigned long long)b[d] & 0xfffffffffffffull) | 0x10000000000000ull) << 10;
            const int sh = k - e[d];
            const unsigned long long q = e[d] == 0 ? 0ull : m >> (sh < 63 ? sh : 63);
            const unsigned long long s = (unsigned long long)(b[d] >> 63);
            c[d] = (long long)((q ^ s) - s);             // c_d = c[d] 2^(k - 1023 - 62)
        }
    }
    template <int D> ADER_DEV Vec<NV, Fix> times(const Vec<NV, Fix>& f) const {
        Vec<NV, Fix> r;
#pragma unroll
        for (int v = 0; v < NV; ++v) r[v].q = fix_mulhi(f[v].q, c[D]);
        return r;
    }
    ADER_DEV FixFrame<NV, LSH> out(const FixFrame<NV, LSH>& f) const {
        FixFrame<NV, LSH> r = f;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const int e = (int)f.e[v] + 2 + k - 1023;
            r.e[v] = (unsigned)(e < 64 ? 64 : e);
            if (e > 2046 - 16 || k == 0x7ff) r.bad[v] = 0x7ff80000u;
        }
        return r;
    }
};

// Sum of the Euler flux of direction D over face nodes, kept by its factors so that a node costs few
// instructions (FP32 faces, one thread a zone): with r = 1 / rho, v = m_D r and w = |m|^2 r (twice the kinetic energy) the node adds m_i v to the
// momentum products, E v and w v to the energy's and w to the pressure's.  The pressure P = (gamma - 1)(E - w / 2)
// is applied to the sums, and the weighted sums of m_D and E themselves are the face averages of the state (the
// facial quadrature is exact on its basis).  14 instructions a node where the flux and its addition took 22.
template <int D, class R>
struct FluxSum {
    R p[3] = {R(0), R(0), R(0)}, w = R(0), ev = R(0), wv = R(0);

    ADER_DEV void add(const Vec<5, R>& u) {
        const R r = rcp(u[0]);
        const R v = u[1 + D] * r;
        const R k = (u[1] * u[1] + u[2] * u[2] + u[3] * u[3]) * r;
#pragma unroll
        for (int c = 0; c < 3; ++c) p[c] += u[1 + c] * v;
        w += k;
        ev += u[4] * v;
        wv += k * v;
    }
    // c times the sum; avg the face average of the state
    ADER_DEV Vec<5, R> mean(const Vec<5, R>& avg, R gm1, R c) const {
        Vec<5, R> f;
        f[0] = avg[1 + D];
#pragma unroll
        for (int i = 0; i < 3; ++i) f[1 + i] = c * p[i];
        f[1 + D] += gm1 * (avg[4] - (R(0.5) * c) * w);
        f[4] = c * (ev + gm1 * (ev - R(0.5) * wv));
        return f;
    }
};

// The frame of an order: integers for FP64, with LSH = 5 of the 10 bits below the mantissa at orders 2 and 3, and 3
// at order 4, whose node formulas form larger sums (up to 106 times a mode).
template <int LSH, int NV, class R> struct FrameAt { using T = PlainFrame<NV, R>; };
template <int LSH, int NV> struct FrameAt<LSH, NV, double> { using T = FixFrame<NV, LSH>; };
template <int ORDER, int NV, class R> using FrameOf = typename FrameAt<ORDER == 4 ? 3 : 5, NV, R>::T;

}  // namespace ader
