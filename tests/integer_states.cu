// Host check of the integer forms of FP64 work (fixed.cuh, weno.cuh): prints one line per property, "name value bound".
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include "../paper_1006_2146_gb300/csrc/weno.cuh"
using namespace ader;
typedef long double LD;

static double rnd() { return rand() / (double)RAND_MAX * 2 - 1; }
static void line(const char* name, double value, double bound) { std::printf("%s %.17g %.17g\n", name, value, bound); }

// a zone of three modes around 2^scale: sums of the modes, with the rounding of one unit per mode and one of FP64
template <int LSH>
static void frames(int scale) {
    double worst = 0, exact = 0, scaled = 0;
    for (int n = 0; n < 20000; ++n) {
        Vec<1, double> m[3];
        FixFrame<1, LSH> fr;
        const double top = std::ldexp(1.0, scale);
        for (int k = 0; k < 3; ++k) {
            m[k][0] = k == 0 ? top * (1 + 0.5 * rnd()) : top * rnd() * std::pow(2.0, -(rand() % 70));
            fr.include(m[k]);
        }
        fr.close();
        Vec<1, Fix> q[3];
        for (int k = 0; k < 3; ++k) q[k] = fr.enter(m[k]);
        exact = std::fmax(exact, std::fabs(fr.leave(q[0])[0] - m[0][0]) / top);
        const LD want = (LD)m[0][0] + 0.5L * m[1][0] - (LD)m[2][0] / 3;
        worst = std::fmax(worst, (double)(std::fabs((LD)fr.leave(q[0] + 0.5 * q[1] - q[2] / 3.0)[0] - want) / top));
        const double c[3] = {0.3 * (1 + rnd() * 0.9), 1e-5 * (1.5 + rnd()), 40 * (1.5 + rnd())};
        const AxisScale<FixFrame<1, LSH>> s(c[0], c[1], c[2]);
        const LD cw = c[0] * (LD)m[0][0] - c[1] * (LD)m[1][0] + c[2] * (LD)m[2][0];
        const double got = s.out(fr).leave(s.template times<0>(q[0]) - s.template times<1>(q[1]) + s.template times<2>(q[2]))[0];
        scaled = std::fmax(scaled, (double)(std::fabs(got - cw) / (c[2] * top)));
    }
    // the largest mode is held exactly; a sum carries at most 4 units of 2^-(52 + LSH) and FP64's half unit of 2^-52
    line("largest", exact, 0.0);
    line("sum", worst, 4 * std::ldexp(1.0, -52 - LSH) + std::ldexp(1.0, -52));
    // products: the same units times the largest factor, one unit of the upper half each, FP64's rounding
    line("scaled", scaled, 8 * std::ldexp(1.0, -52 - LSH) + std::ldexp(1.0, -51));
}

static void specials() {
    Vec<1, double> z, t, big;
    z[0] = 0.0;
    t[0] = -0.0;
    FixFrame<1, 5> f0;
    f0.include(z);
    f0.include(t);
    f0.close();
    line("zero", std::fabs(f0.leave(f0.enter(z) + f0.enter(t))[0]), 0.0);
    for (double bad : {(double)NAN, (double)INFINITY, -(double)INFINITY}) {
        big[0] = bad;
        FixFrame<1, 5> f;
        Vec<1, double> one;
        one[0] = 1.0;
        f.include(one);
        f.include(big);
        f.close();
        line("nonfinite", std::isnan(f.leave(f.enter(one))[0]) ? 0.0 : 1.0, 0.0);
    }
    const double u[7] = {2, 2, 2, 2, 2, 2, 2}, n[7] = {2, 2, (double)NAN, 2, 2, 2, 2};
    double b, c, d;
    weno3(u, b, c);
    line("uniform3", std::fabs(b) + std::fabs(c), 0.0);
    weno4(u, b, c, d);
    line("uniform4", std::fabs(b) + std::fabs(c) + std::fabs(d), 0.0);
    weno3(n, b, c);
    line("nan3", std::isnan(b) && std::isnan(c) ? 0.0 : 1.0, 0.0);
    weno4(n, b, c, d);
    line("nan4", std::isnan(b) && std::isnan(c) && std::isnan(d) ? 0.0 : 1.0, 0.0);
}

// blends against the same formulas in 80-bit arithmetic: within a few units of the largest neighbour difference
static void blends(double amp, int kind) {
    double e3 = 0, e4 = 0;
    for (int n = 0; n < 20000; ++n) {
        double a[7];
        const double k = 0.5 * rnd(), ph = 3 * rnd();
        for (int i = 0; i < 7; ++i)
            a[i] = kind == 0 ? amp * rnd() : kind == 1 ? 1 + amp * std::sin(k * i + ph) : (i < 1 + n % 6 ? amp : 0.1 * amp);
        double top = 0;
        for (int i = 0; i < 6; ++i) top = std::fmax(top, std::fabs(a[i + 1] - a[i]));
        if (top == 0) continue;
        auto blend = [](const LD (*x)[3], const LD* is, const LD* g, int S, int r) {
            LD w = 0, s = 0;
            for (int q = 0; q < S; ++q) {
                const LD t = 1e-12L + is[q], y = g[q] / (t * t);
                w += y * x[q][r];
                s += y;
            }
            return w / s;
        };
        const double* v = a + 1;
        const LD x3[3][3] = {{(3 * (LD)v[2] - 4 * (LD)v[1] + v[0]) / 2, ((LD)v[2] - 2 * (LD)v[1] + v[0]) / 2, 0},
                             {((LD)v[3] - v[1]) / 2, ((LD)v[3] - 2 * (LD)v[2] + v[1]) / 2, 0},
                             {(4 * (LD)v[3] - 3 * (LD)v[2] - v[4]) / 2, ((LD)v[4] - 2 * (LD)v[3] + v[2]) / 2, 0}};
        LD is[4];
        for (int q = 0; q < 3; ++q) is[q] = x3[q][0] * x3[q][0] + 13 * x3[q][1] * x3[q][1] / 3;
        const LD g3[3] = {1, 10, 1}, g4[4] = {1, 10, 10, 1};
        double b, c, d;
        weno3(v, b, c);
        e3 = std::fmax(e3, (double)std::fmax(std::fabs(b - blend(x3, is, g3, 3, 0)), std::fabs(c - blend(x3, is, g3, 3, 1))) / top);
        const LD m3 = a[0], m2 = a[1], m1 = a[2], u0 = a[3], p1 = a[4], p2 = a[5], p3 = a[6];
        const LD x4[4][3] = {{(109 * u0 - 177 * m1 + 87 * m2 - 19 * m3) / 60, (2 * u0 - 5 * m1 + 4 * m2 - m3) / 2, (u0 - 3 * m1 + 3 * m2 - m3) / 6},
                             {(33 * u0 - 63 * m1 + 11 * m2 + 19 * p1) / 60, (m1 + p1 - 2 * u0) / 2, (3 * m1 - 3 * u0 - m2 + p1) / 6},
                             {(63 * p1 - 33 * u0 - 19 * m1 - 11 * p2) / 60, (m1 + p1 - 2 * u0) / 2, (3 * u0 - m1 - 3 * p1 + p2) / 6},
                             {(177 * p1 - 109 * u0 - 87 * p2 + 19 * p3) / 60, (2 * u0 - 5 * p1 + 4 * p2 - p3) / 2, (3 * p1 - u0 - 3 * p2 + p3) / 6}};
        for (int q = 0; q < 4; ++q) {
            const LD t = x4[q][0] + x4[q][2] / 10;
            is[q] = t * t + 13 * x4[q][1] * x4[q][1] / 3 + 781 * x4[q][2] * x4[q][2] / 20;
        }
        weno4(a, b, c, d);
        e4 = std::fmax(e4, (double)std::fmax(std::fmax(std::fabs(b - blend(x4, is, g4, 4, 0)), std::fabs(c - blend(x4, is, g4, 4, 1))),
                                             std::fabs(d - blend(x4, is, g4, 4, 2))) / top);
    }
    // differences of the zone values round by half a unit of the difference (2^-53 each, factors up to 2 and 109 / 60 +
    // 68 / 60 + 19 / 60), the weights' t by a few units of 2^-53, which moves the blend by at most their spread
    line("weno3", e3, 32 * std::ldexp(1.0, -53));
    line("weno4", e4, 64 * std::ldexp(1.0, -53));
}

int main() {
    srand(11);
    for (int s : {-300, -40, 0, 37, 900}) {
        frames<2>(s);
        frames<5>(s);
    }
    specials();
    for (double amp : {1e-9, 1e-4, 0.3, 1e5, 1e40})
        for (int kind = 0; kind < 3; ++kind) blends(amp, kind);
    return 0;
}
