// Host check that small signals keep their relative accuracy in the FP64 forms that work on integers (fixed.cuh,
// weno.cuh).  Prints "name value bound" lines: relative errors against 80-bit arithmetic.
#include <cmath>
#include <cstdio>
#include <cstdlib>

#include "../paper_1006_2146_gb300/csrc/weno.cuh"
#include "../paper_1006_2146_gb300/csrc/step_inst.cuh"
using namespace ader;
typedef long double LD;

template <int ORDER, int FORM, int NV, class R>
static void predict(const double (*w)[8], const double* c, Vec<NV, R>* m) {
    SerialTeam<NV, R> t;
    t.gm1 = R(0.4);
    t.cx = R(c[0]);
    t.cy = R(c[1]);
    t.cz = R(c[2]);
    constexpr int L = ModeCount<ORDER>::L;
    for (int k = 1; k <= L; ++k)
        for (int v = 0; v < NV; ++v) m[k][v] = k <= ModeCount<ORDER>::LS ? R(w[k][v]) : R(0);
    PredCtl ctl{ORDER - 1, 0.0, 0, 0, false};
    if (FORM == FORM_MODAL) ZoneOps<ORDER>::template predict_modal<false>(t, m, ctl, nullptr, nullptr);
    else ZoneOps<ORDER>::template predict_nodal<false>(t, m, ctl, nullptr, nullptr);
}

// A momentum of amplitude a across a uniform flow along axis d, varying along d: only the flux of direction d carries it,
// beside the pressure in the other directions' fluxes of the same variable (which it does not change: a^2 is below the
// pressure's last place in either arithmetic).  c_d is the smallest of the three.
template <int ORDER, int FORM, int NV>
static void transverse(const char* name, double bound) {
    constexpr int L = ModeCount<ORDER>::L;
    double worst = 0;
    for (double a : {1e-12, 1e-14, 1e-17, 1e-30})
        for (int d = 0; d < 3; ++d)
            for (int e = 1; e < 3; ++e) {
                const int v = 1 + (d + e) % 3;
                double w[36][8] = {}, c[3] = {0.21, 0.17, 0.13};
                c[d] = 3e-5;
                w[1][0] = 1.1;
                w[1][1 + d] = 0.37;
                w[1][4] = 2.6;
                w[2 + d][v] = 0.9 * a;
                if (ORDER >= 3) w[5 + d][v] = -0.31 * a;
                if (ORDER == 4) w[11 + d][v] = 0.17 * a;
                Vec<NV, double> m[L + 1];
                Vec<NV, LD> l[L + 1];
                predict<ORDER, FORM, NV, double>(w, c, m);
                predict<ORDER, FORM, NV, LD>(w, c, l);
                // in units of the largest scaled flux
                const double unit = c[d] * 0.37 / 1.1 * a;
                for (int k = ModeCount<ORDER>::LS + 1; k <= L; ++k)
                    worst = std::fmax(worst, (double)std::fabs(m[k][v] - l[k][v]) / unit);
            }
    std::printf("%s %.17g %.17g\n", name, worst, bound);
}

// The largest time mode of a uniform oblique flow: exactly zero.
template <int ORDER, int FORM, int NV, class R>
static void uniform(const char* name) {
    constexpr int L = ModeCount<ORDER>::L;
    const double c[3] = {0.21, 0.17, 0.13}, state[8] = {1.1, 0.37, -0.53, 0.71, 2.6, 0.9, -0.4, 0.7};
    double w[36][8] = {}, worst = 0;
    for (int v = 0; v < NV; ++v) w[1][v] = state[v];
    Vec<NV, R> m[L + 1];
    predict<ORDER, FORM, NV, R>(w, c, m);
    for (int k = ModeCount<ORDER>::LS + 1; k <= L; ++k)
        for (int v = 0; v < NV; ++v) worst = std::fmax(worst, (double)std::fabs(m[k][v]));
    std::printf("%s %.17g 0\n", name, worst);
}

// A smooth signal of size s beside a jump of 1 at one or two of the stencil's end values: the blend is of the stencils
// that the jump does not reach.
static void beside_a_jump(const char* name, double bound) {
    const double x[7] = {0.31, 0.62, 0.90, 1.27, 1.75, 2.31, 2.96};
    double worst = 0;
    for (double s : {1e-4, 1e-6, 1e-10, 1e-14, 1e-17})
        for (int n = 1; n <= 2; ++n)
            for (int end = 0; end < 2; ++end) {
                double a[7], b, c, d;
                LD l[7], bl, cl, dl;
                for (int k = 0; k < 7; ++k) {
                    a[k] = (end ? k >= 7 - n : k < n) ? 1.0 + 0.1 * k : s * x[k];
                    l[k] = a[k];
                }
                weno4(a, b, c, d);
                weno4(l, bl, cl, dl);
                worst = std::fmax(worst, (double)std::fabs((b - bl) / bl));
                worst = std::fmax(worst, (double)std::fabs((c - cl) / bl));
                worst = std::fmax(worst, (double)std::fabs((d - dl) / bl));
            }
    std::printf("%s %.17g %.17g\n", name, worst, bound);
}

int main() {
    // A flux carries four roundings, a mode's sums amplify them by at most 16 (order 3) and 212 (order 4), and the
    // order's further iterations add the same again.
    const double b3 = std::ldexp(1.0, -53 + 2 + 4 + 1), b4 = std::ldexp(1.0, -53 + 2 + 8 + 2);
    transverse<2, FORM_MODAL, 5>("modal2", b3);
    transverse<2, FORM_NODAL, 5>("nodal2", b3);
    // (the nodal form takes its time modes from differences of node values: their last places too)
    transverse<3, FORM_NODAL, 5>("nodal3", b3 + std::ldexp(1.0, -53 + 4) / (3e-5 * 0.37 / 1.1));
    transverse<3, FORM_MODAL, 5>("modal3", b3);
    transverse<3, FORM_MODAL, 8>("modal3_mhd", b3);
    transverse<4, FORM_MODAL, 5>("modal4", b4);
    transverse<4, FORM_MODAL, 8>("modal4_mhd", b4);
    uniform<2, FORM_NODAL, 5, double>("uniform2");
    uniform<2, FORM_NODAL, 8, double>("uniform2_mhd");
    uniform<2, FORM_NODAL, 5, float>("uniform2_f32");
    uniform<3, FORM_NODAL, 5, double>("uniform3");
    uniform<3, FORM_NODAL, 8, double>("uniform3_mhd");
    uniform<3, FORM_NODAL, 5, float>("uniform3_f32");
    // 60 b sums up to 196 differences of a unit and more; a blend's weights carry a few roundings and move it by its spread
    beside_a_jump("weno4", std::ldexp(1.0, -53 + 6));
    return 0;
}
