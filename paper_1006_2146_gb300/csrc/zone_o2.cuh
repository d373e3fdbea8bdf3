// Second order: ADER-CG predictor (modal Sec. IV.1, nodal App. A) and the x+
// face quantities (Sec. V.1, App. D).  Modes m[1..5] (Eq. 14).
#pragma once
#include "common.cuh"
#include "fixed.cuh"
#include "modes.cuh"
#include "team.cuh"

namespace ader {
namespace o2 {

// The update without sources uses only tau = 0 fluxes, so one step reaches the fixed point (in converged mode a second
// step confirms it).  With a source the update of u5 depends on u5 through the source at the tau = 1 node, so each
// iteration recomputes it: `next(m5)` gives the new u5 for the current one.
template <class T, class Next>
ADER_DEV void iterate_o2(const T& t, typename T::V* m, PredCtl& ctl, Next next) {
    using R = typename T::R;
    using V = typename T::V;
    const bool conv = positive_arg(ctl.tol);
    const int cap = conv ? ctl.max_iter : ctl.n_iter;
    R ref = R(1);
    if (conv) ref = t.zone_max(max_abs(m[1])) + R(sizeof(R) == 8 ? 1e-300 : 1e-30);   // never zero in R
    ctl.iters = 0;
    bool done = false;                  // this zone has converged (others of the team may go on)
    for (int it = 0; it < cap; ++it) {
        const V n5 = next(m[5]);
        R change = R(0);
        if (!t.waits(done)) {
            change = max_abs_diff(n5, m[5]);
            m[5] = n5;
            ++ctl.iters;
        }
        if (conv) {
            change = t.zone_max(change);
            done = done || change < R(ctl.tol) * ref;
            if (!t.any(!done)) break;
        }
    }
    ctl.capped = conv && !done;
}

// Eqs. 31-33 and 30; with a source Eqs. 34-35: s at the seven nodes of Eq. 31 (node 7 = u1 + u5 at tau = 1), sdt
// receives dt S-bar from the final iterate
template <class T, bool SRC = false>
ADER_DEV void predict_modal(const T& t, typename T::V* m, PredCtl& ctl, const Src<typename T::R>* src = nullptr,
                            typename T::V* sdt = nullptr) {
    using V = typename T::V;
    // x+, x-, y+, y-, z+, z-, the order of T::fluxes
    const V u[6] = {m[1] + 0.5 * m[2], m[1] - 0.5 * m[2], m[1] + 0.5 * m[3],
                    m[1] - 0.5 * m[3], m[1] + 0.5 * m[4], m[1] - 0.5 * m[4]};
    V f[2], g[2], h[2];
    t.template fluxes<0, 2, false>(u, f, g, h);
    const V div = scale(t.cx, f[0] - f[1]) + scale(t.cy, g[0] - g[1]) + scale(t.cz, h[0] - h[1]);
    if constexpr (SRC) {
        V s[6], s7;
        t.template sources<6>(u, *src, s);
        const V s1 = (s[0] + s[1] + s[2] + s[3] + s[4] + s[5]) / 6.0;                  // Eq. 34
        const V base = s1 - div;
        iterate_o2(t, m, ctl, [&](const V& m5) {
            const V u7 = m[1] + m5;
            V s5;
            t.template sources<1>(&u7, *src, &s5);
            return base + (2.0 / 3.0) * (s5 - s1);                                     // Eqs. 34 and 30
        });
        const V u7 = m[1] + m[5];
        t.template sources<1>(&u7, *src, &s7);
        *sdt = s1 + 0.5 * (s7 - s1);                                                   // Eq. 35 (times dt)
    } else {
        iterate_o2(t, m, ctl, [&](const V&) { return -div; });
    }
}

// Eqs. A.5, A.4 (h term at node 4, the zeta node of Eq. A.1) and A.6; with a source A.7: s at node 1 (tau = 0) and
// node 5 (tau = 1)
template <class T, bool SRC = false>
ADER_DEV void predict_nodal(const T& t, typename T::V* m, PredCtl& ctl, const Src<typename T::R>* src = nullptr,
                            typename T::V* sdt = nullptr) {
    using V = typename T::V;
    using R = typename T::R;
    const V u1 = m[1];
    const V u[4] = {u1, m[1] + 0.5 * m[2], m[1] + 0.5 * m[3], m[1] + 0.5 * m[4]};
    const V d = t.axis_differences(u, R(2));                // 2 sum_d c_d (F_d(u1) - F_d(u_{1+d}))
    if constexpr (SRC) {
        V s1, s5;
        t.template sources<1>(&u1, *src, &s1);
        const V base = d + s1 / 3.0;
        iterate_o2(t, m, ctl, [&](const V& m5) {
            const V u5 = u1 + m5;
            V s;
            t.template sources<1>(&u5, *src, &s);
            return base + (2.0 / 3.0) * s;                                             // Eqs. A.4 and A.6
        });
        const V u5 = u1 + m[5];
        t.template sources<1>(&u5, *src, &s5);
        *sdt = 0.5 * (s1 + s5);                                                        // Eq. A.7 (times dt)
    } else {
        iterate_o2(t, m, ctl, [&](const V&) { return d; });
    }
}

// Eqs. 58-59 and D.3-D.5: composing D.4 with D.5, <F> is the mean of the flux
// at the four tau = 1/2 facial nodes (node 5 enters only through the time mode).
template <int D, class R>
ADER_DEV void face(const Vec<5, R>* p, R gm1, Vec<5, R>& ub, Vec<5, R>& avg, Vec<5, R>& Fa) {
    ub = p[1] + 0.5 * (p[2] + p[5]);
    avg = ub;
    FluxSum<D, R> sum;
    sum.add(ub + 0.5 * p[3]);
    sum.add(ub - 0.5 * p[3]);
    sum.add(ub + 0.5 * p[4]);
    sum.add(ub - 0.5 * p[4]);
    Fa = sum.mean(avg, gm1, R(0.25));
}

// The states of a face and its five nodes (Eqs. 58-59, D.3), and the mean of the flux at the first four.
template <bool ALL, class V>
ADER_DEV void face_states(const V* p, V& ub, V& avg, V* t) {
    ub = p[1] + 0.5 * (p[2] + p[5]);
    avg = ub;
    t[1] = ub + 0.5 * p[3];
    t[2] = ub - 0.5 * p[3];
    t[3] = ub + 0.5 * p[4];
    t[4] = ub - 0.5 * p[4];
    if (ALL) t[5] = ub + 0.5 * p[5];
}
constexpr int FACE_NODES = 5, MEAN_NODES = 4;
ADER_DEV constexpr int mean_node(int k) { return k + 1; }
template <class F_>
ADER_DEV auto face_mean(const F_& F) {
    return 0.25 * (F[1] + F[2] + F[3] + F[4]);
}

// the edge averages (Eqs. D.4-D.5) of the facial flux f[n] on the edges of the transverse direction
// s (0: t1, 1: t2), upper and lower
template <class V>
ADER_DEV void edge_fluxes(const V* f, int s, V& plus, V& minus) {
    const V m2 = f[1] - f[2], m3 = f[3] - f[4];
    const V m4 = 2.0 * f[5] - 0.5 * (f[1] + f[2] + f[3] + f[4]);
    const V af = f[5] - m4 + 0.5 * m4;
    const V half = 0.5 * (s == 0 ? m2 : m3);
    plus = af + half;
    minus = af - half;
}

// Edge-averaged states (Eq. 60) on the edges t1+, t1-, t2+, t2-.
template <class V>
ADER_DEV void edge_states(const V* p, const V& ub, const V& avg, V* e) {
    (void)avg;
    e[0] = ub + 0.5 * p[3];
    e[1] = ub - 0.5 * p[3];
    e[2] = ub + 0.5 * p[4];
    e[3] = ub - 0.5 * p[4];
}

}  // namespace o2
}  // namespace ader
