// Third order: ADER-CG predictor (modal Sec. IV.2, nodal App. B) and the
// x+ face quantities (Sec. V.2, App. D) of one zone.
//
// Modes m[1..15] use the paper's numbering (Eq. 15): m[1..10] = w1..w10,
// m[11..15] = u11..u15.  The scaled fluxes of Eq. 5 are c_d * F_d with
// c_d = dt / dx_d; the extraction rules are linear, so the scaling is applied
// to the extracted flux modes.
#pragma once
#include "common.cuh"
#include "fixed.cuh"
#include "modes.cuh"
#include "team.cuh"

namespace ader {
namespace o3 {


// ------------------------------------------------------------------ modal, Sec. IV.2
// SRC: with a non-stiff source (s = dt S at every node of the current iterate,
// Eqs. 40-43 with f, g, h -> s, Eq. 36 with its source terms); sdt receives
// dt S-bar of Eq. 44 from the source at the final iterate.
template <class T, bool SRC = false>
ADER_DEV void predict_modal(const T& t, typename T::V* m, PredCtl& ctl, const Src<typename T::R>* src = nullptr,
                            typename T::V* sdt = nullptr) {
    using R = typename T::R;
    using V = typename T::V;
    constexpr int NL = T::NL;
    using FR = FrameOf<3, NL, R>;
    using VS = Vec<NL, typename FR::S>;
    const R cx = t.cx, cy = t.cy, cz = t.cz;
    // Eq. 38: the thirteen tau = 0 nodes of Eq. 37, and the parts of the tau = 1/2 nodes (Eq. 39) that do not
    // change with the iterate: base[k] is node 14 + k without its evolutionary modes
    FR fr;
    V u[14], base[6];
    {
        VS w[11], s[14];
#pragma unroll
        for (int k = 1; k <= 10; ++k) fr.include(m[k]);
        fr.close();
#pragma unroll
        for (int k = 1; k <= 10; ++k) w[k] = fr.enter(m[k]);
        s[1] = w[1] - (w[5] + w[6] + w[7]) / 12.0;
        s[2] = s[1] + 0.5 * (w[2] + w[3]) + 0.25 * (w[5] + w[6] + w[8]);
        s[3] = s[2] - w[3] - 0.5 * w[8];
        s[4] = s[1] + 0.5 * (w[2] + w[4]) + 0.25 * (w[5] + w[7] + w[10]);
        s[5] = s[4] - w[4] - 0.5 * w[10];
        s[6] = s[3] - w[2] + w[3];
        s[7] = s[2] - w[2] - w[3];
        s[8] = s[5] - w[2] + w[4];
        s[9] = s[4] - w[2] - w[4];
        s[10] = s[1] + 0.5 * (w[3] + w[4]) + 0.25 * (w[6] + w[7] + w[9]);
        s[11] = s[10] - w[3] - 0.5 * w[9];
        s[12] = s[11] + w[3] - w[4];
        s[13] = s[10] - w[3] - w[4];
        const VS b14 = 0.25 * (s[2] + s[3] + s[4] + s[5]) - 0.125 * (w[6] + w[7]);
        const VS b16 = 0.25 * (s[2] + s[6] + s[10] + s[12]) - 0.125 * (w[5] + w[7]);
        const VS b18 = 0.25 * (s[4] + s[8] + s[10] + s[11]) - 0.125 * (w[5] + w[6]);
        base[0] = fr.leave(b14);
        base[1] = fr.leave(b14 - w[2]);
        base[2] = fr.leave(b16);
        base[3] = fr.leave(b16 - w[3]);
        base[4] = fr.leave(b18);
        base[5] = fr.leave(b18 - w[4]);
#pragma unroll
        for (int k = 1; k <= 13; ++k) u[k] = fr.leave(s[k]);
    }
    // fluxes at the tau = 0 nodes, built once (Sec. IV.2); the sums of Eqs. 40-42 in the state scalar (up to 16 times a
    // flux), one frame per direction, and Eq. 36's sum over the directions in R
    V e11, e13, e14, e15;       // Eq. 36 without sources: the modes fed by tau = 0 fluxes alone
    {
        using FF = typename FrameAt<2, NL, R>::T;
        using VF = Vec<NL, typename FF::S>;
        V fn[14], gn[14], hn[14];
        t.template fluxes<13, 0, false>(u + 1, fn + 1, gn + 1, hn + 1);
        // one direction after the other: the values of one frame at a time
        auto enter = [&](const V* x, FF& ff, VF* f) {
#pragma unroll
            for (int n = 1; n <= 13; ++n) ff.include(x[n]);
            ff.close();
#pragma unroll
            for (int n = 1; n <= 13; ++n) f[n] = ff.enter(x[n]);
        };
        {
            FF ff;
            VF f[14];
            enter(fn, ff, f);
            const VF q1 = f[2] + f[3] + f[4] + f[5], q2 = f[6] + f[7] + f[8] + f[9], q3 = f[10] + f[11] + f[12] + f[13];
            e11 = scale(cx, ff.leave(0.25 * (q1 - q2)));                                // F2
            e13 = scale(cx, ff.leave(2.0 * (0.5 * (q1 + q2 - q3) - 2.0 * f[1])));       // 2 F5
            e14 = scale(cx, ff.leave(f[2] - f[3] - f[6] + f[7]));                       // F8
            e15 = scale(cx, ff.leave(f[4] - f[5] - f[8] + f[9]));                       // F10
        }
        {
            FF ff;
            VF g[14];
            enter(gn, ff, g);
            const VF q4 = g[2] + g[6] + g[10] + g[12], q5 = g[3] + g[7] + g[11] + g[13], q6 = g[4] + g[5] + g[8] + g[9];
            e11 += scale(cy, ff.leave(0.25 * (q4 - q5)));                               // G3
            e13 += scale(cy, ff.leave(g[2] - g[3] - g[6] + g[7]));                      // G8
            e14 += scale(cy, ff.leave(2.0 * (0.5 * (q4 + q5 - q6) - 2.0 * g[1])));      // 2 G6
            e15 += scale(cy, ff.leave(g[10] - g[11] - g[12] + g[13]));                  // G9
        }
        {
            FF ff;
            VF h[14];
            enter(hn, ff, h);
            const VF q7 = h[4] + h[8] + h[10] + h[11], q8 = h[5] + h[9] + h[12] + h[13], q9 = h[2] + h[3] + h[6] + h[7];
            e11 = -(e11 + scale(cz, ff.leave(0.25 * (q7 - q8))));                       // H4
            e13 = -(e13 + scale(cz, ff.leave(h[4] - h[5] - h[8] + h[9])));              // H10
            e14 = -(e14 + scale(cz, ff.leave(h[10] - h[11] - h[12] + h[13])));          // H9
            e15 = -(e15 + scale(cz, ff.leave(2.0 * (0.5 * (q7 + q8 - q9) - 2.0 * h[1]))));   // 2 H7
        }
    }
    // source modes from the tau = 0 nodes (Eqs. 40-43 with f, g, h -> s), built once
    V S1, S2, S3, S4, s1;
    if constexpr (SRC) {
        V sn[14];
        t.template sources<13>(u + 1, *src, sn + 1);
        const V a1 = sn[2] + sn[3] + sn[4] + sn[5], a2 = sn[6] + sn[7] + sn[8] + sn[9];
        const V a3 = sn[10] + sn[11] + sn[12] + sn[13];
        const V b4 = sn[2] + sn[6] + sn[10] + sn[12], b5 = sn[3] + sn[7] + sn[11] + sn[13];
        const V b6 = sn[4] + sn[5] + sn[8] + sn[9];
        const V c7 = sn[4] + sn[8] + sn[10] + sn[11], c8 = sn[5] + sn[9] + sn[12] + sn[13];
        const V c9 = sn[2] + sn[3] + sn[6] + sn[7];
        S2 = 0.25 * (a1 - a2);
        S3 = 0.25 * (b4 - b5);
        S4 = 0.25 * (c7 - c8);
        const V S5 = 0.5 * (a1 + a2 - a3) - 2.0 * sn[1];
        const V S6 = 0.5 * (b4 + b5 - b6) - 2.0 * sn[1];
        const V S7 = 0.5 * (c7 + c8 - c9) - 2.0 * sn[1];
        s1 = sn[1];
        S1 = s1 + (S5 + S6 + S7) / 12.0;
    }
    const bool conv = positive_arg(ctl.tol);
    const int cap = conv ? ctl.max_iter : ctl.n_iter;
    R ref = R(1);
    if (conv) ref = t.zone_max(max_abs(m[1])) + R(sizeof(R) == 8 ? 1e-300 : 1e-30);   // never zero in R
    ctl.iters = 0;
    bool done = false;                  // this zone has converged (others of the team may go on)
    for (int it = 0; it < cap; ++it) {
        // Eq. 39: the tau = 1/2 nodes (node 20 serves only source terms)
        // in the order of T::fluxes: x+, x-, y+, y-, z+, z-
        const V half = 0.5 * m[11] + 0.25 * m[12];
        const V ut[6] = {base[0] + half + 0.25 * m[13], base[1] + half - 0.25 * m[13],
                         base[2] + half + 0.25 * m[14], base[3] + half - 0.25 * m[14],
                         base[4] + half + 0.25 * m[15], base[5] + half - 0.25 * m[15]};
        V ft[2], gt[2], ht[2];
        t.template fluxes<0, 2, true>(ut, ft, gt, ht);
        // Eqs. 40-42 give F13 = 2 (cx (f14 - f15) - F2) and so on, and Eq. 36 u12 = -(F13 + G14 + H15) / 2 =
        // -u11 - sum_d c_d (f_d(upper) - f_d(lower))
        V n11 = e11;
        V n12 = -e11 - ((ft[0] - ft[1]) + (gt[0] - gt[1]) + (ht[0] - ht[1]));
        V n13 = e13, n14 = e14, n15 = e15;
        if constexpr (SRC) {
            const V us[7] = {ut[0], ut[1], ut[2], ut[3], ut[4], ut[5], u[1] + m[11] + m[12]};
            V st[7];
            t.template sources<7>(us, *src, st);
            const V s14 = st[0], s15 = st[1], s16 = st[2], s17 = st[3], s18 = st[4], s19 = st[5], s20 = st[6];
            const V S13 = 2.0 * (s14 - s15 - S2), S14 = 2.0 * (s16 - s17 - S3), S15 = 2.0 * (s18 - s19 - S4);
            const V S11 = 2.0 * (s14 + s15 + s16 + s17 + s18 + s19 - 6.0 * S1) / 3.0 - s20 + s1;
            const V S12 = s20 - s1 - S11;
            n11 += S1 - 0.3 * S12;
            n12 += 0.5 * S11 + 0.6 * S12;
            n13 += S2 + (2.0 / 3.0) * S13;
            n14 += S3 + (2.0 / 3.0) * S14;
            n15 += S4 + (2.0 / 3.0) * S15;
        }
        R change = R(0);
        if (!t.waits(done)) {
            if (conv)
                change = fmax(fmax(fmax(max_abs_diff(n11, m[11]), max_abs_diff(n12, m[12])),
                                   fmax(max_abs_diff(n13, m[13]), max_abs_diff(n14, m[14]))),
                              max_abs_diff(n15, m[15]));
            m[11] = n11;
            m[12] = n12;
            m[13] = n13;
            m[14] = n14;
            m[15] = n15;
            ++ctl.iters;
        }
        if (conv) {
            change = t.zone_max(change);
            done = done || change < R(ctl.tol) * ref;
            if (!t.any(!done)) break;
        }
    }
    ctl.capped = conv && !done;
    if constexpr (SRC) {        // Eq. 44 from the source at the final iterate's tau > 0 nodes (Eq. 39)
        const V half = 0.5 * m[11] + 0.25 * m[12];
        const V us[7] = {base[0] + half + 0.25 * m[13], base[1] + half - 0.25 * m[13],
                         base[2] + half + 0.25 * m[14], base[3] + half - 0.25 * m[14],
                         base[4] + half + 0.25 * m[15], base[5] + half - 0.25 * m[15], u[1] + m[11] + m[12]};
        V st[7];
        t.template sources<7>(us, *src, st);
        const V ssum = st[0] + st[1] + st[2] + st[3] + st[4] + st[5], s20 = st[6];
        const V S11 = 2.0 * (ssum - 6.0 * S1) / 3.0 - s20 + s1;
        const V S12 = s20 - s1 - S11;
        *sdt = S1 + 0.5 * S11 + S12 / 3.0;
    }
}

// ------------------------------------------------------------------ nodal, App. B
// SRC: with a non-stiff source (s = dt S at nodes 1-7 once and at the tau > 0
// nodes of the current iterate; the source terms of Eqs. B.2-B.3); sdt
// receives dt S-bar of Eq. B.6 from the source at the final iterate.
template <class T, bool SRC = false>
ADER_DEV void predict_nodal(const T& t, typename T::V* m, PredCtl& ctl, const Src<typename T::R>* src = nullptr,
                            typename T::V* sdt = nullptr) {
    using R = typename T::R;
    using V = typename T::V;
    constexpr int NL = T::NL;
    using FR = FrameOf<3, NL, R>;
    using VS = Vec<NL, typename FR::S>;
    const R cx = t.cx, cy = t.cy, cz = t.cz;
    // Eq. B.4: the ten tau = 0 nodes of Eq. B.1
    FR fr;
    V u[11];
    {
        VS w[11], s[11];
#pragma unroll
        for (int k = 1; k <= 10; ++k) fr.include(m[k]);
        fr.close();
#pragma unroll
        for (int k = 1; k <= 10; ++k) w[k] = fr.enter(m[k]);
        s[1] = w[1] - (w[5] + w[6] + w[7]) / 12.0;
        s[2] = s[1] + 0.5 * w[2] + 0.25 * w[5];
        s[3] = 2.0 * s[1] - s[2] + 0.5 * w[5];
        s[4] = s[1] + 0.5 * w[3] + 0.25 * w[6];
        s[5] = 2.0 * s[1] - s[4] + 0.5 * w[6];
        s[6] = s[1] + 0.5 * w[4] + 0.25 * w[7];
        s[7] = 2.0 * s[1] - s[6] + 0.5 * w[7];
        s[8] = s[4] + s[6] - s[1] + 0.25 * w[9];
        s[9] = s[2] + s[6] - s[1] + 0.25 * w[10];
        s[10] = s[2] + s[4] - s[1] + 0.25 * w[8];
#pragma unroll
        for (int k = 1; k <= 10; ++k) u[k] = fr.leave(s[k]);
    }
    // Eq. B.2 without sources.  Each direction enters it through four differences of its fluxes; for x
    //   X = f3 - f1, A = (f2 - f1) + X / 2, f4 - f10 and f6 - f9
    // (1.5 f1 - f2 - f3 / 2 = -A and f2 + f3 - 2 f1 = A + X / 2), for y and z the same with the axes exchanged.
    V q11, q12, q13, q14, q15;
    {
        // all directions at nodes 1, 2, 4, 6, 8, 9, 10; x alone at 3, y at 5, z at 7; the differences of a direction in
        // the state scalar, one frame per direction, and their sum in R
        using FF = typename FrameAt<2, NL, R>::T;
        using VF = Vec<NL, typename FF::S>;
        const V un[10] = {u[1], u[2], u[4], u[6], u[8], u[9], u[10], u[3], u[5], u[7]};
        V fn[8], gn[8], hn[8];
        t.template fluxes<7, 1, false>(un, fn, gn, hn);
        FF ff, fg, fh;
        VF f[8], g[8], h[8];
#pragma unroll
        for (int n = 0; n < 8; ++n) {
            if (n != 4) ff.include(fn[n]);
            if (n != 5) fg.include(gn[n]);
            if (n != 6) fh.include(hn[n]);
        }
        ff.close();
        fg.close();
        fh.close();
#pragma unroll
        for (int n = 0; n < 8; ++n) {
            if (n != 4) f[n] = ff.enter(fn[n]);
            if (n != 5) g[n] = fg.enter(gn[n]);
            if (n != 6) h[n] = fh.enter(hn[n]);
        }
        auto sum = [&](const VF& x, const VF& y, const VF& z) {
            return scale(cx, ff.leave(x)) + scale(cy, fg.leave(y)) + scale(cz, fh.leave(z));
        };
        const VF X = f[7] - f[0], Y = g[7] - g[0], Z = h[7] - h[0];
        const VF ax = f[1] - f[0] + 0.5 * X, ay = g[2] - g[0] + 0.5 * Y, az = h[3] - h[0] + 0.5 * Z;
        q11 = u[1] + 0.5 * sum(X, Y, Z);
        q12 = u[2] + sum(-ax, g[1] - g[6] + ay, h[1] - h[5] + az);
        q13 = u[4] + sum(f[2] - f[6] + ax, -ay, h[2] - h[4] + az);
        q14 = u[6] + sum(f[3] - f[5] + ax, g[3] - g[4] + ay, -az);
        q15 = u[1] + sum(0.5 * X + ax, 0.5 * Y + ay, 0.5 * Z + az);   // u1 + sum_d c_d (A + X / 2)
    }
    V s0sum, s1;         // with a source: s2 + ... + s7 and s1 (nodes 1-7, built once)
    if constexpr (SRC) {          // Eq. B.2, source terms
        V sn[8];
        t.template sources<7>(u + 1, *src, sn + 1);
        s1 = sn[1];
        s0sum = sn[2] + sn[3] + sn[4] + sn[5] + sn[6] + sn[7];
        q11 += (-9.0 * sn[1] + 2.0 * s0sum) / 24.0;
        q12 += (7.0 * sn[1] - 10.0 * sn[2] - 6.0 * sn[3] + 2.0 * s0sum) / 24.0;
        q13 += (7.0 * sn[1] - 10.0 * sn[4] - 6.0 * sn[5] + 2.0 * s0sum) / 24.0;
        q14 += (7.0 * sn[1] - 10.0 * sn[6] - 6.0 * sn[7] + 2.0 * s0sum) / 24.0;
        q15 += (-27.0 * sn[1] + 5.0 * s0sum) / 30.0;
    }
    // initial guess: the evolutionary modes in m[11..15] (zero: no time evolution) at the
    // tau > 0 nodes of Eq. B.1
    const V g0 = 0.5 * m[11] + 0.25 * m[12];
    V u11 = u[1] + g0, u12 = u[2] + g0 + 0.25 * m[13], u13 = u[4] + g0 + 0.25 * m[14];
    V u14 = u[6] + g0 + 0.25 * m[15], u15 = u[1] + m[11] + m[12];
    const bool conv = positive_arg(ctl.tol);
    const int cap = conv ? ctl.max_iter : ctl.n_iter;
    R ref = R(1);
    if (conv) ref = t.zone_max(max_abs(m[1])) + R(sizeof(R) == 8 ? 1e-300 : 1e-30);   // never zero in R
    ctl.iters = 0;
    bool done = false;                  // this zone has converged (others of the team may go on)
    for (int it = 0; it < cap; ++it) {
        // Eq. B.3 without sources (node 15 serves only source terms)
        const V ua[4] = {u11, u12, u13, u14};
        const V q1 = t.axis_differences(ua, R(0.5));
        if constexpr (SRC) {      // Eq. B.3 with its source terms, at the current iterate
            const V us[5] = {u11, u12, u13, u14, u15};
            V se[5];
            t.template sources<5>(us, *src, se);
            if (!t.waits(done)) {
                const V q2 = q1 + (-4.0 * se[0] - 3.0 * se[4]) / 24.0;
                u11 = q11 + q1 + 0.125 * (4.0 * se[0] - se[4]);
                u12 = q12 + q2 + (2.0 / 3.0) * se[1];
                u13 = q13 + q2 + (2.0 / 3.0) * se[2];
                u14 = q14 + q2 + (2.0 / 3.0) * se[3];
                u15 = q15 + 4.0 * q1 + 0.1 * (8.0 * se[0] + se[4]);
            }
        } else if (!t.waits(done)) {
            u11 = q11 + q1;
            u12 = q12 + q1;
            u13 = q13 + q1;
            u14 = q14 + q1;
            u15 = q15 + 4.0 * q1;
        }
        if (!t.waits(done)) ++ctl.iters;
        if (conv) {
            R change = R(0);
            if (!t.waits(done)) {
                // Eq. B.5 each iteration, to measure the change in mode space
                const V n12 = 2.0 * (u15 - 2.0 * u11 + u[1]);
                const V n11 = 2.0 * (u11 - u[1] - 0.25 * n12);
                const V n13 = 4.0 * (u12 - u11 - u[2] + u[1]);
                const V n14 = 4.0 * (u13 - u11 - u[4] + u[1]);
                const V n15 = 4.0 * (u14 - u11 - u[6] + u[1]);
                change = fmax(fmax(fmax(max_abs_diff(n11, m[11]), max_abs_diff(n12, m[12])),
                                   fmax(max_abs_diff(n13, m[13]), max_abs_diff(n14, m[14]))),
                              max_abs_diff(n15, m[15]));
                m[11] = n11;
                m[12] = n12;
                m[13] = n13;
                m[14] = n14;
                m[15] = n15;
            }
            change = t.zone_max(change);
            done = done || change < R(ctl.tol) * ref;
            if (!t.any(!done)) break;
        }
    }
    ctl.capped = conv && !done;
    if (!conv) {
        // Eq. B.5: nodal -> modal
        FR fm;
        const V in[9] = {u[1], u[2], u[4], u[6], u11, u12, u13, u14, u15};
        VS s[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) fm.include(in[k]);
        fm.close();
#pragma unroll
        for (int k = 0; k < 9; ++k) s[k] = fm.enter(in[k]);
        const VS n12 = 2.0 * (s[8] - 2.0 * s[4] + s[0]);
        m[12] = fm.leave(n12);
        m[11] = fm.leave(2.0 * (s[4] - s[0] - 0.25 * n12));
        m[13] = fm.leave(4.0 * (s[5] - s[4] - s[1] + s[0]));
        m[14] = fm.leave(4.0 * (s[6] - s[4] - s[2] + s[0]));
        m[15] = fm.leave(4.0 * (s[7] - s[4] - s[3] + s[0]));
    }
    if constexpr (SRC)            // Eq. B.6 from the source at the final iterate (times dt)
    {
        const V us[2] = {u11, u15};
        V se[2];
        t.template sources<2>(us, *src, se);
        *sdt = (-5.0 * s1 + s0sum + 4.0 * se[0] + se[1]) / 6.0;
    }
}

// ------------------------------------------------------------------ x+ face, Sec. V.2 and App. D
// p = the zone's modes in the face's x-frame (modes.cuh).  The barycentre state (Eq. 61), the face average of u
// (Eq. 62) and the face average of the physical normal flux: composing Eq. D.9 with D.10 gives
// <F> = (F1 + F6 + F7 + F8 + F9 + F10) / 6 over the facial nodes of Eq. D.6 (the four corner nodes enter only the
// edge averages).
// Both x-faces of one direction at once (FP32 Euler).  p is in the frame of the upper face; the lower face's frame
// differs only in the sign of the modes odd in the normal coordinate (2, 8, 10, 13), so each of the node states of
// Eq. D.8 is E + O on the upper face and E - O on the lower one, with E its part from the even modes and O from the
// odd ones, each computed once; the nodes are taken in an order that keeps few of them alive at a time.
// Index 0 of ub, avg, Fa is the upper face (S = +1), index 1 the lower.
template <int D, class R>
ADER_DEV void face_pair(const Vec<5, R>* p, R gm1, Vec<5, R>* ub, Vec<5, R>* avg, Vec<5, R>* Fa) {
    using V = Vec<5, R>;
    const V t1e = p[1] + (2.0 * p[5] - p[6] - p[7]) / 12.0, t1o = 0.5 * p[2];
    const V q1e = 0.5 * p[11] + 0.25 * p[12], q1o = 0.25 * p[13];
    {
        const V ube = t1e + q1e, ubo = t1o + q1o;
        const V avge = ube + (p[6] + p[7] + p[12]) / 12.0;
        ub[0] = ube + ubo;
        ub[1] = ube - ubo;
        avg[0] = avge + ubo;
        avg[1] = avge - ubo;
    }
    FluxSum<D, R> up, lo;
    up.add(t1e + t1o);                                                        // node 1
    lo.add(t1e - t1o);
    {
        const V e = t1e + p[11] + p[12], o = t1o + 0.5 * p[13];                   // node 10
        up.add(e + o);
        lo.add(e - o);
    }
    const V t2e = t1e + 0.5 * (p[3] + p[4]) + 0.25 * (p[6] + p[7] + p[9]), t2o = t1o + 0.25 * (p[8] + p[10]);
    const V t3e = t2e - p[3] - 0.5 * p[9], t3o = t2o - 0.5 * p[8];
    const V t4e = t2e - p[4] - 0.5 * p[9], t4o = t2o - 0.5 * p[10];
    {
        const V e = 0.5 * (t2e + t4e) + q1e + 0.25 * (p[14] - p[7]), o = 0.5 * (t2o + t4o) + q1o;   // 6
        up.add(e + o);
        lo.add(e - o);
    }
    {
        const V e = 0.5 * (t2e + t3e) + q1e + 0.25 * (p[15] - p[6]), o = 0.5 * (t2o + t3o) + q1o;   // 8
        up.add(e + o);
        lo.add(e - o);
    }
    const V t5e = t4e - p[3] + 0.5 * p[9], t5o = t4o - 0.5 * p[8];
    {
        const V e = 0.5 * (t4e + t5e) + q1e - 0.25 * (p[6] + p[15]), o = 0.5 * (t4o + t5o) + q1o;   // 9
        up.add(e + o);
        lo.add(e - o);
    }
    {
        const V e = 0.5 * (t3e + t5e) + q1e - 0.25 * (p[7] + p[14]), o = 0.5 * (t3o + t5o) + q1o;   // 7
        up.add(e + o);
        lo.add(e - o);
    }
    Fa[0] = up.mean(avg[0], gm1, R(1.0 / 6.0));
    Fa[1] = lo.mean(avg[1], gm1, R(1.0 / 6.0));
}

// One face at a time: the barycentre state, the face average and all ten facial nodes of Eq. D.6 (Eq. D.8).
template <bool ALL, class V>
ADER_DEV void face_states(const V* p, V& ub, V& avg, V* t) {
    ub = p[1] + 0.5 * (p[2] + p[11]) + 0.25 * (p[12] + p[13]) + (2.0 * p[5] - p[6] - p[7]) / 12.0;
    avg = ub + (p[6] + p[7] + p[12]) / 12.0;
    const V q1 = 0.5 * p[11] + 0.25 * (p[12] + p[13]);
    t[1] = p[1] + 0.5 * p[2] + (2.0 * p[5] - p[6] - p[7]) / 12.0;
    t[2] = t[1] + 0.5 * (p[3] + p[4]) + 0.25 * (p[6] + p[7] + p[8] + p[9] + p[10]);
    t[3] = t[2] - p[3] - 0.5 * (p[8] + p[9]);
    t[4] = t[2] - p[4] - 0.5 * (p[9] + p[10]);
    t[5] = t[4] - p[3] - 0.5 * (p[8] - p[9]);
    t[6] = 0.5 * (t[2] + t[4]) + q1 + 0.25 * (p[14] - p[7]);
    t[7] = 0.5 * (t[3] + t[5]) + q1 - 0.25 * (p[7] + p[14]);
    t[8] = 0.5 * (t[2] + t[3]) + q1 + 0.25 * (p[15] - p[6]);
    t[9] = 0.5 * (t[4] + t[5]) + q1 - 0.25 * (p[6] + p[15]);
    t[10] = t[1] + p[11] + p[12] + 0.5 * p[13];
}

// composing Eq. D.9 with D.10 the face average of the flux needs six of the nodes (the four corner nodes enter only
// the edge averages)
constexpr int FACE_NODES = 10, MEAN_NODES = 6;
ADER_DEV constexpr int mean_node(int k) { return k == 0 ? 1 : k + 5; }
template <class F_>
ADER_DEV auto face_mean(const F_& F) {
    return (F[1] + F[6] + F[7] + F[8] + F[9] + F[10]) / 6.0;
}

// the edge averages (Eqs. D.9-D.10) of the facial flux f[n] on the edges of the transverse
// direction s (0: t1, 1: t2), upper and lower
template <class V>
ADER_DEV void edge_fluxes(const V* f, int s, V& plus, V& minus) {
    // Eq. D.9 (the modes the edge averages need)
    const V q2 = 0.5 * (f[2] + f[4] - 4.0 * f[1] + f[3] + f[5]);
    const V q3 = f[6] + f[7] - f[8] - f[9];
    const V m1 = (2.0 / 3.0) * (f[1] + 0.125 * (f[2] + f[3] + f[4] + f[5]));
    const V m2 = 0.5 * (f[2] + f[4] - f[3] - f[5]);
    const V m3 = 0.5 * (f[2] + f[3] - f[4] - f[5]);
    const V m4 = q2 + q3, m5 = q2 - q3;
    const V m8 = 2.0 * (f[1] + f[10]) - (f[6] + f[7] + f[8] + f[9]) + q2;
    const V m7 = f[10] - f[1] - m8;
    const V m9 = 2.0 * (f[6] - f[7] - m2);
    const V m10 = 2.0 * (f[8] - f[9] - m3);
    // Eq. D.10
    const V af = m1 + 0.5 * m7 + m8 / 3.0;
    const V qs = s == 0 ? 0.5 * m2 + 0.25 * m9 : 0.5 * m3 + 0.25 * m10;
    plus = af + qs + (s == 0 ? m4 : m5) / 6.0;
    minus = plus - 2.0 * qs;
}

// Edge-averaged states (Eq. 63) on the edges t1+, t1-, t2+, t2-.
template <class V>
ADER_DEV void edge_states(const V* p, const V& ub, const V& avg, V* e) {
    (void)ub;
    const V q1 = 0.5 * p[3] + 0.25 * (p[8] + p[14]), q2 = 0.5 * p[4] + 0.25 * (p[10] + p[15]);
    const V u1 = avg + p[6] / 6.0 + q1, u2 = avg + p[7] / 6.0 + q2;
    e[0] = u1;
    e[1] = u1 - 2.0 * q1;
    e[2] = u2;
    e[3] = u2 - 2.0 * q2;
}

}  // namespace o3
}  // namespace ader
