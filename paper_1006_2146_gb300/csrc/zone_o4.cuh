// Fourth order: ADER-CG predictor (modal Sec. IV.3, nodal App. C) and the x+
// face quantities (Sec. V.3, App. D).  Modes m[1..35] (Eq. 16).
#pragma once
#include "common.cuh"
#include "fixed.cuh"
#include "modes.cuh"
#include "nodal_o4_coeffs.cuh"
#include "team.cuh"

namespace ader {
namespace o4 {


// ------------------------------------------------------------------ modal, Sec. IV.3
// SRC: with a non-stiff source (s = dt S at every node of Eq. 46 of the current iterate; the source
// modes by Eqs. 49-51 with f, g, h -> s and Eq. 52; Eq. 45 with its source terms); sdt receives dt S-bar
// of Eq. 53 from the final iterate.
template <class T, bool SRC = false>
ADER_DEV void predict_modal(const T& t, typename T::V* m, PredCtl& ctl, const Src<typename T::R>* src = nullptr,
                            typename T::V* sdt = nullptr) {
    using R = typename T::R;
    using V = typename T::V;
    constexpr int NL = T::NL;
    using FR = FrameOf<4, NL, R>;
    using VS = Vec<NL, typename FR::S>;
    const R cx = t.cx, cy = t.cy, cz = t.cz;
    // Eq. 47: the 21 tau = 0 nodes of Eq. 46
    FR fr;
    VS s[22], w[21];
    {
#pragma unroll
        for (int k = 1; k <= 20; ++k) fr.include(m[k]);
        fr.close();
#pragma unroll
        for (int k = 1; k <= 20; ++k) w[k] = fr.enter(m[k]);
        s[1] = w[1] - (w[5] + w[6] + w[7]) / 12.0;
        s[2] = s[1] + (60.0 * w[2] + 30.0 * w[5] + 6.0 * w[11] - 5.0 * w[16] - 5.0 * w[18]) / 120.0;
        s[3] = 0.5 * (s[1] + s[2]) - 0.015625 * (4.0 * w[5] + 3.0 * w[11]);
        s[4] = 3.0 * s[1] + s[2] - 3.0 * s[3] - 0.09375 * w[11];
        s[5] = 6.0 * s[1] + 3.0 * s[2] - 8.0 * s[3] - 0.375 * w[11];
        s[6] = s[1] + (60.0 * w[3] + 30.0 * w[6] + 6.0 * w[12] - 5.0 * w[14] - 5.0 * w[19]) / 120.0;
        s[7] = 0.5 * (s[1] + s[6]) - 0.015625 * (4.0 * w[6] + 3.0 * w[12]);
        s[8] = 3.0 * s[1] + s[6] - 3.0 * s[7] - 0.09375 * w[12];
        s[9] = 6.0 * s[1] + 3.0 * s[6] - 8.0 * s[7] - 0.375 * w[12];
        s[10] = s[1] + (60.0 * w[4] + 30.0 * w[7] + 6.0 * w[13] - 5.0 * w[15] - 5.0 * w[17]) / 120.0;
        s[11] = 0.5 * (s[1] + s[10]) - 0.015625 * (4.0 * w[7] + 3.0 * w[13]);
        s[12] = 3.0 * s[1] + s[10] - 3.0 * s[11] - 0.09375 * w[13];
        s[13] = 6.0 * s[1] + 3.0 * s[10] - 8.0 * s[11] - 0.375 * w[13];
        s[14] = s[2] + s[7] + s[10] - 2.0 * s[1] + 0.25 * (w[3] + w[8] + w[9] + w[10]) + (5.0 / 48.0) * (w[14] + w[19]) +
                (23.0 / 320.0) * w[12] + 0.125 * (w[15] + w[16] + w[17] + w[18] + w[20]) + 0.1875 * w[6];
        s[15] = s[14] + s[9] - s[6] - 0.5 * (w[8] + w[9]) - 0.25 * (w[14] + w[19] + w[20]);
        s[16] = s[14] + s[13] - s[10] - 0.5 * (w[9] + w[10]) - 0.25 * (w[15] + w[17] + w[20]);
        s[18] = s[14] + s[5] - s[2] - 0.5 * (w[8] + w[10]) - 0.25 * (w[16] + w[18] + w[20]);
        s[19] = s[18] + s[9] - s[6] + 0.5 * (w[8] - w[9]) - 0.25 * (w[14] + w[19] - w[20]);
        s[20] = s[18] + s[13] - s[10] - 0.5 * (w[9] - w[10]) - 0.25 * (w[15] + w[17] - w[20]);
        s[17] = s[15] + s[16] - s[14] + w[9] + 0.5 * w[20];
        s[21] = s[19] + s[20] - s[18] + w[9] - 0.5 * w[20];
    }

    // tau = 0 parts of Eqs. 49-51 (built once), in the state scalar: sums of up to 212 fluxes, a frame per direction
    using FF = typename FrameAt<2, NL, R>::T;
    using VF = Vec<NL, typename FF::S>;
    FF ff, fg, fh;
    VF F2, F5, F8, F10, F11, F20, PF14, PF15, PF16, QF12;
    VF G3, G6, G8, G9, G12, G20, PG14, PG15, PG16, QG34;
    VF H4, H7, H9, H10, H13, H20, PH14, PH15, PH16, QH56;
    {
        V u[22], fn[22], gn[22], hn[22];
        VF f[22], g[22], h[22];
#pragma unroll
        for (int k = 1; k <= 21; ++k) u[k] = fr.leave(s[k]);
        t.template fluxes<21, 0, false>(u + 1, fn + 1, gn + 1, hn + 1);
#pragma unroll
        for (int k = 1; k <= 21; ++k) {
            ff.include(fn[k]);
            fg.include(gn[k]);
            fh.include(hn[k]);
        }
        ff.close();
        fg.close();
        fh.close();
#pragma unroll
        for (int k = 1; k <= 21; ++k) {
            f[k] = ff.enter(fn[k]);
            g[k] = fg.enter(gn[k]);
            h[k] = fh.enter(hn[k]);
        }
        // q1..q6 of Eqs. 49-51 (corner sums), per flux
        const VF fq1 = f[14] + f[15] + f[16] + f[17], fq2 = f[18] + f[19] + f[20] + f[21];
        const VF fq3 = f[14] + f[16] + f[18] + f[20], fq4 = f[15] + f[17] + f[19] + f[21];
        const VF fq5 = f[14] + f[15] + f[18] + f[19], fq6 = f[16] + f[17] + f[20] + f[21];
        F5 = 2.0 * (f[2] - 2.0 * f[1] + f[5]);
        F8 = 0.5 * (f[14] - f[15] + f[16] - f[17] - f[18] + f[19] - f[20] + f[21]);
        F10 = 0.5 * (f[14] + f[15] - f[16] - f[17] - f[18] - f[19] + f[20] + f[21]);
        F11 = (16.0 / 3.0) * (f[2] - 2.0 * f[3] + 2.0 * f[4] - f[5]);
        F2 = (2.0 / 3.0) * (f[2] - f[5]) - 0.1 * F11 + (fq1 - fq2) / 12.0;
        F20 = f[14] - f[15] - f[16] + f[17] - f[18] + f[19] + f[20] - f[21];
        PF14 = 0.5 * (fq3 - fq4) - 2.0 * (f[6] - f[9]);
        PF15 = 0.5 * (fq5 - fq6) - 2.0 * (f[10] - f[13]);
        PF16 = 0.5 * (fq1 - fq2) - 2.0 * (f[2] - f[5]);
        QF12 = fq1 - fq2;
        const VF gq1 = g[14] + g[15] + g[16] + g[17], gq2 = g[18] + g[19] + g[20] + g[21];
        const VF gq3 = g[14] + g[16] + g[18] + g[20], gq4 = g[15] + g[17] + g[19] + g[21];
        const VF gq5 = g[14] + g[15] + g[18] + g[19], gq6 = g[16] + g[17] + g[20] + g[21];
        G6 = 2.0 * (g[6] - 2.0 * g[1] + g[9]);
        G8 = 0.5 * (g[14] - g[15] + g[16] - g[17] - g[18] + g[19] - g[20] + g[21]);
        G9 = 0.5 * (g[14] - g[15] - g[16] + g[17] + g[18] - g[19] - g[20] + g[21]);
        G12 = (16.0 / 3.0) * (g[6] - 2.0 * g[7] + 2.0 * g[8] - g[9]);
        G3 = (2.0 / 3.0) * (g[6] - g[9]) - 0.1 * G12 + (gq3 - gq4) / 12.0;
        G20 = g[14] - g[15] - g[16] + g[17] - g[18] + g[19] + g[20] - g[21];
        PG14 = 0.5 * (gq3 - gq4) - 2.0 * (g[6] - g[9]);
        PG15 = 0.5 * (gq5 - gq6) - 2.0 * (g[10] - g[13]);
        PG16 = 0.5 * (gq1 - gq2) - 2.0 * (g[2] - g[5]);
        QG34 = gq3 - gq4;
        const VF hq1 = h[14] + h[15] + h[16] + h[17], hq2 = h[18] + h[19] + h[20] + h[21];
        const VF hq3 = h[14] + h[16] + h[18] + h[20], hq4 = h[15] + h[17] + h[19] + h[21];
        const VF hq5 = h[14] + h[15] + h[18] + h[19], hq6 = h[16] + h[17] + h[20] + h[21];
        H7 = 2.0 * (h[10] - 2.0 * h[1] + h[13]);
        H9 = 0.5 * (h[14] - h[15] - h[16] + h[17] + h[18] - h[19] - h[20] + h[21]);
        H10 = 0.5 * (h[14] + h[15] - h[16] - h[17] - h[18] - h[19] + h[20] + h[21]);
        H13 = (16.0 / 3.0) * (h[10] - 2.0 * h[11] + 2.0 * h[12] - h[13]);
        H4 = (2.0 / 3.0) * (h[10] - h[13]) - 0.1 * H13 + (hq5 - hq6) / 12.0;
        H20 = h[14] - h[15] - h[16] + h[17] - h[18] + h[19] + h[20] - h[21];
        PH14 = 0.5 * (hq3 - hq4) - 2.0 * (h[6] - h[9]);
        PH15 = 0.5 * (hq5 - hq6) - 2.0 * (h[10] - h[13]);
        PH16 = 0.5 * (hq1 - hq2) - 2.0 * (h[2] - h[5]);
        QH56 = hq5 - hq6;
    }
    // source modes from the tau = 0 nodes (Eqs. 49-52 with f, g, h -> s), built once
    V s1, S1, S2, S3, S4, S5, S6, S7, S8, S9, S10, PS14, PS15, PS16, QS12, QS34, QS56;
    if constexpr (SRC) {
        V u[22], sn[22];
#pragma unroll
        for (int k = 1; k <= 21; ++k) u[k] = fr.leave(s[k]);
        t.template sources<21>(u + 1, *src, sn + 1);
        const V a1 = sn[14] + sn[15] + sn[16] + sn[17], a2 = sn[18] + sn[19] + sn[20] + sn[21];
        const V a3 = sn[14] + sn[16] + sn[18] + sn[20], a4 = sn[15] + sn[17] + sn[19] + sn[21];
        const V a5 = sn[14] + sn[15] + sn[18] + sn[19], a6 = sn[16] + sn[17] + sn[20] + sn[21];
        s1 = sn[1];
        S5 = 2.0 * (sn[2] - 2.0 * sn[1] + sn[5]);
        S6 = 2.0 * (sn[6] - 2.0 * sn[1] + sn[9]);
        S7 = 2.0 * (sn[10] - 2.0 * sn[1] + sn[13]);
        S8 = 0.5 * (sn[14] - sn[15] + sn[16] - sn[17] - sn[18] + sn[19] - sn[20] + sn[21]);
        S9 = 0.5 * (sn[14] - sn[15] - sn[16] + sn[17] + sn[18] - sn[19] - sn[20] + sn[21]);
        S10 = 0.5 * (sn[14] + sn[15] - sn[16] - sn[17] - sn[18] - sn[19] + sn[20] + sn[21]);
        const V S11 = (16.0 / 3.0) * (sn[2] - 2.0 * sn[3] + 2.0 * sn[4] - sn[5]);
        const V S12 = (16.0 / 3.0) * (sn[6] - 2.0 * sn[7] + 2.0 * sn[8] - sn[9]);
        const V S13 = (16.0 / 3.0) * (sn[10] - 2.0 * sn[11] + 2.0 * sn[12] - sn[13]);
        S2 = (2.0 / 3.0) * (sn[2] - sn[5]) - 0.1 * S11 + (a1 - a2) / 12.0;
        S3 = (2.0 / 3.0) * (sn[6] - sn[9]) - 0.1 * S12 + (a3 - a4) / 12.0;
        S4 = (2.0 / 3.0) * (sn[10] - sn[13]) - 0.1 * S13 + (a5 - a6) / 12.0;
        PS14 = 0.5 * (a3 - a4) - 2.0 * (sn[6] - sn[9]);
        PS15 = 0.5 * (a5 - a6) - 2.0 * (sn[10] - sn[13]);
        PS16 = 0.5 * (a1 - a2) - 2.0 * (sn[2] - sn[5]);
        QS12 = a1 - a2;
        QS34 = a3 - a4;
        QS56 = a5 - a6;
        S1 = 0.125 * (a1 + a2) - (S5 + S6 + S7) / 6.0;
    }
    // the time modes of the source (Eqs. 49-52 with f, g, h -> s) from the nodes 22..42 of an iterate
    auto time_source_modes = [&](const V* w, V* ts) {
        V sw[43];
        t.template sources<21>(w + 22, *src, sw + 22);
        const V q7 = sw[23] + sw[24] - sw[25] - sw[26] - sw[27] - sw[28] + sw[29] + sw[30];
        const V q8 = sw[23] + sw[27] - sw[24] - sw[28] - sw[31] - sw[33] + sw[32] + sw[34];
        const V q9 = sw[25] + sw[29] - sw[26] - sw[30] - sw[31] - sw[32] + sw[33] + sw[34];
        const V q10 = sw[23] + sw[24] + sw[25] + sw[26] - sw[27] - sw[28] - sw[29] - sw[30];
        const V q11 = sw[23] - sw[24] + sw[27] - sw[28] + sw[31] - sw[32] + sw[33] - sw[34];
        const V q12 = sw[25] - sw[26] + sw[29] - sw[30] + sw[31] + sw[32] - sw[33] - sw[34];
        const V S16 = q7 + PS16, S18 = -2.0 * q7 + S16;
        const V S14 = q8 + PS14, S19 = -2.0 * q8 + S14;
        const V S15 = q9 + PS15, S17 = -2.0 * q9 + S15;
        // ts[k - 21] = s mode k for k = 21..35
        ts[6] = 1.125 * QS12 + 4.5 * (sw[36] - sw[37]) - 2.25 * q10;                               // 27
        ts[3] = 3.0 * (sw[36] - sw[37]) - 0.75 * q10 + 0.375 * (S16 + S18) - ts[6];                // 24
        ts[7] = 1.125 * QS34 + 4.5 * (sw[38] - sw[39]) - 2.25 * q11;                               // 28
        ts[4] = 3.0 * (sw[38] - sw[39]) - 0.75 * q11 + 0.375 * (S14 + S19) - ts[7];                // 25
        ts[8] = 1.125 * QS56 + 4.5 * (sw[40] - sw[41]) - 2.25 * q12;                               // 29
        ts[5] = 3.0 * (sw[40] - sw[41]) - 0.75 * q12 + 0.375 * (S15 + S17) - ts[8];                // 26
        ts[9] = 3.0 * (sw[36] - 2.0 * sw[35] + sw[37]) - 1.5 * S5;                                // 30
        ts[10] = 3.0 * (sw[38] - 2.0 * sw[35] + sw[39]) - 1.5 * S6;                               // 31
        ts[11] = 3.0 * (sw[40] - 2.0 * sw[35] + sw[41]) - 1.5 * S7;                               // 32
        ts[12] = 3.0 * (sw[23] - sw[27] - sw[24] + sw[28]) - 3.0 * S8;                            // 33
        ts[13] = 3.0 * (sw[31] - sw[32] - sw[33] + sw[34]) - 3.0 * S9;                            // 34
        ts[14] = 3.0 * (sw[25] - sw[29] - sw[26] + sw[30]) - 3.0 * S10;                           // 35
        ts[2] = 4.5 * (sw[42] - s1) - 13.5 * (sw[35] - sw[22]);                                   // 23 (Eq. 52)
        ts[1] = 2.25 * (s1 - sw[22] - sw[35] + sw[42]) - 1.5 * ts[2];                              // 22
        ts[0] = sw[42] - s1 - ts[1] - ts[2] + (ts[9] + ts[10] + ts[11]) / 12.0;                        // 21
    };
    // Eq. 48: the tau > 0 nodes 22..41 of Eq. 46 of the current iterate (22 and 42 serve only source
    // terms; 42 = (0, 0, 0, 1) only with a source)
    auto build_w = [&](V* out) {
        const FR fw = fr.extended(m + 21, 15);
        VS x[43], u[22], y[21], e[15];
#pragma unroll
        for (int k = 1; k <= 21; ++k) u[k] = fw.from(fr, s[k]);
#pragma unroll
        for (int k = 1; k <= 20; ++k) y[k] = fw.from(fr, w[k]);
#pragma unroll
        for (int k = 0; k < 15; ++k) e[k] = fw.enter(m[21 + k]);
        x[22] = u[1] + (36.0 * e[0] + 12.0 * e[1] + 4.0 * e[2] - 3.0 * e[9] - 3.0 * e[10] - 3.0 * e[11]) / 108.0;
        x[23] = x[22] + u[2] + u[6] - 2.0 * u[1] +
                (18.0 * y[8] + 9.0 * y[14] + 9.0 * y[16] + 12.0 * e[3] + 12.0 * e[4] + 4.0 * e[6] + 4.0 * e[7] +
                 6.0 * e[9] + 6.0 * e[10] + 6.0 * e[12]) / 72.0;
        x[24] = x[23] - u[6] + u[9] - 0.5 * y[8] - 0.25 * y[14] - (6.0 * e[4] + 2.0 * e[7] + 3.0 * e[12]) / 18.0;
        x[25] = 0.5 * (u[14] + u[15] + x[23] + x[24]) - u[2] - 0.5 * y[6] - 0.25 * y[16] - 0.125 * y[17] +
                (6.0 * e[5] + 2.0 * e[8] - 3.0 * e[10] + 3.0 * e[11] + 3.0 * e[14]) / 36.0;
        x[26] = x[23] + x[24] - x[25] - 0.5 * (y[6] - y[7]) - 0.25 * (y[16] - y[18]) - (e[10] - e[11]) / 6.0;
        x[27] = u[5] + x[23] - u[2] - 0.5 * y[8] - 0.25 * y[16] - (6.0 * e[3] + 2.0 * e[6] + 3.0 * e[12]) / 18.0;
        x[28] = u[9] + x[27] - u[6] + 0.5 * y[8] - 0.25 * y[14] - (6.0 * e[4] + 2.0 * e[7] - 3.0 * e[12]) / 18.0;
        x[29] = 0.5 * (u[18] + u[19] + x[27] + x[28]) - u[5] - 0.5 * y[6] + 0.25 * y[16] - 0.125 * y[17] +
                (6.0 * e[5] + 2.0 * e[8] - 3.0 * e[10] + 3.0 * e[11] - 3.0 * e[14]) / 36.0;
        x[30] = x[27] + x[28] - x[29] - 0.5 * (y[6] - y[7]) + 0.25 * (y[16] - y[18]) - (e[10] - e[11]) / 6.0;
        x[31] = 0.5 * (u[14] + u[18] + x[25] + x[29]) - u[10] - 0.5 * y[5] - 0.25 * y[15] - 0.125 * y[14] +
                (6.0 * e[4] + 2.0 * e[7] - 3.0 * e[9] + 3.0 * e[10] + 3.0 * e[13]) / 36.0;
        x[32] = u[9] + x[31] - u[6] - 0.5 * y[9] - 0.25 * y[19] - (6.0 * e[4] + 2.0 * e[7] + 3.0 * e[13]) / 18.0;
        x[33] = x[23] + x[27] - x[31] - 0.5 * (y[5] - y[7]) - 0.25 * (y[14] - y[19]) - (e[9] - e[11]) / 6.0;
        x[34] = x[24] + x[28] - x[32] - 0.5 * (y[5] - y[7]) + 0.25 * (y[14] - y[19]) - (e[9] - e[11]) / 6.0;
        const VS r1 = (36.0 * e[0] + 24.0 * e[1] + 16.0 * e[2]) / 54.0;
        const VS r2 = (18.0 * e[3] + 12.0 * e[6]) / 54.0;
        const VS r3 = (6.0 * e[9] - 3.0 * e[10] - 3.0 * e[11]) / 54.0;
        const VS r4 = (18.0 * e[4] + 12.0 * e[7]) / 54.0;
        const VS r5 = (-3.0 * e[9] + 6.0 * e[10] - 3.0 * e[11]) / 54.0;
        const VS r6 = (18.0 * e[5] + 12.0 * e[8]) / 54.0;
        const VS r7 = (-3.0 * e[9] - 3.0 * e[10] + 6.0 * e[11]) / 54.0;
        x[35] = 2.0 * x[22] - u[1] + 2.0 * (e[1] + e[2]) / 9.0;
        x[36] = u[2] + r1 + r2 + r3;
        x[37] = u[5] + r1 - r2 + r3;
        x[38] = u[6] + r1 + r4 + r5;
        x[39] = u[9] + r1 - r4 + r5;
        x[40] = u[10] + r1 + r6 + r7;
        x[41] = u[13] + r1 - r6 + r7;
        if constexpr (SRC) x[42] = u[1] + e[0] + e[1] + e[2] - (e[9] + e[10] + e[11]) / 12.0;   // (0, 0, 0, 1)
        if constexpr (SRC) out[22] = fw.leave(x[22]);
#pragma unroll
        for (int k = 23; k <= (SRC ? 42 : 41); ++k) out[k] = fw.leave(x[k]);
    };
    // Eq. 45 without sources: the modes fed by tau = 0 fluxes only
    V e21, e24, e25, e26;
    {
        auto sum = [&](const VF& x, const VF& y, const VF& z) {
            return scale(cx, ff.leave(x)) + scale(cy, fg.leave(y)) + scale(cz, fh.leave(z));
        };
        e21 = -sum(F2 + 0.1 * F11, G3 + 0.1 * G12, H4 + 0.1 * H13);
        e24 = -sum(2.0 * F5, G8, H10);
        e25 = -sum(F8, 2.0 * G6, H9);
        e26 = -sum(F10, G9, 2.0 * H7);
    }

    const bool conv = positive_arg(ctl.tol);
    const int cap = conv ? ctl.max_iter : ctl.n_iter;
    R ref = R(1);
    if (conv) ref = t.zone_max(max_abs(m[1])) + R(sizeof(R) == 8 ? 1e-300 : 1e-30);   // never zero in R
    ctl.iters = 0;
    bool done = false;                  // this zone has converged (others of the team may go on)
    for (int it = 0; it < cap; ++it) {
        V w[43];
        build_w(w);
        // fluxes at nodes 23..35 (all three directions) and the axis nodes 36..41
        V fn[38], gn[38], hn[38];
        t.template fluxes<13, 2, false>(w + 23, fn + 23, gn + 23, hn + 23);
        FF fi, gi, hi;
        VF f[38], g[38], h[38];
#pragma unroll
        for (int k = 23; k <= 37; ++k) {
            fi.include(fn[k]);
            gi.include(gn[k]);
            hi.include(hn[k]);
        }
        fi.close();
        gi.close();
        hi.close();
        fi.join(ff);
        gi.join(fg);
        hi.join(fh);
#pragma unroll
        for (int k = 23; k <= 37; ++k) {
            f[k] = fi.enter(fn[k]);
            g[k] = gi.enter(gn[k]);
            h[k] = hi.enter(hn[k]);
        }
        // a tau = 0 part in this iterate's frame
        auto keepx = [&](const VF& x) { return fi.from(ff, x); };
        auto keepy = [&](const VF& x) { return gi.from(fg, x); };
        auto keepz = [&](const VF& x) { return hi.from(fh, x); };
        auto sum = [&](const VF& x, const VF& y, const VF& z) {
            return scale(cx, fi.leave(x)) + scale(cy, gi.leave(y)) + scale(cz, hi.leave(z));
        };
        const VF f36 = f[36], f37 = f[37], g38 = g[36], g39 = g[37], h40 = h[36], h41 = h[37];
        // Eq. 49 (x)
        VF F14, F15, F16, F18, F24, F27, F30, F33, F35;
        {
            const VF q7 = f[23] + f[24] - f[25] - f[26] - f[27] - f[28] + f[29] + f[30];
            const VF q8 = f[23] + f[27] - f[24] - f[28] - f[31] - f[33] + f[32] + f[34];
            const VF q9 = f[25] + f[29] - f[26] - f[30] - f[31] - f[32] + f[33] + f[34];
            const VF q10 = f[23] + f[24] + f[25] + f[26] - f[27] - f[28] - f[29] - f[30];
            F14 = q8 + keepx(PF14);
            F15 = q9 + keepx(PF15);
            F16 = q7 + keepx(PF16);
            F18 = -2.0 * q7 + F16;
            F27 = 1.125 * keepx(QF12) + 4.5 * (f36 - f37) - 2.25 * q10;
            F24 = 3.0 * (f36 - f37) - 0.75 * q10 + 0.375 * (F16 + F18) - F27;
            F30 = 3.0 * (f36 - 2.0 * f[35] + f37) - 1.5 * keepx(F5);
            F33 = 3.0 * (f[23] - f[27] - f[24] + f[28]) - 3.0 * keepx(F8);
            F35 = 3.0 * (f[25] - f[29] - f[26] + f[30]) - 3.0 * keepx(F10);
        }
        // Eq. 50 (y)
        VF G14, G16, G17, G19, G25, G28, G31, G33, G34;
        {
            const VF q7 = g[23] + g[24] - g[25] - g[26] - g[27] - g[28] + g[29] + g[30];
            const VF q8 = g[23] + g[27] - g[24] - g[28] - g[31] - g[33] + g[32] + g[34];
            const VF q9 = g[25] + g[29] - g[26] - g[30] - g[31] - g[32] + g[33] + g[34];
            const VF q11 = g[23] - g[24] + g[27] - g[28] + g[31] - g[32] + g[33] - g[34];
            G14 = q8 + keepy(PG14);
            const VF G15 = q9 + keepy(PG15);
            G16 = q7 + keepy(PG16);
            G17 = -2.0 * q9 + G15;
            G19 = -2.0 * q8 + G14;
            G28 = 1.125 * keepy(QG34) + 4.5 * (g38 - g39) - 2.25 * q11;
            G25 = 3.0 * (g38 - g39) - 0.75 * q11 + 0.375 * (G14 + G19) - G28;
            G31 = 3.0 * (g38 - 2.0 * g[35] + g39) - 1.5 * keepy(G6);
            G33 = 3.0 * (g[23] - g[27] - g[24] + g[28]) - 3.0 * keepy(G8);
            G34 = 3.0 * (g[31] - g[32] - g[33] + g[34]) - 3.0 * keepy(G9);
        }
        // Eq. 51 (z)
        VF H15, H17, H18, H19, H26, H29, H32, H34, H35;
        {
            const VF q7 = h[23] + h[24] - h[25] - h[26] - h[27] - h[28] + h[29] + h[30];
            const VF q8 = h[23] + h[27] - h[24] - h[28] - h[31] - h[33] + h[32] + h[34];
            const VF q9 = h[25] + h[29] - h[26] - h[30] - h[31] - h[32] + h[33] + h[34];
            const VF q12 = h[25] - h[26] + h[29] - h[30] + h[31] + h[32] - h[33] - h[34];
            const VF H14 = q8 + keepz(PH14);
            H15 = q9 + keepz(PH15);
            const VF H16 = q7 + keepz(PH16);
            H17 = -2.0 * q9 + H15;
            H18 = -2.0 * q7 + H16;
            H19 = -2.0 * q8 + H14;
            H29 = 1.125 * keepz(QH56) + 4.5 * (h40 - h41) - 2.25 * q12;
            H26 = 3.0 * (h40 - h41) - 0.75 * q12 + 0.375 * (H15 + H17) - H29;
            H32 = 3.0 * (h40 - 2.0 * h[35] + h41) - 1.5 * keepz(H7);
            H34 = 3.0 * (h[31] - h[32] - h[33] + h[34]) - 3.0 * keepz(H9);
            H35 = 3.0 * (h[25] - h[26] - h[29] + h[30]) - 3.0 * keepz(H10);
        }
        // Eq. 45 without sources
        V n[16];
        n[0] = e21;
        n[1] = -0.5 * sum(F24, G25, H26);
        n[2] = -(1.0 / 3.0) * sum(F27, G28, H29);
        n[3] = e24;
        n[4] = e25;
        n[5] = e26;
        n[6] = -sum(F30, 0.5 * G33, 0.5 * H35);
        n[7] = -sum(0.5 * F33, G31, 0.5 * H34);
        n[8] = -sum(0.5 * F35, 0.5 * G34, H32);
        n[9] = -sum(3.0 * keepx(F11), G14, H15);
        n[10] = -sum(F16, 3.0 * keepy(G12), H17);
        n[11] = -sum(F18, G19, 3.0 * keepz(H13));
        n[12] = -sum(2.0 * F14, 2.0 * G16, keepz(H20));
        n[13] = -sum(keepx(F20), 2.0 * G17, 2.0 * H19);
        n[14] = -sum(2.0 * F15, keepy(G20), 2.0 * H18);
        if constexpr (SRC) {        // Eq. 45, source terms
            V ts[15];
            time_source_modes(w, ts);
            n[0] += S1 + (8.0 / 70.0) * ts[2];
            n[1] += 0.5 * ts[0] - (3.0 / 7.0) * ts[2];
            n[2] += ts[1] / 3.0 + (4.0 / 7.0) * ts[2];
            n[3] += S2 - 0.3 * ts[6];
            n[4] += S3 - 0.3 * ts[7];
            n[5] += S4 - 0.3 * ts[8];
            n[6] += 0.5 * ts[3] + 0.6 * ts[6];
            n[7] += 0.5 * ts[4] + 0.6 * ts[7];
            n[8] += 0.5 * ts[5] + 0.6 * ts[8];
            n[9] += S5 + (2.0 / 3.0) * ts[9];
            n[10] += S6 + (2.0 / 3.0) * ts[10];
            n[11] += S7 + (2.0 / 3.0) * ts[11];
            n[12] += S8 + (2.0 / 3.0) * ts[12];
            n[13] += S9 + (2.0 / 3.0) * ts[13];
            n[14] += S10 + (2.0 / 3.0) * ts[14];
        }
        R change = R(0);
        if (!t.waits(done)) {
#pragma unroll
            for (int k = 0; k < 15; ++k) {
                if (conv) change = fmax(change, max_abs_diff(n[k], m[21 + k]));
                m[21 + k] = n[k];
            }
            ++ctl.iters;
        }
        if (conv) {
            change = t.zone_max(change);
            done = done || change < R(ctl.tol) * ref;
            if (!t.any(!done)) break;
        }
    }
    ctl.capped = conv && !done;
    if constexpr (SRC) {            // Eq. 53 from the source at the final iterate (times dt)
        V w[43], ts[15];
        build_w(w);
        time_source_modes(w, ts);
        *sdt = S1 + 0.5 * ts[0] + ts[1] / 3.0 + 0.25 * ts[2];
    }
}

// ------------------------------------------------------------------ nodal, App. C
// Eq. C.5 (the u35 line with node 26, the zeta node at tau = 1/3; garble G14)
template <int NV, class R>
ADER_DEV void nodal_o4_to_modes(const Vec<NV, R>* u, const Vec<NV, R>* e, Vec<NV, R>* m) {
    const Vec<NV, R>* U = u;
#define UB(n) ((n) <= 20 ? U[(n)] : e[(n) - 21])
    m[21] = 0.5 * (-5.0 * UB(1) - UB(3) - UB(4) - UB(5) - UB(6) - UB(7) - UB(8) + 12.0 * UB(21) + UB(22) + UB(23) +
                   UB(24) + UB(25) + UB(26) + UB(27) - 9.0 * UB(31) + 2.0 * UB(35));
    m[22] = 4.5 * (2.0 * UB(1) - 5.0 * UB(21) + 4.0 * UB(31) - UB(35));
    m[23] = -4.5 * (UB(1) - 3.0 * UB(21) + 3.0 * UB(31) - UB(35));
    m[24] = 3.0 * (UB(1) - 2.0 * UB(3) + UB(4) - 2.0 * UB(21) + 3.0 * UB(22) - UB(23) + UB(31) - UB(32));
    m[25] = 3.0 * (UB(1) - 2.0 * UB(5) + UB(6) - 2.0 * UB(21) + 3.0 * UB(24) - UB(25) + UB(31) - UB(33));
    m[26] = 3.0 * (UB(1) - 2.0 * UB(7) + UB(8) - 2.0 * UB(21) + 3.0 * UB(26) - UB(27) + UB(31) - UB(34));
    m[27] = -9.0 * (UB(1) - UB(3) - 2.0 * UB(21) + 2.0 * UB(22) + UB(31) - UB(32));
    m[28] = -9.0 * (UB(1) - UB(5) - 2.0 * UB(21) + 2.0 * UB(24) + UB(31) - UB(33));
    m[29] = -9.0 * (UB(1) - UB(7) - 2.0 * UB(21) + 2.0 * UB(26) + UB(31) - UB(34));
    m[30] = 6.0 * (2.0 * UB(1) - UB(3) - UB(4) - 2.0 * UB(21) + UB(22) + UB(23));
    m[31] = 6.0 * (2.0 * UB(1) - UB(5) - UB(6) - 2.0 * UB(21) + UB(24) + UB(25));
    m[32] = 6.0 * (2.0 * UB(1) - UB(7) - UB(8) - 2.0 * UB(21) + UB(26) + UB(27));
    m[33] = -12.0 * (UB(1) - UB(3) - UB(5) + UB(13) - UB(21) + UB(22) + UB(24) - UB(30));
    m[34] = -12.0 * (UB(1) - UB(5) - UB(7) + UB(9) - UB(21) + UB(24) + UB(26) - UB(28));
    m[35] = -12.0 * (UB(1) - UB(3) - UB(7) + UB(11) - UB(21) + UB(22) + UB(26) - UB(29));
#undef UB
}

// The modes 2..20 of the polynomial through the values n[1..20] at the tau = 0 nodes of Eq. C.1: Eq. C.4 solved for the
// modes, about 100 additions and 15 products, up to 209 times the largest value.  The nodes' quarter points couple w14,
// w17 and w18 in a ring.
template <class V>
ADER_DEV void nodal_o4_flux_modes(const V* n, V* m) {
    m[5] = 2.0 * (n[3] + n[4] - 2.0 * n[1]);
    m[6] = 2.0 * (n[5] + n[6] - 2.0 * n[1]);
    m[7] = 2.0 * (n[7] + n[8] - 2.0 * n[1]);
    m[15] = 4.0 * (n[10] - 2.0 * n[7] + n[11]) - 2.0 * m[5];
    m[16] = 4.0 * (n[12] - 2.0 * n[3] + n[13]) - 2.0 * m[6];
    m[19] = 4.0 * (n[14] - 2.0 * n[5] + n[9]) - 2.0 * m[7];
    const V b8 = n[13] - n[3] - n[5] + n[1], b9 = n[9] - n[5] - n[7] + n[1], b10 = n[11] - n[3] - n[7] + n[1];
    m[20] = 8.0 * (n[2] - n[11] - n[9] + n[7] - b8);
    const V k1 = 8.0 * n[8] - 4.0 * n[14] + 0.25 * m[5] + 2.0 * m[6] - 0.125 * m[15] - 2.0 * (n[15] + n[16]);
    const V k2 = 8.0 * n[4] - 4.0 * n[10] + 0.25 * m[6] + 2.0 * m[7] - 0.125 * m[16] - 2.0 * (n[17] + n[18]);
    const V k3 = 8.0 * n[6] - 4.0 * n[12] + 2.0 * m[5] + 0.25 * m[7] - 0.125 * m[19] - 2.0 * (n[19] + n[20]);
    m[14] = (512.0 / 513.0) * (k3 - 0.125 * k2 + 0.015625 * k1);
    m[17] = k1 - 0.125 * m[14];
    m[18] = k2 - 0.125 * m[17];
    m[8] = 4.0 * b8 - 0.5 * (m[14] + m[16]);
    m[9] = 4.0 * b9 - 0.5 * (m[17] + m[19]);
    m[10] = 4.0 * b10 - 0.5 * (m[15] + m[18]);
    const V h1 = 0.5 * (n[3] - n[1]) - 0.125 * m[5], h2 = 0.5 * (n[5] - n[1]) - 0.125 * m[6],
            h3 = 0.5 * (n[7] - n[1]) - 0.125 * m[7];
    const V g1 = m[16] + m[18], g2 = m[14] + m[19], g3 = m[15] + m[17];
    m[11] = (64.0 / 3.0) * (h1 + 0.0625 * (g1 + m[20]) - 0.125 * (m[8] + m[10]) - 0.5 * (n[16] - n[15]));
    m[12] = (64.0 / 3.0) * (h2 + 0.0625 * (g2 + m[20]) - 0.125 * (m[8] + m[9]) - 0.5 * (n[18] - n[17]));
    m[13] = (64.0 / 3.0) * (h3 + 0.0625 * (g3 + m[20]) - 0.125 * (m[9] + m[10]) - 0.5 * (n[20] - n[19]));
    m[2] = 4.0 * h1 + g1 / 12.0 - 0.1 * m[11];
    m[3] = 4.0 * h2 + g2 / 12.0 - 0.1 * m[12];
    m[4] = 4.0 * h3 + g3 / 12.0 - 0.1 * m[13];
}

// SRC: with a non-stiff source (s = dt S at nodes 1..20 once and at the tau > 0 nodes of the current
// iterate; the source terms of Eqs. C.2-C.3); sdt receives dt S-bar of Eq. C.6 from the final iterate.
template <class T, bool SRC = false>
ADER_DEV void predict_nodal(const T& t, typename T::V* m, PredCtl& ctl, const Src<typename T::R>* src = nullptr,
                            typename T::V* sdt = nullptr) {
    using R = typename T::R;
    using V = typename T::V;
    constexpr int NL = T::NL;
    using FR = typename FrameAt<2, NL, R>::T;       // these nodes form sums of up to 161 modes
    using VS = Vec<NL, typename FR::S>;
    // Eq. C.4: the twenty tau = 0 nodes of Eq. C.1
    V u[21];
    {
        FR fr;
        VS w[21], s[21];
#pragma unroll
        for (int k = 1; k <= 20; ++k) fr.include(m[k]);
        fr.close();
#pragma unroll
        for (int k = 1; k <= 20; ++k) w[k] = fr.enter(m[k]);
        const VS q1 = 0.25 * w[2] - 0.125 * (w[8] + w[10]) + (-21.0 * w[11] + 40.0 * w[16] + 40.0 * w[18] + 60.0 * w[20]) / 960.0;
        const VS q2 = 0.25 * w[3] - 0.125 * (w[8] + w[9]) + (-21.0 * w[12] + 40.0 * w[14] + 40.0 * w[19] + 60.0 * w[20]) / 960.0;
        const VS q3 = 0.25 * w[4] - 0.125 * (w[9] + w[10]) + (-21.0 * w[13] + 40.0 * w[15] + 40.0 * w[17] + 60.0 * w[20]) / 960.0;
        s[1] = w[1] - (w[5] + w[6] + w[7]) / 12.0;
        s[3] = s[1] + 0.5 * w[2] + 0.25 * w[5] + 0.05 * w[11] - (w[16] + w[18]) / 24.0;
        s[4] = 2.0 * s[1] - s[3] + 0.5 * w[5];
        s[5] = s[1] + 0.5 * w[3] + 0.25 * w[6] + 0.05 * w[12] - (w[14] + w[19]) / 24.0;
        s[6] = 2.0 * s[1] - s[5] + 0.5 * w[6];
        s[7] = s[1] + 0.5 * w[4] + 0.25 * w[7] + 0.05 * w[13] - (w[15] + w[17]) / 24.0;
        s[8] = 2.0 * s[1] - s[7] + 0.5 * w[7];
        s[9] = s[5] + s[7] - s[1] + 0.25 * w[9] + 0.125 * (w[17] + w[19]);
        s[11] = s[3] + s[7] - s[1] + 0.25 * w[10] + 0.125 * (w[15] + w[18]);
        s[13] = s[3] + s[5] - s[1] + 0.25 * w[8] + 0.125 * (w[14] + w[16]);
        s[10] = 2.0 * s[7] - s[11] + 0.5 * w[5] + 0.25 * w[15];
        s[12] = 2.0 * s[3] - s[13] + 0.5 * w[6] + 0.25 * w[16];
        s[14] = 2.0 * s[5] - s[9] + 0.5 * w[7] + 0.25 * w[19];
        s[2] = s[11] + s[9] - s[7] + 0.25 * w[8] + 0.125 * (w[14] + w[16] + w[20]);
        s[15] = 2.0 * s[8] - s[14] - q1 + 0.0625 * w[5] + 0.5 * w[6] - 0.03125 * (w[14] + w[15]) - 0.25 * w[17];
        s[17] = 2.0 * s[4] - s[10] - q2 + 0.0625 * w[6] + 0.5 * w[7] - 0.03125 * (w[16] + w[17]) - 0.25 * w[18];
        s[19] = 2.0 * s[6] - s[12] - q3 + 0.5 * w[5] + 0.0625 * w[7] - 0.25 * w[14] - 0.03125 * (w[18] + w[19]);
        s[16] = s[15] + 2.0 * q1;
        s[18] = s[17] + 2.0 * q2;
        s[20] = s[19] + 2.0 * q3;
#pragma unroll
        for (int k = 1; k <= 20; ++k) u[k] = fr.leave(s[k]);
    }
    // Eq. C.2 without sources: q-terms of the tau = 0 fluxes.  FP64 takes them from the fluxes' modes, in integers; the
    // sums over nodes took 879 multiply-adds a variable, an iteration's 282.  Each direction has a frame of its own: its
    // sums reach 209 times the largest flux of the frame's 256 (the three directions together 627), and fluxes of
    // different size keep their own bits.  dt / dx enters in FP64, as the directions' sums are added.
    constexpr bool INTS = !std::is_same<typename FR::S, R>::value;
    using FF = FR;
    using VF = VS;
    V qt[16];
    {
        V f[21], g[21], h[21];
        t.template fluxes<20, 0, !INTS>(u + 1, f + 1, g + 1, h + 1);
        if constexpr (INTS) {
            auto terms = [&](auto dir, const V* x, R c) {
                constexpr int DIR = decltype(dir)::value;
                FF ff;
#pragma unroll
                for (int k = 1; k <= 20; ++k) ff.include(x[k]);
                ff.close();
                VF n[21], F[21], dq[15];
#pragma unroll
                for (int k = 1; k <= 20; ++k) n[k] = ff.enter(x[k]);
                nodal_o4_flux_modes(n, F);
                nodal_o4_qterms_modes<DIR>(F, dq);
#pragma unroll
                for (int k = 0; k < 15; ++k) {
                    const V s = scale(c, ff.leave(dq[k]));
                    qt[k] = DIR == 0 ? s : qt[k] + s;
                }
            };
            terms(std::integral_constant<int, 0>{}, f, t.cx);
            terms(std::integral_constant<int, 1>{}, g, t.cy);
            terms(std::integral_constant<int, 2>{}, h, t.cz);
#pragma unroll
            for (int k = 0; k < 15; ++k) qt[k] = u[nodal_o4_base(k)] + qt[k];
        } else {
            nodal_o4_qterms(u, f, g, h, qt);
        }
    }
    V s0[21];              // with a source: s at the tau = 0 nodes, built once
    if constexpr (SRC) {
        t.template sources<20>(u + 1, *src, s0 + 1);
        nodal_o4_qterms_src(s0, qt);
    }
    auto to_modes = [&](const V* ev) {           // sums of up to 96 node values
        if constexpr (INTS) {
            FR ft;
            VS us[21], es[15], ms[36];
#pragma unroll
            for (int k = 1; k <= 20; ++k) ft.include(u[k]);
#pragma unroll
            for (int k = 0; k < 15; ++k) ft.include(ev[k]);
            ft.close();
#pragma unroll
            for (int k = 1; k <= 20; ++k) us[k] = ft.enter(u[k]);
#pragma unroll
            for (int k = 0; k < 15; ++k) es[k] = ft.enter(ev[k]);
            nodal_o4_to_modes(us, es, ms);
#pragma unroll
            for (int k = 21; k <= 35; ++k) m[k] = ft.leave(ms[k]);
        } else {
            nodal_o4_to_modes(u, ev, m);
        }
    };
    // initial guess: the evolutionary modes in m[21..35] (zero: no time evolution) at the
    // tau > 0 nodes of Eq. C.1
    V e[16];
    nodal_o4_initial(u, m, e);
    const bool conv = positive_arg(ctl.tol);
    const int cap = conv ? ctl.max_iter : ctl.n_iter;
    R ref = R(1);
    if (conv) ref = t.zone_max(max_abs(m[1])) + R(sizeof(R) == 8 ? 1e-300 : 1e-30);   // never zero in R
    ctl.iters = 0;
    bool done = false;                  // this zone has converged (others of the team may go on)
    for (int it = 0; it < cap; ++it) {
        V f[15], g[15], h[15];          // index k - 21 for nodes 21..34
        t.template fluxes<14, 0, !INTS>(e, f, g, h);
        V se[15];
        if constexpr (SRC) t.template sources<15>(e, *src, se);
        if (!t.waits(done)) {                  // Eq. C.3
            if constexpr (INTS) {
                auto terms = [&](auto dir, const V* x, R c) {
                    constexpr int DIR = decltype(dir)::value;
                    FF fi;
#pragma unroll
                    for (int k = 0; k < 14; ++k) fi.include(x[k]);
                    fi.close();
                    VF F[15], de[15];
#pragma unroll
                    for (int k = 0; k < 14; ++k) F[k] = fi.enter(x[k]);
                    nodal_o4_update_terms<DIR>(F, de);
#pragma unroll
                    for (int k = 0; k < 15; ++k) {
                        const V s = scale(c, fi.leave(de[k]));
                        e[k] = DIR == 0 ? s : e[k] + s;
                    }
                };
                terms(std::integral_constant<int, 0>{}, f, t.cx);
                terms(std::integral_constant<int, 1>{}, g, t.cy);
                terms(std::integral_constant<int, 2>{}, h, t.cz);
#pragma unroll
                for (int k = 0; k < 15; ++k) e[k] = qt[k] + e[k];
            } else {
                nodal_o4_update(qt, f, g, h, e);
            }
            if constexpr (SRC) nodal_o4_update_src(se, e);
            ++ctl.iters;
        }
        if (conv) {
            R change = R(0);
            if (!t.waits(done)) {
                V old[15];
#pragma unroll
                for (int k = 0; k < 15; ++k) old[k] = m[21 + k];
                to_modes(e);
#pragma unroll
                for (int k = 0; k < 15; ++k) change = fmax(change, max_abs_diff(old[k], m[21 + k]));
            }
            change = t.zone_max(change);
            done = done || change < R(ctl.tol) * ref;
            if (!t.any(!done)) break;
        }
    }
    ctl.capped = conv && !done;
    if (!conv) to_modes(e);
    if constexpr (SRC) {            // Eq. C.6 from the source at the final iterate (times dt)
        V se[15];
        t.template sources<15>(e, *src, se);
        *sdt = nodal_o4_sbar(s0, se);
    }
}

// ------------------------------------------------------------------ x+ face, Sec. V.3 and App. D
// p = the zone's modes in the face's x-frame (modes.cuh).  The barycentre state (Eq. 64), the face average of u
// (Eq. 65) and the facial nodes of Eq. D.11 (Eq. D.13, caret terms of spatial modes read as w, G6); ALL: also those
// that only the edge averages take.
template <bool ALL, class V>
ADER_DEV void face_states(const V* p, V& ub, V& avg, V* t) {
    const V c1 = p[1] + 0.5 * p[21] + 0.25 * p[22] + 0.125 * p[23] +
                         (4.0 * p[5] - 2.0 * p[6] - 2.0 * p[7] + 2.0 * p[30] - p[31] - p[32]) / 24.0;
    const V c2 = 0.5 * p[2] + 0.05 * p[11] + 0.25 * p[24] + 0.125 * p[27] - (p[16] + p[18]) / 24.0;
    ub = c1 + c2;
    avg = ub + (2.0 * p[6] + 2.0 * p[7] + p[16] + p[18] + 2.0 * p[22] + 3.0 * p[23] + p[27] + p[31] + p[32]) / 24.0;
    t[1] = p[1] + 0.5 * p[2] + 0.05 * p[11] + (4.0 * p[5] - 2.0 * p[6] - 2.0 * p[7] - p[16] - p[18]) / 24.0;
    t[2] = t[1] + 0.5 * p[3] + 0.25 * (p[6] + p[8]) + 0.05 * p[12] + 0.125 * p[16] + (0.25 * p[14] - 0.125 * p[19]) / 3.0;
    t[3] = 0.5 * (t[1] + t[2]) - 0.0625 * p[6] - 0.046875 * p[12] - 0.03125 * p[16];
    if (ALL) t[4] = 3.0 * t[1] + t[2] - 3.0 * t[3] - 0.09375 * p[12];
    t[5] = 6.0 * t[1] + 3.0 * t[2] - 8.0 * t[3] - 0.375 * p[12];
    t[6] = t[1] + 0.5 * p[4] + 0.25 * (p[7] + p[10]) + 0.05 * p[13] + 0.125 * p[18] + (0.25 * p[15] - 0.125 * p[17]) / 3.0;
    t[7] = 0.5 * (t[1] + t[6]) - 0.0625 * p[7] - 0.046875 * p[13] - 0.03125 * p[18];
    if (ALL) t[8] = 3.0 * t[1] + t[6] - 3.0 * t[7] - 0.09375 * p[13];
    t[9] = 6.0 * t[1] + 3.0 * t[6] - 8.0 * t[7] - 0.375 * p[13];
    t[10] = t[2] + t[6] - t[1] + 0.25 * p[9] + 0.125 * (p[17] + p[19] + p[20]);
    t[11] = t[10] + t[5] - t[2] - 0.5 * p[9] - 0.25 * (p[19] + p[20]);
    t[12] = t[10] + t[9] - t[6] - 0.5 * p[9] - 0.25 * (p[17] + p[20]);
    if (ALL) t[13] = t[11] + t[12] - t[10] + p[9] + 0.5 * p[20];
    t[14] = t[1] - (p[31] + p[32]) / 36.0 + (9.0 * p[21] + 3.0 * p[22] + p[23]) / 27.0 + p[24] / 6.0 + (p[27] + p[30]) / 18.0;
    t[15] = t[14] + t[10] - t[1] + (6.0 * p[25] + 6.0 * p[26] + 2.0 * p[28] + 2.0 * p[29] + 3.0 * p[31] + 3.0 * p[32] +
                                    3.0 * p[33] + 3.0 * p[34] + 3.0 * p[35]) / 36.0;
    t[16] = t[15] + t[11] - t[10] - (6.0 * p[25] + 2.0 * p[28] + 3.0 * p[33] + 3.0 * p[34]) / 18.0;
    t[17] = t[15] + t[12] - t[10] - (6.0 * p[26] + 2.0 * p[29] + 3.0 * p[34] + 3.0 * p[35]) / 18.0;
    t[18] = t[16] + t[17] - t[15] + p[9] + 0.5 * p[20] + p[34] / 3.0;
    t[19] = 2.0 * t[14] - t[1] + (2.0 * p[22] + 2.0 * p[23] + p[27]) / 9.0;
    if (ALL) t[20] = t[19] + t[2] - t[1] + (6.0 * p[25] + 4.0 * p[28] + 3.0 * p[31] + 3.0 * p[33]) / 18.0;
    if (ALL) t[21] = 2.0 * t[19] - t[20] + 0.5 * p[6] + 0.25 * p[16] + p[31] / 3.0;
    if (ALL) t[22] = t[19] + t[6] - t[1] + (6.0 * p[26] + 4.0 * p[29] + 3.0 * p[32] + 3.0 * p[35]) / 18.0;
    if (ALL) t[23] = 2.0 * t[19] - t[22] + 0.5 * p[7] + 0.25 * p[18] + p[32] / 3.0;
    t[24] = t[1] - 3.0 * t[14] + 3.0 * t[19] + 2.0 * p[23] / 9.0;
}

// the facial nodes the face average of the flux needs: composing Eq. D.14 with D.15, <F> = (11 F1 - 2 (F2 + F5 + F6
// + F9) - 3 F14 + 3 (F15 + F16 + F17 + F18) + 9 F19 + 3 F24) / 24.  MHD takes all 24, for the edge averages.
constexpr int FACE_NODES = 24, MEAN_NODES = 12;
ADER_DEV constexpr int mean_node(int k) {
    constexpr int n[12] = {1, 2, 5, 6, 9, 14, 15, 16, 17, 18, 19, 24};
    return n[k];
}
template <class F_>
ADER_DEV auto face_mean(const F_& F) {
    return (11.0 * F[1] - 2.0 * (F[2] + F[5] + F[6] + F[9]) - 3.0 * F[14] + 3.0 * (F[15] + F[16] + F[17] + F[18]) +
            9.0 * F[19] + 3.0 * F[24]) / 24.0;
}

// the edge averages (Eqs. D.14-D.15) of the facial flux f[n] on the edges of the transverse
// direction s (0: t1, 1: t2), upper and lower
template <class V>
ADER_DEV void edge_fluxes(const V* f, int s, V& plus, V& minus) {
    // Eq. D.14 (the modes the edge averages need)
    const V q1 = 3.0 * (f[20] - f[21]) - 1.5 * (f[15] - f[16] + f[17] - f[18]);
    const V q2 = 1.5 * (f[20] - f[21] - f[2] + f[5]);
    const V q3 = 3.0 * (f[22] - f[23]) - 1.5 * (f[15] + f[16] - f[17] - f[18]);
    const V q4 = 1.5 * (f[22] - f[23] - f[6] + f[9]);
    const V m1 = (2.0 * f[1] + f[2] + f[5] + f[6] + f[9]) / 6.0;
    const V m4 = 2.0 * (f[2] - 2.0 * f[1] + f[5]);
    const V m5 = 2.0 * (f[6] - 2.0 * f[1] + f[9]);
    const V m7 = (16.0 / 3.0) * (f[2] - 2.0 * f[3] + 2.0 * f[4] - f[5]);
    const V m8 = (16.0 / 3.0) * (f[6] - 2.0 * f[7] + 2.0 * f[8] - f[9]);
    const V m9 = 2.0 * (f[10] - 2.0 * f[6] + f[11] - f[12] + 2.0 * f[9] - f[13]);
    const V m10 = 2.0 * (f[10] - 2.0 * f[2] + f[12] - f[11] + 2.0 * f[5] - f[13]);
    const V m2 = f[2] - f[5] + m10 / 12.0 - 0.1 * m7;
    const V m3 = f[6] - f[9] + m9 / 12.0 - 0.1 * m8;
    const V m13 = 4.5 * (f[24] - f[1]) - 13.5 * (f[19] - f[14]);
    const V m12 = 2.25 * (f[24] - f[19] - f[14] + f[1] - (2.0 / 3.0) * m13);
    const V m11 = 1.5 * f[24] - 2.5 * f[14] + 0.25 * (f[15] + f[16] + f[17] + f[18]) - 0.25 * m4 -
                  0.25 * m5 - (4.0 / 3.0) * m12 - (13.0 / 9.0) * m13;
    const V m14 = 3.0 * q2 - 2.0 * q1 - 1.5 * m10;
    const V m16 = 3.0 * (q1 - q2) + 2.25 * m10;
    const V m15 = 3.0 * q4 - 2.0 * q3 - 1.5 * m9;
    const V m17 = 3.0 * (q3 - q4) + 2.25 * m9;
    const V m18 = 3.0 * (f[20] - 2.0 * f[19] + f[21]) - 1.5 * m4;
    const V m19 = 3.0 * (f[22] - 2.0 * f[19] + f[23]) - 1.5 * m5;
    // Eq. D.15
    const V af = m1 + 0.5 * m11 + m12 / 3.0 + 0.25 * m13;
    const V qa = s == 0 ? af + (2.0 * m4 + m18) / 12.0 : af + (2.0 * m5 + m19) / 12.0;
    const V qb = s == 0 ? 0.5 * m2 + 0.05 * m7 + 0.25 * m14 + m16 / 6.0
                        : 0.5 * m3 + 0.05 * m8 + 0.25 * m15 + m17 / 6.0;
    plus = qa + qb;
    minus = qa - qb;
}

// Edge-averaged states (Eq. 66) on the edges t1+, t1-, t2+, t2-.
template <class V>
ADER_DEV void edge_states(const V* p, const V& ub, const V& avg, V* e) {
    (void)ub;
    const V q1 = p[3] + 0.5 * (p[8] + p[25]) + 0.25 * p[33] + 0.1 * p[12] + (p[14] + 2.0 * p[28]) / 6.0;
    const V q2 = p[4] + 0.5 * (p[10] + p[26]) + 0.25 * p[35] + 0.1 * p[13] + (p[15] + 2.0 * p[29]) / 6.0;
    const V u1 = avg + (2.0 * p[6] + p[16] + p[31]) / 12.0 + 0.5 * q1;
    const V u2 = avg + (2.0 * p[7] + p[18] + p[32]) / 12.0 + 0.5 * q2;
    e[0] = u1;
    e[1] = u1 - q1;
    e[2] = u2;
    e[3] = u2 - q2;
}

}  // namespace o4
}  // namespace ader
