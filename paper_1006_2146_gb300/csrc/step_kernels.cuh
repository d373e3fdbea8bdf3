// The per-zone predictor + face kernel, the flux + update kernel and, for
// MHD, the edge-EMF and constrained-transport kernels of one ADER step
// (Sec. II: reconstruction -> space-time predictor -> face fluxes -> Eqs. 6, 8).
// Instantiated per (order, variables, precision) through step_inst.cuh.
//
// S3 layout: S3[(side*NQ + q)*N + zone], side = 2*D + (S < 0), NQ =
// side_values(NV): q in [0, NV) barycentre state u_b (Eq. 54), [NV, 2NV) face
// average <u> (Eq. 55), [2NV, 3NV) face average of the physical flux <F>
// (App. D); MHD adds, for the four edges t1+, t1-, t2+, t2- of the face, the
// edge averages <u_c> and <F_c> (Eq. 57, Eqs. D.5/D.10/D.15) of the field
// component c = 5 + t the edge's EMF needs.
#pragma once
#include <type_traits>

#include "common.cuh"
#include "fixed.cuh"
#include "kernels.cuh"
#include "modes.cuh"
#include "riemann.cuh"
#include "mlp.cuh"
#include "team.cuh"

namespace ader {

template <int ORDER> struct ZoneOps;

// the spatial modes of the team's variables (every variable for a thread of its own, one for a warp of a team)
template <int ORDER, class T>
ADER_DEV void load_modes(const T& t, const StepArgs& a, const double* __restrict__ U, long long z, typename T::V* m) {
    using R = typename T::R;
    constexpr int NV = T::NV;
    const long long N = a.grid.n;
    const R* S1 = (const R*)a.S1;
    const R* S2 = (const R*)a.S2;
#pragma unroll
    for (int i = 0; i < T::NL; ++i) {
        const int v = t.var(i);
        if constexpr (sizeof(R) == 4)       // FP32 bulk: the zone means from the FP32 copy of the state
            m[1][i] = v < 5 ? (a.Uf ? a.Uf[v * N + z] : R(U[v * N + z])) : ((const R*)a.ZB)[(v - 5) * N + z];
        else
            m[1][i] = v < 5 ? R(U[v * N + z]) : ((const R*)a.ZB)[(v - 5) * N + z];
#pragma unroll
        for (int d = 0; d < 3; ++d) m[2 + d][i] = S1[((0 * 3 + d) * NV + v) * N + z];          // w2 w3 w4
        if (ORDER >= 3) {
#pragma unroll
            for (int d = 0; d < 3; ++d) m[5 + d][i] = S1[((1 * 3 + d) * NV + v) * N + z];      // w5 w6 w7
#pragma unroll
            for (int c = 0; c < 3; ++c) m[8 + c][i] = S2[(c * NV + v) * N + z];                 // w8 w9 w10
        }
        if (ORDER == 4) {
#pragma unroll
            for (int d = 0; d < 3; ++d) m[11 + d][i] = S1[((2 * 3 + d) * NV + v) * N + z];     // w11 w12 w13
#pragma unroll
            for (int c = 0; c < 7; ++c) m[14 + c][i] = S2[((3 + c) * NV + v) * N + z];          // w14..w20
        }
    }
}

// ------------------------------------------------------------------ faces in a team
// NS faces of direction D (S0 = 0 the upper first, 1 the lower) from the zone's modes s in the frame fr: face_states
// per side, every facial flux and the check of the barycentre states in one exchange, then each variable's share of
// the face data to S3.  `store` is false for the lanes past the grid's end, which only take part in the exchanges.
template <int ORDER, int D, int S0, int NS, class T>
ADER_DEV void store_sides(const T& t, const StepArgs& a, long long z, bool store, const typename T::V& mean,
                               const FrameOf<ORDER, T::NL, typename T::R>& fr,
                               const Vec<T::NL, typename FrameOf<ORDER, T::NL, typename T::R>::S>* s) {
    using R = typename T::R;
    using V = typename T::V;
    using Z = ZoneOps<ORDER>;
    constexpr int NV = T::NV, NL = T::NL, L = ModeCount<ORDER>::L, NQ = side_values(NV);
    constexpr int NN = NV == 8 ? Z::FACE_NODES : Z::MEAN_NODES;
    constexpr int T1 = D == 0 ? 1 : 0, T2 = D == 2 ? 1 : 2;
    using VS = Vec<NL, typename FrameOf<ORDER, NL, R>::S>;
    V ub[NS], avg[NS], u[NS * NN], es[NV == 8 ? 4 * NS : 1];
#pragma unroll
    for (int side = 0; side < NS; ++side) {
        VS p[L + 1], b, av, n[Z::FACE_NODES + 1];
        if (S0 + side == 0) to_face_frame<ORDER, D, +1>(s, p);
        else to_face_frame<ORDER, D, -1>(s, p);
        Z::template face_states<NV == 8>(p, b, av, n);
        ub[side] = fr.leave(b);
        avg[side] = fr.leave(av);
#pragma unroll
        for (int k = 0; k < NN; ++k) u[side * NN + k] = fr.leave(n[NV == 8 ? k + 1 : Z::mean_node(k)]);
        if constexpr (NV == 8) {
            VS e[4];
            Z::edge_states(p, b, av, e);
#pragma unroll
            for (int k = 0; k < 4; ++k) es[side * 4 + k] = fr.leave(e[k]);
        }
    }
    V f[NS * NN];
    bool ok[NS];
    t.template face_fluxes<D, NS * NN, NS>(u, ub, f, ok);
    R* S3 = (R*)a.S3;
    const long long N = a.grid.n;
#pragma unroll
    for (int side = 0; side < NS; ++side) {
        // the sums over the nodes in the state scalar too (up to 110 times a flux: 8 bits of headroom)
        using FF = typename FrameAt<2, NL, R>::T;
        FF ff;
        Vec<NL, typename FF::S> F[Z::FACE_NODES + 1];
#pragma unroll
        for (int k = 0; k < NN; ++k) ff.include(f[side * NN + k]);
        ff.close();
#pragma unroll
        for (int k = 0; k < NN; ++k) F[NV == 8 ? k + 1 : Z::mean_node(k)] = ff.enter(f[side * NN + k]);
        const V Fa = ff.leave(Z::face_mean(F));
        R* out = S3 + (long long)((2 * D + S0 + side) * NQ) * N + z;
#pragma unroll
        for (int i = 0; i < NL; ++i) {
            const int v = t.var(i);
            if (store) {
                // the zone average replaces a barycentre state that is not physical, for the wave speeds
                out[v * N] = ok[side] ? ub[side][i] : mean[i];
                out[(NV + v) * N] = avg[side][i];
                out[(2 * NV + v) * N] = Fa[i];
            }
            if constexpr (NV == 8) {
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    if (v != 5 + (e == 0 ? T1 : T2)) continue;
                    Vec<NL, typename FF::S> plus, minus;
                    Z::edge_fluxes(F, e, plus, minus);
                    if (store) {
                        out[(3 * NV + 4 * e) * N] = es[side * 4 + 2 * e][i];
                        out[(3 * NV + 4 * e + 1) * N] = ff.leave(plus)[i];
                        out[(3 * NV + 4 * e + 2) * N] = es[side * 4 + 2 * e + 1][i];
                        out[(3 * NV + 4 * e + 3) * N] = ff.leave(minus)[i];
                    }
                }
                if (store && a.solver == SOLVER_LINEARIZED) {   // the linearized edge fluxes need every component
                    R* X = S3 + (long long)6 * NQ * N + (long long)((2 * D + S0 + side) * EDGE_STATE_VALUES) * N + z;
#pragma unroll
                    for (int e = 0; e < 4; ++e) X[(e * 8 + v) * N] = es[side * 4 + e][i];
                }
            }
        }
    }
}

// both faces: in one exchange of a team, one after the other in a thread of its own (fewer live values)
template <int ORDER, int D, class T>
ADER_DEV void store_faces_team(const T& t, const StepArgs& a, long long z, bool store, const typename T::V& mean,
                               const FrameOf<ORDER, T::NL, typename T::R>& fr,
                               const Vec<T::NL, typename FrameOf<ORDER, T::NL, typename T::R>::S>* s) {
    if constexpr (T::NL == 1) {
        store_sides<ORDER, D, 0, 2>(t, a, z, store, mean, fr, s);
    } else {
        store_sides<ORDER, D, 0, 1>(t, a, z, store, mean, fr, s);
        store_sides<ORDER, D, 1, 1>(t, a, z, store, mean, fr, s);
    }
}

// the zone's modes in the state scalar of its frame (fixed.cuh)
template <int ORDER, int NV, class R>
ADER_DEV void enter_frame(const Vec<NV, R>* m, FrameOf<ORDER, NV, R>& fr,
                          Vec<NV, typename FrameOf<ORDER, NV, R>::S>* s) {
    constexpr int L = ModeCount<ORDER>::L;
#pragma unroll
    for (int k = 1; k <= L; ++k) fr.include(m[k]);
    fr.close();
#pragma unroll
    for (int k = 1; k <= L; ++k) s[k] = fr.enter(m[k]);
}

// ------------------------------------------------------------------ FP32 Euler faces, one thread per zone
// one face side: the barycentre state (replaced by the zone average for the wave speeds when it is not physical),
// <u> and <F>
template <int D, int S, int NV, class R>
ADER_DEV void write_side(const StepArgs& a, long long z, const Vec<NV, R>& mean, Vec<NV, R> ub, const Vec<NV, R>& avg,
                         const Vec<NV, R>& Fa, R gm1) {
    constexpr int NQ = side_values(NV);
    if (!physical_state(ub, gm1)) ub = mean;
    constexpr int side = 2 * D + (S < 0 ? 1 : 0);
    R* S3 = (R*)a.S3;
    const long long N = a.grid.n;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        S3[(side * NQ + v) * N + z] = ub[v];
        S3[(side * NQ + NV + v) * N + z] = avg[v];
        S3[(side * NQ + 2 * NV + v) * N + z] = Fa[v];
    }
}

template <int D, class R>
ADER_DEV void both_faces_o2(const Vec<5, R>* m, R gm1, Vec<5, R>* ub, Vec<5, R>* avg, Vec<5, R>* Fa);
template <int D, class R>
ADER_DEV void both_faces_o3(const Vec<5, R>* m, R gm1, Vec<5, R>* ub, Vec<5, R>* avg, Vec<5, R>* Fa);

// the two faces of direction D (index 0 upper, 1 lower)
template <int ORDER, int D, class R>
ADER_DEV void both_faces(const Vec<5, R>* m, R gm1, Vec<5, R>* ub, Vec<5, R>* avg, Vec<5, R>* Fa) {
    if constexpr (ORDER == 2) both_faces_o2<D, R>(m, gm1, ub, avg, Fa);
    else both_faces_o3<D, R>(m, gm1, ub, avg, Fa);
}

// the flux of direction D at node k of u, evaluated where a sum takes it
template <int D, class R>
struct FluxAt {
    const Vec<5, R>* u;
    R gm1;
    ADER_DEV Vec<5, R> operator[](int k) const { return flux<D>(u[k], gm1); }
};

template <int ORDER, int D, int S, class R>
ADER_DEV void store_face(const StepArgs& a, long long z, const Vec<5, R>* m, R gm1) {
    using Z = ZoneOps<ORDER>;
    Vec<5, R> p[ModeCount<ORDER>::L + 1], n[Z::FACE_NODES + 1], ub, avg;
    to_face_frame<ORDER, D, S>(m, p);
    Z::template face_states<false>(p, ub, avg, n);
    write_side<D, S>(a, z, m[1], ub, avg, Z::face_mean(FluxAt<D, R>{n, gm1}), gm1);
}

template <int ORDER, int D, class R>
ADER_DEV void store_faces(const StepArgs& a, long long z, const Vec<5, R>* m, R gm1) {
    if constexpr (ORDER == 4) {            // one at a time: fewer live values
        store_face<ORDER, D, +1>(a, z, m, gm1);
        store_face<ORDER, D, -1>(a, z, m, gm1);
    } else {
        Vec<5, R> ub[2], avg[2], Fa[2];
        both_faces<ORDER, D, R>(m, gm1, ub, avg, Fa);
        write_side<D, +1>(a, z, m[1], ub[0], avg[0], Fa[0], gm1);
        write_side<D, -1>(a, z, m[1], ub[1], avg[1], Fa[1], gm1);
    }
}

// Iteration statistics of the converged predictor: sum, maximum and capped zones.
ADER_DEV void record_iterations(unsigned long long* stats, const PredCtl& ctl) {
#ifdef __CUDA_ARCH__
    // one set of atomics per warp: the counters are shared by every zone of the grid
    const unsigned mask = __activemask();
    const unsigned sum = __reduce_add_sync(mask, (unsigned)ctl.iters);
    const unsigned mx = __reduce_max_sync(mask, (unsigned)ctl.iters);
    const unsigned capped = __reduce_add_sync(mask, ctl.capped ? 1u : 0u);
    if ((threadIdx.x & 31) == __ffs(mask) - 1) {
        atomicAdd(&stats[0], (unsigned long long)sum);
        atomicMax(&stats[1], (unsigned long long)mx);
        if (capped) atomicAdd(&stats[2], (unsigned long long)capped);
    }
#else
    stats[0] += ctl.iters;
    if ((unsigned long long)ctl.iters > stats[1]) stats[1] = ctl.iters;
    if (ctl.capped) stats[2] += 1;
#endif
}

// The ADER-CG predictor of zone z (Sec. II.2): the spatial modes, the learned or zero initial guess of
// the evolutionary modes, the iteration, and what the step keeps besides the face data (dt S-bar with a
// source, the whole space-time polynomial for dense output).  m[1..L] holds the space-time modes after.
// SRC: the context carries a non-stiff source; the predictor then also writes dt S-bar of Eq. 6 for the update
// (a.Sb).  `store` is false for a team's lanes past the grid's end.
template <int ORDER, int FORM, bool SRC, class T>
ADER_DEV void zone_predict(const T& t, const StepArgs& a, const double* __restrict__ U, long long z, bool store,
                           typename T::V* m, typename T::R dt) {
    using R = typename T::R;
    using V = typename T::V;
    constexpr int LS = ModeCount<ORDER>::LS, L = ModeCount<ORDER>::L, NV = T::NV, NL = T::NL;
    load_modes<ORDER>(t, a, U, z, m);
#pragma unroll
    for (int k = LS + 1; k <= L; ++k) m[k] = vzero<NL, R>();
    if (a.n_iter > 0) {      // n_iter = 0: spatial polynomial only (SSP-RK face rule)
        if constexpr (ORDER == 3) {
            if (a.G && (!a.Gact || a.Gact[z])) {          // learned initial guess of the evolutionary modes
#pragma unroll
                for (int j = 0; j < 5; ++j)
#pragma unroll
                    for (int i = 0; i < NL; ++i) m[11 + j][i] = R(a.G[(long long)(j * NV + t.var(i)) * a.grid.n + z]);
            }
        }
        PredCtl ctl{a.n_iter, a.tol, a.max_iter, 0, false};
        Src<R> src;
        V sdt;
        if constexpr (SRC) {
            src.kind = a.src_kind;
#pragma unroll
            for (int i = 0; i < 3; ++i) src.a[i] = dt * bulk_arg<R>(a.src_par[i]);
        }
        if constexpr (FORM == FORM_MODAL) ZoneOps<ORDER>::template predict_modal<SRC>(t, m, ctl, &src, &sdt);
        else ZoneOps<ORDER>::template predict_nodal<SRC>(t, m, ctl, &src, &sdt);
        if constexpr (SRC) {
            R* Sb = (R*)a.Sb;
#pragma unroll
            for (int i = 0; i < NL; ++i)
                if (store && t.var(i) < 5) Sb[t.var(i) * a.grid.n + z] = sdt[i];
        }
        if (store && t.lead()) {
            if (a.stats && positive_arg(a.tol)) record_iterations(a.stats, ctl);
            if (ctl.capped) raise_flag(a.flag, FLAG_NOT_CONVERGED);
        }
    }
    if (a.modes_out && store) {      // dense output (Sec. VII): keep the whole space-time polynomial of the step
        R* o = (R*)a.modes_out;
#pragma unroll
        for (int k = 1; k <= L; ++k)
#pragma unroll
            for (int i = 0; i < NL; ++i) o[(long long)((k - 1) * NV + t.var(i)) * a.grid.n + z] = m[k][i];
    }
}

template <class T>
ADER_DEV void team_scales(T& t, const StepArgs& a, typename T::R dt) {
    using R = typename T::R;
    t.gm1 = arg_gm1<R>(a);
    t.cx = dt * arg_idx<R>(a, 0);
    t.cy = dt * arg_idx<R>(a, 1);
    t.cz = dt * arg_idx<R>(a, 2);
}

// predictor and face data of one zone by one team
template <int ORDER, int FORM, bool SRC, class T>
ADER_DEV void team_predict_faces(T& t, const StepArgs& a, const double* __restrict__ U, long long z, bool store) {
    using R = typename T::R;
    constexpr int L = ModeCount<ORDER>::L;
    const R dt = bulk_arg<R>(a.dt_dev ? *a.dt_dev : a.dt);
    team_scales(t, a, dt);
    typename T::V m[L + 1];
    zone_predict<ORDER, FORM, SRC>(t, a, U, z, store, m, dt);
    if constexpr (T::NL == 5 && sizeof(R) == 4) {
        store_faces<ORDER, 0, R>(a, z, m, t.gm1);
        store_faces<ORDER, 1, R>(a, z, m, t.gm1);
        store_faces<ORDER, 2, R>(a, z, m, t.gm1);
    } else {
        FrameOf<ORDER, T::NL, R> fr;
        Vec<T::NL, typename FrameOf<ORDER, T::NL, R>::S> s[L + 1];
        enter_frame<ORDER>(m, fr, s);
        store_faces_team<ORDER, 0>(t, a, z, store, m[1], fr, s);
        store_faces_team<ORDER, 1>(t, a, z, store, m[1], fr, s);
        store_faces_team<ORDER, 2>(t, a, z, store, m[1], fr, s);
    }
}

// one thread per zone
template <int ORDER, int FORM, int NV, class R, bool SRC = false>
ADER_DEV void zone_predict_faces(const StepArgs& a, const double* __restrict__ U, long long z) {
    SerialTeam<NV, R> t;
    team_predict_faces<ORDER, FORM, SRC>(t, a, U, z, true);
}

// Where a team of warps computes a zone (team.cuh): FP64, order 4 and MHD, except
//   * FP32 MHD at order 2, whose forty modes fit one thread (56^3 zones: 176 us a step against the team's 199);
//   * the FP32 nodal form of order 4 (Euler): behind strong jumps its predicted density comes near zero at a node,
//     which amplifies the rounding of the fluxes by up to 10^4, and the team sums them with other roundings.
// FP32 Euler at orders 2-3 has the tiles below (third order, 128^3 zones: 0.33 ms against the team's 0.64).
template <int ORDER, int FORM, int NV, class R>
constexpr bool uses_team() {
    if (sizeof(R) == 8) return true;
    if ((ORDER == 2 && NV == 8) || (ORDER == 4 && NV == 5 && FORM == FORM_NODAL)) return false;
    return ORDER == 4 || NV == 8;
}

// FP32 bulk asks for three 128-thread blocks per SM (at most 168 registers): the extra warps hide more latency than
// what spills costs (about 12% per 256^3 step at orders 2-3); order 4 spills kilobytes per zone there and takes two
// blocks and 255 registers.
template <int ORDER, int FORM, int NV, class R, bool SRC = false>
__global__ void __launch_bounds__(128, ORDER == 4 ? 2 : 3) k_predict_faces(StepArgs a, const double* __restrict__ U) {
    const long long z = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (z < a.grid.n) zone_predict_faces<ORDER, FORM, NV, R, SRC>(a, U, z);
}

// The team kernel: a block of NV warps takes 32 zones, a warp one variable of each.
template <int ORDER, int NV, class R>
constexpr int team_smem() { return team_values<ORDER, NV>() * 32 * (int)sizeof(R); }
// Blocks an SM holds: as many as registers and shared memory allow without a kilobyte of spills (FP64 Euler: five at
// second order instead of three, 1.3% of a 96^3 step; four at third order instead of two, 3%; FP64 MHD at second order
// four, 3%; FP32 Euler at order 4 four instead of three, 3%).
template <int ORDER, int NV, class R>
constexpr int team_blocks() {
    if (NV == 5) return sizeof(R) == 4 ? 4 : ORDER == 2 ? 5 : ORDER == 3 ? 4 : 2;
    return sizeof(R) == 4 ? 2 : ORDER == 2 ? 4 : ORDER == 3 ? 2 : 1;
}

template <int ORDER, int FORM, int NV, bool SRC, class R>
__device__ __forceinline__ void team_zone(const StepArgs& a, const double* __restrict__ U, long long z, R* sh) {
    WarpTeam<NV, R> t;
    t.sh = sh + (threadIdx.x & 31);
    t.v = threadIdx.x >> 5;
    const bool store = z < a.grid.n;
    team_predict_faces<ORDER, FORM, SRC>(t, a, U, store ? z : a.grid.n - 1, store);
}

template <int ORDER, int FORM, int NV, class R, bool SRC>
__global__ void __launch_bounds__(NV * 32, team_blocks<ORDER, NV, R>())
    k_team_predict_faces(StepArgs a, const double* __restrict__ U) {
    extern __shared__ __align__(16) unsigned char team_raw[];
    team_zone<ORDER, FORM, NV, SRC, R>(a, U, (long long)blockIdx.x * 32 + (threadIdx.x & 31), (R*)team_raw);
}

template <int NV, class R>
ADER_DEV FaceSide<NV, R> load_side(const StepArgs& a, int side, long long z) {
    constexpr int NQ = side_values(NV);
    const R* S3 = (const R*)a.S3;
    const long long N = a.grid.n;
    FaceSide<NV, R> s;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        s.ub[v] = S3[(side * NQ + v) * N + z];
        s.avg[v] = S3[(side * NQ + NV + v) * N + z];
        s.F[v] = S3[(side * NQ + 2 * NV + v) * N + z];
    }
    return s;
}

// Eq. 6 for zone z: out = base + c sum_D (F(i_D - 1/2) - F(i_D + 1/2)) / dx_D,
// accumulated in FP64 for the five hydrodynamic variables.  Two ways to the
// same fluxes:
//  * fused (zone_flux_update): each zone solves the two faces of each
//    direction itself -- every face twice over the grid, in one pass.  The
//    same function with the same operands gives both zones of a face the same
//    value, so Eq. 6 telescopes exactly.  Used by FP32 Euler zones whose face
//    data lie in memory (order 4, tiles off, the batch), where the FP64
//    accumulation is the cost, not the Riemann solves.
//  * stored (zone_face_fluxes, then zone_flux_update_stored): every face is
//    solved once, by the zone below it, into the WENO scratch S1 (dead once
//    the face data exist; at least 15 values per zone at every order), and
//    the update takes differences of stored values.  Used by FP64, where the
//    solves are FP64 work on the critical path, and by MHD in both precisions,
//    whose faces also give four edge fluxes; the FP32 Euler tiles store their
//    fluxes in the same place.
template <int SOLVER, int D, int NV, class R>
ADER_DEV Vec<NV, R> upper_face_flux(const StepArgs& a, long long z, int i, int j, int k, R gamma, R gm1) {
    const long long zp = nbr_along(a.grid, z, i, j, k, D, 1);
    return riemann<SOLVER, D>(load_side<NV, R>(a, 2 * D, z), load_side<NV, R>(a, 2 * D + 1, zp), gamma, gm1);
}

template <int SOLVER, int D, int NV, class R>
ADER_DEV void flux_difference(const StepArgs& a, long long z, int i, int j, int k, R gamma, R gm1, double* acc) {
    const long long zm = nbr_along(a.grid, z, i, j, k, D, -1);
    const Vec<NV, R> Fp = upper_face_flux<SOLVER, D, NV, R>(a, z, i, j, k, gamma, gm1);
    const Vec<NV, R> Fm = riemann<SOLVER, D>(load_side<NV, R>(a, 2 * D, zm), load_side<NV, R>(a, 2 * D + 1, z),
                                             gamma, gm1);
    const double inv = a.idx[D];
#pragma unroll
    for (int v = 0; v < 5; ++v) acc[v] -= ((double)Fp[v] - (double)Fm[v]) * inv;
}

// out = base + c acc (+ dt S-bar of Eq. 6 where the predictor wrote one, a.Sb in the bulk precision R)
template <class R>
ADER_DEV void store_update(const StepArgs& a, double* out, const double* base, double c_host, int use_dt_dev,
                           const double* acc, long long z) {
    const double c = use_dt_dev ? c_host * (*a.dt_dev) : c_host;
    const long long N = a.grid.n;
    const R* Sb = (const R*)a.Sb;
    bool bad = false;
#pragma unroll
    for (int v = 0; v < 5; ++v) {
        double val = (base ? base[v * N + z] : 0.0) + c * acc[v];
        if (Sb) val += (double)Sb[v * N + z];
        bad |= !isfinite(val);
        out[v * N + z] = val;
    }
    if (bad && !a.defer_nonfinite) raise_flag(a.flag, FLAG_NONFINITE);
}

// both faces of each direction solved for one zone (the form zone_flux_update_pair carries in FP32 pairs; counted by
// flopcount)
template <int SOLVER, int NV, class R>
ADER_DEV void zone_flux_update(const StepArgs& a, double* out, const double* base, double c_host, int use_dt_dev,
                               long long z) {
    int i, j, k;
    zone_ijk(a.grid, z, i, j, k);
    const R gamma = arg_gamma<R>(a), gm1 = arg_gm1<R>(a);
    double acc[5] = {0, 0, 0, 0, 0};
    flux_difference<SOLVER, 0, NV, R>(a, z, i, j, k, gamma, gm1, acc);
    flux_difference<SOLVER, 1, NV, R>(a, z, i, j, k, gamma, gm1, acc);
    flux_difference<SOLVER, 2, NV, R>(a, z, i, j, k, gamma, gm1, acc);
    store_update<R>(a, out, base, c_host, use_dt_dev, acc, z);
}

// ------------------------------------------------------------------ FP32 bulk: Eq. 6 without FP64 arithmetic per face
// GB300 runs FP64 at 1/64 of the FP32 rate, so converting and differencing the twelve face fluxes of a
// zone in FP64 (about 70 FP64 instructions) bounded the FP32-bulk update.  Here the flux differences
// and their scaling by c_d = dt / dx_d are carried exactly in pairs of FP32 numbers (error-free
// transformations: Knuth's two-sum for Fm - Fp, the FMA two-product for s * c_d), so that the zone's
// increment sum_d c_d (Fm - Fp) reaches FP64 as hi + lo with a relative error near 2^-47, and only the
// accumulation U + hi + lo (and the source term) is FP64: 4 FP64 operations per variable.  c_d is split
// once per block into its FP32 head and tail.
ADER_DEV void two_sum(float a, float b, float& s, float& e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// true when the FP64 value is finite (exponent field not all ones), without an FP64 instruction
ADER_DEV bool finite_bits(double x) {
#ifdef __CUDA_ARCH__
    return ((__double2hiint(x) >> 20) & 0x7ff) != 0x7ff;
#else
    return isfinite(x);
#endif
}

// out = base + hi + lo (+ dt S-bar), FP64.  An addition that cannot change its FP64 sum is skipped when
// no lane of the warp needs it, so the result equals the plain sum bit for bit: hi = 0 (a zone whose
// faces all carry the same flux), and lo below half a unit in the last place of base + hi (checked on
// the exponents: |lo| < 2^(e_lo - 126) <= 2^(e_t - 1077) = ulp(t) / 2 when e_lo + 951 <= e_t).
__device__ __forceinline__ void store_pair_update(const StepArgs& a, double* out, const double* base, const float* hi,
                                                  const float* lo, long long z) {
    const long long N = a.grid.n;
    const float* Sb = (const float*)a.Sb;
    const unsigned lanes = __activemask();         // the lanes of this zone's warp still running
    bool bad = false;
    // every load before the first store (out may be base: in place)
    double b[5];
    float sb[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
        b[v] = base ? base[v * N + z] : 0.0;
        sb[v] = Sb ? Sb[v * N + z] : 0.0f;
    }
#pragma unroll
    for (int v = 0; v < 5; ++v) {
        double val = b[v];
        if (__any_sync(lanes, hi[v] != 0.0f)) val += f64_of_f32(hi[v]);
        const unsigned e_lo = (__float_as_uint(lo[v]) >> 23) & 0xffu;
        const unsigned e_t = ((unsigned)__double2hiint(val) >> 20) & 0x7ffu;
        if (__any_sync(lanes, lo[v] != 0.0f && e_lo + 951u > e_t)) val += f64_of_f32(lo[v]);
        if (Sb) val += f64_of_f32(sb[v]);
        bad |= !finite_bits(val);
        out[v * N + z] = val;
    }
    if (bad && !a.defer_nonfinite) raise_flag(a.flag, FLAG_NONFINITE);
}

template <int SOLVER, int D>
ADER_DEV void flux_difference_pair(const StepArgs& a, long long z, int i, int j, int k, float gamma, float gm1,
                                   float chi, float clo, float* hi, float* lo) {
    const long long zm = nbr_along(a.grid, z, i, j, k, D, -1);
    const Vec<5, float> Fp = upper_face_flux<SOLVER, D, 5, float>(a, z, i, j, k, gamma, gm1);
    const Vec<5, float> Fm = riemann<SOLVER, D>(load_side<5, float>(a, 2 * D, zm),
                                                load_side<5, float>(a, 2 * D + 1, z), gamma, gm1);
#pragma unroll
    for (int v = 0; v < 5; ++v) {
        float s, e;
        two_sum(Fm[v], -Fp[v], s, e);                   // Fm - Fp = s + e exactly
        const float p = s * chi;
        const float pe = fmaf(s, chi, -p);              // s chi = p + pe exactly
        const float t = pe + fmaf(s, clo, e * chi);     // the small terms of (s + e)(chi + clo)
        float h, he;
        two_sum(hi[v], p, h, he);
        hi[v] = h;
        lo[v] += he + t;
    }
}

template <int SOLVER>
__global__ void __launch_bounds__(128) k_flux_update_pair(StepArgs a, double* out, const double* base, double c_host,
                                                          int use_dt_dev) {
    __shared__ float c_hi[3], c_lo[3];
    if (threadIdx.x < 3) {
        const double c = use_dt_dev ? c_host * (*a.dt_dev) : c_host;
        const double cd = c * a.idx[threadIdx.x];
        const float h = (float)cd;
        c_hi[threadIdx.x] = h;
        c_lo[threadIdx.x] = (float)(cd - (double)h);
    }
    __syncthreads();
    const long long z = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (z >= a.grid.n) return;
    int i, j, k;
    zone_ijk(a.grid, z, i, j, k);
    const float gamma = a.gamma_f, gm1 = a.gm1_f;
    float hi[5] = {0, 0, 0, 0, 0}, lo[5] = {0, 0, 0, 0, 0};
    flux_difference_pair<SOLVER, 0>(a, z, i, j, k, gamma, gm1, c_hi[0], c_lo[0], hi, lo);
    flux_difference_pair<SOLVER, 1>(a, z, i, j, k, gamma, gm1, c_hi[1], c_lo[1], hi, lo);
    flux_difference_pair<SOLVER, 2>(a, z, i, j, k, gamma, gm1, c_hi[2], c_lo[2], hi, lo);
    store_pair_update(a, out, base, hi, lo, z);
}

// The same updates for one zone whose block may not share its problem (the batched kernels): c_d's FP32
// head and tail taken per zone, the split by integer conversions (one FP64 product and one difference
// per direction).
__device__ __forceinline__ void split_scales(const StepArgs& a, double c_host, int use_dt_dev, float* chi, float* clo) {
    const double c = use_dt_dev ? c_host * (*a.dt_dev) : c_host;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const double cd = c * a.idx[d];
        chi[d] = f32_of_f64(cd);
        clo[d] = f32_of_f64(cd - f64_of_f32(chi[d]));
    }
}

template <int SOLVER>
__device__ __forceinline__ void zone_flux_update_pair(const StepArgs& a, double* out, const double* base,
                                                      double c_host, int use_dt_dev, long long z) {
    int i, j, k;
    zone_ijk(a.grid, z, i, j, k);
    float chi[3], clo[3];
    split_scales(a, c_host, use_dt_dev, chi, clo);
    const float gamma = a.gamma_f, gm1 = a.gm1_f;
    float hi[5] = {0, 0, 0, 0, 0}, lo[5] = {0, 0, 0, 0, 0};
    flux_difference_pair<SOLVER, 0>(a, z, i, j, k, gamma, gm1, chi[0], clo[0], hi, lo);
    flux_difference_pair<SOLVER, 1>(a, z, i, j, k, gamma, gm1, chi[1], clo[1], hi, lo);
    flux_difference_pair<SOLVER, 2>(a, z, i, j, k, gamma, gm1, chi[2], clo[2], hi, lo);
    store_pair_update(a, out, base, hi, lo, z);
}

// Eq. 6 from the stored face fluxes: the differences in FP32 pairs, the accumulation in FP64
__device__ __forceinline__ void zone_flux_update_stored_pair(const StepArgs& a, double* out, const double* base,
                                                             const float* c_hi, const float* c_lo, long long z) {
    int i, j, k;
    zone_ijk(a.grid, z, i, j, k);
    const float* F = (const float*)a.S1;
    const long long N = a.grid.n;
    float hi[5] = {0, 0, 0, 0, 0}, lo[5] = {0, 0, 0, 0, 0};
#pragma unroll
    for (int D = 0; D < 3; ++D) {
        const long long zm = nbr_along(a.grid, z, i, j, k, D, -1);
        const float chi = c_hi[D], clo = c_lo[D];
#pragma unroll
        for (int v = 0; v < 5; ++v) {
            float s, e;
            two_sum(F[(D * 5 + v) * N + zm], -F[(D * 5 + v) * N + z], s, e);
            const float p = s * chi;
            const float pe = fmaf(s, chi, -p);
            const float t = pe + fmaf(s, clo, e * chi);
            float h, he;
            two_sum(hi[v], p, h, he);
            hi[v] = h;
            lo[v] += he + t;
        }
    }
    store_pair_update(a, out, base, hi, lo, z);
}

// ------------------------------------------------------------------ MHD: faces and their edge fluxes (Sec. II.3, Eq. 7)
// A face's Riemann problem is transonic when a fast wave speed changes sign between its two states.
template <class R>
ADER_DEV bool transonic(R vl, R cl, R vr, R cr) {
    return (vl - cl) * (vr - cr) < R(0) || (vl + cl) * (vr + cr) < R(0);
}

// The flux of the face of direction D between the states L and Rt with its edge values uL, FL and uR, FR (of the field
// component the edge's EMF needs): HLL with the face's own frozen wave speeds.
template <int D, class R>
ADER_DEV R edge_hll(const Vec<8, R>& ubl, const Vec<8, R>& ubr, int emf_transonic, R uL, R FL, R uR, R FR, R gamma, R gm1) {
    const Prim<8, R> pl = primitives(ubl, gm1), pr = primitives(ubr, gm1);
    const R vl = D == 0 ? pl.vx : (D == 1 ? pl.vy : pl.vz);
    const R vr = D == 0 ? pr.vx : (D == 1 ? pr.vy : pr.vz);
    const R cl = fast_speed<D>(ubl, pl, gamma), cr = fast_speed<D>(ubr, pr, gamma);
    const R lamL = fmin(fmin(vl - cl, vr - cr), R(0));
    const R lamR = fmax(fmax(vl + cl, vr + cr), R(0));
    // optional: twice the third (dissipative) term of Eq. 17 where a fast speed changes sign (Sec. V)
    const R w = (emf_transonic && transonic(vl, cl, vr, cr)) ? R(2) : R(1);
    return (lamR * FL - lamL * FR + (w * lamR) * lamL * (uR - uL)) * rcp(lamR - lamL);
}

// The same flux with the linearized solver: |A| at the mean of the face's two
// barycentre states applied to the jump dU of the full edge-averaged states.
template <int D, class R>
ADER_DEV R edge_linearized(const Vec<8, R>& ubl, const Vec<8, R>& ubr, int emf_transonic, int c, const Vec<8, R>& dU, R FL,
                           R FR, R gamma, R gm1) {
    const MeanState<R> m = mhd_mean_state(ubl, ubr, gm1);
    const Vec<8, R> diss = mhd_abs_jacobian_apply<D, R>(m.rho, m.v, m.p, m.B, gamma, gm1, dU);
    R w = R(1);
    if (emf_transonic) {           // optional doubled dissipation at transonic faces (Sec. V)
        const Prim<8, R> pl = primitives(ubl, gm1), pr = primitives(ubr, gm1);
        const R vl = D == 0 ? pl.vx : (D == 1 ? pl.vy : pl.vz);
        const R vr = D == 0 ? pr.vx : (D == 1 ? pr.vy : pr.vz);
        if (transonic(vl, fast_speed<D>(ubl, pl, gamma), vr, fast_speed<D>(ubr, pr, gamma))) w = R(2);
    }
    return R(0.5) * (FL + FR) - (R(0.5) * w) * diss[c];
}

// The upper face of zone z in direction D (zp the zone above it): its flux into F and the fluxes of its four edges
// (t1+, t1-, t2+, t2-) into q, the wave speeds or eigenvectors taken once.  A zone's EMFs used to solve each face
// again for every edge that met it, twelve solves a zone beside the update's.
template <int SOLVER, int D, class R>
ADER_DEV void mhd_face(const StepArgs& a, long long z, long long zp, R gamma, R gm1, Vec<8, R>& f, R* q) {
    constexpr int NQ = side_values(8);
    constexpr int T1 = D == 0 ? 1 : 0, T2 = D == 2 ? 1 : 2;
    const long long N = a.grid.n;
    const R* S3 = (const R*)a.S3;
    const FaceSide<8, R> L = load_side<8, R>(a, 2 * D, z), Rt = load_side<8, R>(a, 2 * D + 1, zp);
    f = riemann<SOLVER, D>(L, Rt, gamma, gm1);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const R* pl = S3 + (long long)(2 * D * NQ + 24 + 2 * e) * N + z;
        const R* pr = S3 + (long long)((2 * D + 1) * NQ + 24 + 2 * e) * N + zp;
        if constexpr (SOLVER == SOLVER_HLL) {
            q[e] = edge_hll<D>(L.ub, Rt.ub, a.emf_transonic, pl[0], pl[N], pr[0], pr[N], gamma, gm1);
        } else {
            const R* X = S3 + (long long)6 * NQ * N;
            Vec<8, R> dU;
#pragma unroll
            for (int v = 0; v < 8; ++v)
                dU[v] = X[(long long)((2 * D + 1) * EDGE_STATE_VALUES + e * 8 + v) * N + zp] -
                        X[(long long)(2 * D * EDGE_STATE_VALUES + e * 8 + v) * N + z];
            q[e] = edge_linearized<D>(L.ub, Rt.ub, a.emf_transonic, 5 + (e < 2 ? T1 : T2), dU, pl[N], pr[N], gamma, gm1);
        }
    }
}

template <int SOLVER, int NV, class R>
ADER_DEV void zone_face_fluxes(const StepArgs& a, long long z) {
    int i, j, k;
    zone_ijk(a.grid, z, i, j, k);
    const R gamma = arg_gamma<R>(a), gm1 = arg_gm1<R>(a);
    R* F = (R*)a.S1;
    const long long N = a.grid.n;
    auto face = [&](auto dir) {
        constexpr int D = decltype(dir)::value;
        if constexpr (NV == 8) {
            Vec<8, R> f;
            R q[4];
            mhd_face<SOLVER, D, R>(a, z, nbr_along(a.grid, z, i, j, k, D, 1), gamma, gm1, f, q);
            R* Q = (R*)a.S2;            // the cross moments, read by now
#pragma unroll
            for (int e = 0; e < 4; ++e) Q[(long long)(D * 4 + e) * N + z] = q[e];
#pragma unroll
            for (int v = 0; v < 5; ++v) F[(D * 5 + v) * N + z] = f[v];
        } else {
            const Vec<NV, R> f = upper_face_flux<SOLVER, D, NV, R>(a, z, i, j, k, gamma, gm1);
#pragma unroll
            for (int v = 0; v < 5; ++v) F[(D * 5 + v) * N + z] = f[v];
        }
    };
    face(std::integral_constant<int, 0>{});
    face(std::integral_constant<int, 1>{});
    face(std::integral_constant<int, 2>{});
}

template <int SOLVER, int NV, class R>
__global__ void __launch_bounds__(128) k_face_fluxes(StepArgs a) {
    const long long z = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (z < a.grid.n) zone_face_fluxes<SOLVER, NV, R>(a, z);
}

template <class R>
ADER_DEV void zone_flux_update_stored(const StepArgs& a, double* out, const double* base, double c_host,
                                      int use_dt_dev, long long z) {
    int i, j, k;
    zone_ijk(a.grid, z, i, j, k);
    const R* F = (const R*)a.S1;
    const long long N = a.grid.n;
    double acc[5] = {0, 0, 0, 0, 0};
#pragma unroll
    for (int D = 0; D < 3; ++D) {
        const long long zm = nbr_along(a.grid, z, i, j, k, D, -1);
        const double inv = a.idx[D];
#pragma unroll
        for (int v = 0; v < 5; ++v)
            acc[v] -= ((double)F[(D * 5 + v) * N + z] - (double)F[(D * 5 + v) * N + zm]) * inv;
    }
    store_update<R>(a, out, base, c_host, use_dt_dev, acc, z);
}

template <class R>
__global__ void __launch_bounds__(128) k_flux_update_stored(StepArgs a, double* out, const double* base,
                                                            double c_host, int use_dt_dev) {
    const long long z = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (z < a.grid.n) zone_flux_update_stored<R>(a, out, base, c_host, use_dt_dev, z);
}

// ------------------------------------------------------------------ FP32 Euler: predictor and face solves per tile
// A block owns a PT_X x PT_Y tile of (x, y) columns and marches through a chunk of z planes, one zone per
// thread and plane.  Each zone's predictor writes its six face sides (barycentre state, <u>, <F>; 15
// values each) to shared memory; after a barrier every face inside the tile is solved once, by the zone
// above it, with the side of the zone below it read from shared memory (x, y) or kept from the previous
// plane (z), and the flux is stored at the lower zone, as k_face_fluxes does: F[(D*5 + v)*N + zone] is the
// flux through the upper face of zone in direction D, in the WENO scratch S1 (each zone's modes were read
// before any flux lands on its slots).  Only the sides of the tile's and chunk's boundary zones go to
// S3, and k_tile_faces solves those faces afterwards.  The face data of the interior never reaches HBM,
// and no zone is predicted twice.
#ifndef ADER_PT_X
#define ADER_PT_X 32
#endif
#ifndef ADER_PT_Y
#define ADER_PT_Y 4
#endif
constexpr int PT_X = ADER_PT_X, PT_Y = ADER_PT_Y, PT_THREADS = PT_X * PT_Y;
constexpr int PT_NQ = 15;                     // values per Euler face side
constexpr int PT_SLOTS = 7;                   // x+, x-, y+, y-, z+ (even planes), z-, z+ (odd planes)

ADER_DEV float* pt_slot(float* sh, int slot, int tid) { return sh + slot * PT_NQ * PT_THREADS + tid; }

// one side into a slot: u_b (replaced by the zone mean for the wave speeds when not physical, as
// write_side does), <u>, <F>
ADER_DEV void pt_side(float* dst, const Vec<5, float>& mean, Vec<5, float> ub, const Vec<5, float>& avg, const Vec<5, float>& Fa, float gm1) {
    if (!physical_state(ub, gm1)) ub = mean;
#pragma unroll
    for (int v = 0; v < 5; ++v) {
        dst[v * PT_THREADS] = ub[v];
        dst[(5 + v) * PT_THREADS] = avg[v];
        dst[(10 + v) * PT_THREADS] = Fa[v];
    }
}

template <int ORDER, int D>
ADER_DEV void pt_sides(float* sh, int tid, int slot_plus, int slot_minus, const Vec<5, float>* m, float gm1) {
    Vec<5, float> ub[2], avg[2], Fa[2];
    both_faces<ORDER, D, float>(m, gm1, ub, avg, Fa);
    pt_side(pt_slot(sh, slot_plus, tid), m[1], ub[0], avg[0], Fa[0], gm1);
    pt_side(pt_slot(sh, slot_minus, tid), m[1], ub[1], avg[1], Fa[1], gm1);
}

ADER_DEV FaceSide<5, float> pt_load(const float* sh, int slot, int tid) {
    const float* s = sh + slot * PT_NQ * PT_THREADS + tid;
    FaceSide<5, float> f;
#pragma unroll
    for (int v = 0; v < 5; ++v) {
        f.ub[v] = s[v * PT_THREADS];
        f.avg[v] = s[(5 + v) * PT_THREADS];
        f.F[v] = s[(10 + v) * PT_THREADS];
    }
    return f;
}

// Boundary sides for k_tile_faces, packed in S3 (unused otherwise on this path) so that both their
// writes and k_tile_faces's reads are coalesced.  Three arrays, each [s][q][...] with s = 0 for the
// lower side of a boundary face (the x+, y+ or z+ side of the zone below it) and s = 1 for its upper
// side, q the 15 values of a side:
//   x: [2][15][tiles_x][nz][ny]   the tile's last column (s = 0) and first column (s = 1), j fastest
//   y: [2][15][tiles_y][nz][nx]   the tile's last row and first row, i fastest
//   z: [2][15][chunks][ny][nx]    the chunk's last plane and first plane, i fastest
// Each array has at most 30 N values (tiles_x <= nx, and so on), so the three fit in S3's 90 N.
struct PtBoundary {
    long long sx, sy, sz;          // values per (s, q) slice of each array
    long long ox, oy, oz;          // offsets of the arrays in S3
};

ADER_DEV PtBoundary pt_boundary(const Grid& g, int cz) {
    const long long ntx = (g.nx + PT_X - 1) / PT_X, nty = (g.ny + PT_Y - 1) / PT_Y, ncz = (g.nz + cz - 1) / cz;
    PtBoundary b;
    b.sx = ntx * g.nz * g.ny;
    b.sy = nty * g.nz * g.nx;
    b.sz = ncz * g.ny * g.nx;
    b.ox = 0;
    b.oy = 2 * PT_NQ * b.sx;
    b.oz = b.oy + 2 * PT_NQ * b.sy;
    return b;
}

// one side from shared memory into a packed boundary array: slice stride `slice`, position `pos`
ADER_DEV void pt_to_boundary(float* base, long long slice, long long pos, const float* sh, int slot, int tid) {
    const float* s = sh + slot * PT_NQ * PT_THREADS + tid;
#pragma unroll
    for (int q = 0; q < PT_NQ; ++q) base[q * slice + pos] = s[q * PT_THREADS];
}

ADER_DEV FaceSide<5, float> pt_from_boundary(const float* base, long long slice, long long pos) {
    FaceSide<5, float> f;
#pragma unroll
    for (int v = 0; v < 5; ++v) {
        f.ub[v] = base[v * slice + pos];
        f.avg[v] = base[(5 + v) * slice + pos];
        f.F[v] = base[(10 + v) * slice + pos];
    }
    return f;
}

template <int D>
ADER_DEV void pt_store_flux(const StepArgs& a, long long zl, const Vec<5, float>& f) {
    float* F = (float*)a.S1;
#pragma unroll
    for (int v = 0; v < 5; ++v) F[(D * 5 + v) * a.grid.n + zl] = f[v];
}

// grid: (tiles_x * tiles_y, ceil(nz / cz)); dynamic shared memory PT_SLOTS * PT_NQ * PT_THREADS floats
template <int ORDER, int FORM, int SOLVER, bool SRC>
__global__ void __launch_bounds__(PT_THREADS, 3)
    k_pf_tile(StepArgs a, const double* __restrict__ U, int cz) {

    extern __shared__ __align__(16) unsigned char pt_raw[];
    float* sh = reinterpret_cast<float*>(pt_raw);
    const Grid& g = a.grid;
    const int tid = threadIdx.x, tx = tid % PT_X, ty = tid / PT_X;
    const int tiles_x = (g.nx + PT_X - 1) / PT_X;
    const int i = (int)(blockIdx.x % tiles_x) * PT_X + tx, j = (int)(blockIdx.x / tiles_x) * PT_Y + ty;
    const int k0 = (int)blockIdx.y * cz, k1 = min(k0 + cz, g.nz);
    const bool valid = i < g.nx && j < g.ny;
    const bool last_x = tx == PT_X - 1 || i == g.nx - 1, last_y = ty == PT_Y - 1 || j == g.ny - 1;
    const float gamma = arg_gamma<float>(a), gm1 = arg_gm1<float>(a);
    const long long nxy = (long long)g.nx * g.ny;
    const float dt = bulk_arg<float>(a.dt_dev ? *a.dt_dev : a.dt);     // once per thread, for every plane
    const PtBoundary bd = pt_boundary(g, cz);
    float* S3 = (float*)a.S3;
    float* bx = S3 + bd.ox;
    float* by = S3 + bd.oy;
    float* bz = S3 + bd.oz;
    const long long tile_x = blockIdx.x % tiles_x, tile_y = blockIdx.x / tiles_x, chunk = blockIdx.y;
    for (int k = k0; k < k1; ++k) {
        const long long z = (long long)k * nxy + (long long)j * g.nx + i;
        const int zp_slot = (k & 1) ? 6 : 4;          // this plane's z+ sides; the previous plane's in the other
        if (valid) {
            Vec<5, float> m[ModeCount<ORDER>::L + 1];
            SerialTeam<5, float> team;
            team_scales(team, a, dt);
            zone_predict<ORDER, FORM, SRC>(team, a, U, z, true, m, dt);
            pt_sides<ORDER, 0>(sh, tid, 0, 1, m, gm1);
            pt_sides<ORDER, 1>(sh, tid, 2, 3, m, gm1);
            pt_sides<ORDER, 2>(sh, tid, zp_slot, 5, m, gm1);
        }
        __syncthreads();
        if (valid) {
            const long long px = (tile_x * g.nz + k) * g.ny + j, py = (tile_y * g.nz + k) * g.nx + i,
                            pz = (chunk * g.ny + j) * g.nx + i;
            if (tx > 0)                                // face i - 1/2: x+ side of the zone on the left
                pt_store_flux<0>(a, z - 1, riemann<SOLVER, 0>(pt_load(sh, 0, tid - 1), pt_load(sh, 1, tid), gamma, gm1));
            else
                pt_to_boundary(bx + PT_NQ * bd.sx, bd.sx, px, sh, 1, tid);
            if (last_x) pt_to_boundary(bx, bd.sx, px, sh, 0, tid);
            if (ty > 0)
                pt_store_flux<1>(a, z - g.nx,
                                 riemann<SOLVER, 1>(pt_load(sh, 2, tid - PT_X), pt_load(sh, 3, tid), gamma, gm1));
            else
                pt_to_boundary(by + PT_NQ * bd.sy, bd.sy, py, sh, 3, tid);
            if (last_y) pt_to_boundary(by, bd.sy, py, sh, 2, tid);
            if (k > k0)
                pt_store_flux<2>(a, z - nxy,
                                 riemann<SOLVER, 2>(pt_load(sh, 10 - zp_slot, tid), pt_load(sh, 5, tid), gamma, gm1));
            else
                pt_to_boundary(bz + PT_NQ * bd.sz, bd.sz, pz, sh, 5, tid);
            if (k == k1 - 1) pt_to_boundary(bz, bd.sz, pz, sh, zp_slot, tid);
        }
        __syncthreads();
    }
}

// The faces on tile and chunk boundaries, from the sides k_pf_tile packed in S3: the tile boundaries in
// x (i = multiples of PT_X, and i = 0 against nx - 1), in y (multiples of PT_Y) and the chunk boundaries
// in z (multiples of cz).  One thread per face, the packed arrays' fastest index fastest across threads.
template <int SOLVER>
__global__ void __launch_bounds__(128) k_tile_faces(StepArgs a, int cz, long long nfx, long long nfy, long long nfz) {
    const Grid& g = a.grid;
    long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const float gamma = arg_gamma<float>(a), gm1 = arg_gm1<float>(a);
    const long long nxy = (long long)g.nx * g.ny;
    const PtBoundary bd = pt_boundary(g, cz);
    const float* S3 = (const float*)a.S3;
    if (t < nfx) {                      // x: t = (tile * nz + k) * ny + j; lower zone in the previous tile
        const int j = (int)(t % g.ny);
        const long long r = t / g.ny;
        const int k = (int)(r % g.nz), tile = (int)(r / g.nz);
        const int ntx = (g.nx + PT_X - 1) / PT_X;
        const int tl = tile == 0 ? ntx - 1 : tile - 1;
        const int il = tile == 0 ? g.nx - 1 : tile * PT_X - 1;
        const long long pl = ((long long)tl * g.nz + k) * g.ny + j;
        const float* bx = S3 + bd.ox;
        pt_store_flux<0>(a, (long long)k * nxy + (long long)j * g.nx + il,
                         riemann<SOLVER, 0>(pt_from_boundary(bx, bd.sx, pl),
                                            pt_from_boundary(bx + PT_NQ * bd.sx, bd.sx, t), gamma, gm1));
        return;
    }
    t -= nfx;
    if (t < nfy) {                      // y: t = (tile * nz + k) * nx + i
        const int i = (int)(t % g.nx);
        const long long r = t / g.nx;
        const int k = (int)(r % g.nz), tile = (int)(r / g.nz);
        const int nty = (g.ny + PT_Y - 1) / PT_Y;
        const int tl = tile == 0 ? nty - 1 : tile - 1;
        const int jl = tile == 0 ? g.ny - 1 : tile * PT_Y - 1;
        const long long pl = ((long long)tl * g.nz + k) * g.nx + i;
        const float* by = S3 + bd.oy;
        pt_store_flux<1>(a, (long long)k * nxy + (long long)jl * g.nx + i,
                         riemann<SOLVER, 1>(pt_from_boundary(by, bd.sy, pl),
                                            pt_from_boundary(by + PT_NQ * bd.sy, bd.sy, t), gamma, gm1));
        return;
    }
    t -= nfy;
    if (t < nfz) {                      // z: t = chunk * nxy + column
        const long long col = t % nxy;
        const int chunk = (int)(t / nxy);
        const int ncz = (g.nz + cz - 1) / cz;
        const int cl = chunk == 0 ? ncz - 1 : chunk - 1;
        const int kl = chunk == 0 ? g.nz - 1 : chunk * cz - 1;
        const float* bz = S3 + bd.oz;
        pt_store_flux<2>(a, (long long)kl * nxy + col,
                         riemann<SOLVER, 2>(pt_from_boundary(bz, bd.sz, (long long)cl * nxy + col),
                                            pt_from_boundary(bz + PT_NQ * bd.sz, bd.sz, t), gamma, gm1));
    }
}

// z planes per chunk: enough blocks for every SM to hold several, at most 16 planes
inline int pt_chunk(const Grid& g) {
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long long tiles = (long long)((g.nx + PT_X - 1) / PT_X) * ((g.ny + PT_Y - 1) / PT_Y);
    long long cz = tiles * g.nz / ((long long)sms * 12);
    if (cz < 1) cz = 1;
    if (cz > 16) cz = 16;
    return (int)cz;
}

template <int ORDER, int FORM, bool SRC>
void launch_pf_tile(const StepArgs& a, const double* U, cudaStream_t st) {
    const Grid& g = a.grid;
    const int cz = pt_chunk(g);
    const int ntx = (g.nx + PT_X - 1) / PT_X, nty = (g.ny + PT_Y - 1) / PT_Y, ncz = (g.nz + cz - 1) / cz;
    const size_t smem = (size_t)PT_SLOTS * PT_NQ * PT_THREADS * sizeof(float);
    const dim3 grid((unsigned)(ntx * nty), (unsigned)ncz);
    const long long nfx = (long long)ntx * g.ny * g.nz, nfy = (long long)nty * g.nx * g.nz,
                    nfz = (long long)ncz * g.nx * g.ny;
    const long long nf = nfx + nfy + nfz;
    const unsigned fblocks = (unsigned)((nf + 127) / 128);
    if (a.solver == SOLVER_HLL) {
        auto kern = k_pf_tile<ORDER, FORM, SOLVER_HLL, SRC>;
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        kern<<<grid, PT_THREADS, smem, st>>>(a, U, cz);
        k_tile_faces<SOLVER_HLL><<<fblocks, 128, 0, st>>>(a, cz, nfx, nfy, nfz);
    } else {
        auto kern = k_pf_tile<ORDER, FORM, SOLVER_LINEARIZED, SRC>;
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        kern<<<grid, PT_THREADS, smem, st>>>(a, U, cz);
        k_tile_faces<SOLVER_LINEARIZED><<<fblocks, 128, 0, st>>>(a, cz, nfx, nfy, nfz);
    }
}

// FP32 bulk, Eq. 6 from the stored face fluxes (the tiles' or MHD's)
template <class R>
__global__ void __launch_bounds__(128) k_flux_update_stored_pair(StepArgs a, double* out, const double* base,
                                                                 double c_host, int use_dt_dev) {
    static_assert(sizeof(R) == 4, "FP32 bulk only");
    __shared__ float c_hi[3], c_lo[3];
    if (threadIdx.x < 3) {
        const double c = use_dt_dev ? c_host * (*a.dt_dev) : c_host;
        const double cd = c * a.idx[threadIdx.x];
        const float h = (float)cd;
        c_hi[threadIdx.x] = h;
        c_lo[threadIdx.x] = (float)(cd - (double)h);
    }
    __syncthreads();
    const long long z = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (z < a.grid.n) zone_flux_update_stored_pair(a, out, base, c_hi, c_lo, z);
}

// ------------------------------------------------------------------ MHD: edge EMFs (Sec. II.3, Eq. 7)
// EMFs at the three upper edges of zone (i, j, k): Ez on (i+1/2, j+1/2),
// Ey on (i+1/2, k+1/2), Ex on (j+1/2, k+1/2); each the mean of the four
// adjacent faces' edge fluxes with Eq. 7's signs (Ez = -F7 = G6,
// Ey = F8 = -H6, Ex = -G8 = H7).
template <class R>
ADER_DEV void zone_emf(const StepArgs& a, long long z) {
    const Grid& g = a.grid;
    int i, j, k;
    zone_ijk(g, z, i, j, k);
    const long long zx = nbr(g, i, j, k, 1, 0, 0), zy = nbr(g, i, j, k, 0, 1, 0), zz = nbr(g, i, j, k, 0, 0, 1);
    // the edge fluxes of zone_face_fluxes, stored at the zone below the face.  x-faces: t1 = y (slots 0, 1), t2 = z
    // (2, 3); y-faces: t1 = x, t2 = z; z-faces: t1 = x, t2 = y
    const R* Q = (const R*)a.S2;
    auto q = [&](int d, int e, long long at) { return Q[(long long)(d * 4 + e) * g.n + at]; };
    const R Ez = R(0.25) * (-q(0, 0, z) - q(0, 1, zy) + q(1, 0, z) + q(1, 1, zx));
    const R Ey = R(0.25) * (q(0, 2, z) + q(0, 3, zz) - q(2, 0, z) - q(2, 1, zx));
    const R Ex = R(0.25) * (-q(1, 2, z) - q(1, 3, zz) + q(2, 2, z) + q(2, 3, zy));
    R* E = (R*)a.E;
    E[z] = Ex;
    E[g.n + z] = Ey;
    E[2 * g.n + z] = Ez;
}

template <class R>
__global__ void __launch_bounds__(128) k_emf(StepArgs a) {
    const long long z = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (z < a.grid.n) zone_emf<R>(a, z);
}

// Eq. 8 on the three faces i-1/2, j-1/2, k-1/2 of zone (i, j, k): each face
// is written by exactly one zone, so the update is in place.
template <class R>
ADER_DEV void zone_ct(const StepArgs& a, double* Bf, double c_host, int use_dt_dev, long long z) {
    const Grid& g = a.grid;
    int i, j, k;
    zone_ijk(g, z, i, j, k);
    const R* E = (const R*)a.E;
    const long long N = g.n;
    // FP32 edge fields widen to FP64 exactly on the integer pipe (f64_of_f32), not by conversions on the
    // FP64 units
    auto wide = [](R e) -> double {
        if constexpr (sizeof(R) == 4) return f64_of_f32(e); else return e;
    };
    auto Ex = [&](int di, int dj, int dk) { return wide(E[nbr(g, i, j, k, di, dj, dk)]); };
    auto Ey = [&](int di, int dj, int dk) { return wide(E[N + nbr(g, i, j, k, di, dj, dk)]); };
    auto Ez = [&](int di, int dj, int dk) { return wide(E[2 * N + nbr(g, i, j, k, di, dj, dk)]); };
    const double dt = use_dt_dev ? c_host * (*a.dt_dev) : c_host;
    const double idx = a.idx[0], idy = a.idx[1], idz = a.idx[2];
    // the edges of face i-1/2 are stored one zone lower in x (likewise for y, z)
    Bf[z] -= dt * ((Ez(-1, 0, 0) - Ez(-1, -1, 0)) * idy - (Ey(-1, 0, 0) - Ey(-1, 0, -1)) * idz);
    Bf[N + z] -= dt * ((Ex(0, -1, 0) - Ex(0, -1, -1)) * idz - (Ez(0, -1, 0) - Ez(-1, -1, 0)) * idx);
    Bf[2 * N + z] -= dt * ((Ey(0, 0, -1) - Ey(-1, 0, -1)) * idx - (Ex(0, 0, -1) - Ex(0, -1, -1)) * idy);
}

template <class R>
__global__ void __launch_bounds__(128) k_ct(StepArgs a, double* Bf, double c_host, int use_dt_dev) {
    const long long z = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (z < a.grid.n) zone_ct<R>(a, Bf, c_host, use_dt_dev, z);
}

// where a context with tiles on takes the tile kernel
template <int ORDER, int NV, class R>
constexpr bool uses_tiles() { return NV == 5 && ORDER <= 3 && sizeof(R) == 4; }

// One variant of the predictor + face kernel, launched over the grid.  Each variant can be compiled in a
// translation unit of its own (the fourth-order ones are, see step_inst.cuh), which keeps the parallel
// build's longest compile short.
template <int ORDER, int FORM, int NV, class R, bool SRC>
void launch_pf_variant(const StepArgs& a, const double* U, cudaStream_t st) {
    if constexpr (uses_tiles<ORDER, NV, R>()) {
        if (a.tiled) {
            launch_pf_tile<ORDER, FORM, SRC>(a, U, st);
            return;
        }
    }
    if constexpr (uses_team<ORDER, FORM, NV, R>()) {
        auto kern = k_team_predict_faces<ORDER, FORM, NV, R, SRC>;
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, team_smem<ORDER, NV, R>());
        kern<<<(unsigned)((a.grid.n + 31) / 32), NV * 32, team_smem<ORDER, NV, R>(), st>>>(a, U);
    } else {
        const int T = 128;
        const unsigned blocks = (unsigned)((a.grid.n + T - 1) / T);
        k_predict_faces<ORDER, FORM, NV, R, SRC><<<blocks, T, 0, st>>>(a, U);
    }
}

template <int ORDER, int NV, class R>
int launch_predict_faces_nv(const StepArgs& a, const double* U, cudaStream_t st) {
    if (a.src_kind != SOURCE_NONE && a.Sb && a.n_iter > 0) {
        if (a.form == FORM_NODAL)
            launch_pf_variant<ORDER, FORM_NODAL, NV, R, true>(a, U, st);
        else
            launch_pf_variant<ORDER, FORM_MODAL, NV, R, true>(a, U, st);
        return uses_tiles<ORDER, NV, R>() && a.tiled ? 2 : 1;
    }
    if (a.form == FORM_MODAL)
        launch_pf_variant<ORDER, FORM_MODAL, NV, R, false>(a, U, st);
    else
        launch_pf_variant<ORDER, FORM_NODAL, NV, R, false>(a, U, st);
    return uses_tiles<ORDER, NV, R>() && a.tiled ? 2 : 1;
}

}  // namespace ader
