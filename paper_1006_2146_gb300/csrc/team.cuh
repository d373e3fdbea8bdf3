// Who computes a zone.  The predictor and the faces alternate two kinds of work: linear combinations of modes and
// node values, the same for every variable, and fluxes at nodes, which need all variables of one node.  The zone
// code is written once on a team of threads:
//   SerialTeam   one thread holds all variables of a zone (NL = NV);
//   WarpTeam     a block of NV warps holds 32 zones, warp v the variable v of each (NL = 1).  A variable's modes,
//                node values and flux modes then fit the registers at every order; for the fluxes the warps put
//                their node values into shared memory, take the nodes in turn, and read their variable's fluxes
//                back.
// One thread per zone spilled 5 KB a zone to local memory in FP64 at order 4 (1.6 KB in FP32, 7-14 KB of traffic for
// MHD), which the L1 of an SM cannot hold for 256 threads; the team spills next to nothing.  At orders 2 and 3 FP64
// had eight warps per SM beside a tile's face data; the team has 20 to 25, and the third-order predictor and faces of
// 256^3 zones went from 75 ms (with the states in integers) to 42.
#pragma once
#include "common.cuh"
#include "fixed.cuh"

namespace ader {

template <int NV, class R>
ADER_DEV bool physical_state(const Vec<NV, R>& u, R gm1) {
    const Prim<NV, R> q = primitives(u, gm1);
    return u[0] > R(0) && q.p > R(0);
}

// a - b, both rounded before: a subtraction that is contracted with the product behind b would leave that product's
// rounding error where a equals b
template <class R> ADER_DEV R apart(R a, R b) { return a - b; }
template <> ADER_DEV float apart<float>(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fsub_rn(a, b);
#else
    return a - b;
#endif
}
template <> ADER_DEV double apart<double>(double a, double b) {
#ifdef __CUDA_ARCH__
    return __dsub_rn(a, b);
#else
    return a - b;
#endif
}
template <int NV, class R>
ADER_DEV Vec<NV, R> apart(const Vec<NV, R>& a, const Vec<NV, R>& b) {
    Vec<NV, R> r;
#pragma unroll
    for (int i = 0; i < NV; ++i) r[i] = apart(a[i], b[i]);
    return r;
}

// MHD: a copy of u that shares no product with another use of it.  The flux adds and subtracts pairs of products, and
// which of a pair is contracted into a multiply-add depends on what else uses them.
template <int NV, class R>
ADER_DEV Vec<NV, R> alone(Vec<NV, R> u) {
#ifdef __CUDA_ARCH__
    if constexpr (NV == 8) {
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            if constexpr (sizeof(R) == 4) asm volatile("" : "+f"(u[i]));
            else asm volatile("" : "+d"(u[i]));
        }
    }
#endif
    return u;
}

template <int NV_, class R_>
struct SerialTeam {
    static constexpr int NV = NV_, NL = NV_;
    using R = R_;
    using V = Vec<NL, R>;
    R gm1, cx, cy, cz;

    ADER_DEV int var(int i) const { return i; }
    ADER_DEV bool lead() const { return true; }
    ADER_DEV R zone_max(R x) const { return x; }
    ADER_DEV bool any(bool x) const { return x; }
    // a converged zone that waits for others of its team (a thread of its own leaves the iteration instead)
    static ADER_DEV bool waits(bool) { return false; }
    // fluxes of N nodes in every direction, then of A nodes in x, A in y and A in z; SC: times cx, cy, cz
    template <int N, int A, bool SC>
    ADER_DEV void fluxes(const V* u, V* f, V* g, V* h) const {
        const R kx = SC ? cx : R(1), ky = SC ? cy : R(1), kz = SC ? cz : R(1);
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const Prim<NV, R> q = primitives(u[k], gm1);
            if constexpr (sizeof(R) == 4) {     // (the three-way form costs 4% of a nodal fourth-order step here)
                f[k] = SC ? scale(kx, flux_from<0>(u[k], q)) : flux_from<0>(u[k], q);
                g[k] = SC ? scale(ky, flux_from<1>(u[k], q)) : flux_from<1>(u[k], q);
                h[k] = SC ? scale(kz, flux_from<2>(u[k], q)) : flux_from<2>(u[k], q);
            } else {
                V fx, fy, fz;
                fluxes_from(u[k], q, fx, fy, fz);
                f[k] = SC ? scale(kx, fx) : fx;
                g[k] = SC ? scale(ky, fy) : fy;
                h[k] = SC ? scale(kz, fz) : fz;
            }
        }
#pragma unroll
        for (int k = 0; k < A; ++k) f[N + k] = SC ? flux_scaled<0>(u[N + k], gm1, kx) : flux<0>(u[N + k], gm1);
#pragma unroll
        for (int k = 0; k < A; ++k) g[N + k] = SC ? flux_scaled<1>(u[N + A + k], gm1, ky) : flux<1>(u[N + A + k], gm1);
#pragma unroll
        for (int k = 0; k < A; ++k)
            h[N + k] = SC ? flux_scaled<2>(u[N + 2 * A + k], gm1, kz) : flux<2>(u[N + 2 * A + k], gm1);
    }
    // sum over d of c_d (F_d(u[0]) - F_d(u[1 + d])), times k.  Direction by direction, with the same flux on both sides
    // and a subtraction of rounded values (apart): equal states give exactly zero.  (One flux along (cx, cy, cz) for u[0]
    // rounds unlike the three it meets.)
    ADER_DEV V axis_differences(const V* u, R k) const {
        return scale(k * cx, apart(flux<0>(alone(u[0]), gm1), flux<0>(u[1], gm1))) +
               scale(k * cy, apart(flux<1>(alone(u[0]), gm1), flux<1>(u[2], gm1))) +
               scale(k * cz, apart(flux<2>(alone(u[0]), gm1), flux<2>(u[3], gm1)));
    }
    // fluxes of direction D at N nodes; ok[s]: whether the M states ub[s] are physical
    template <int D, int N, int M>
    ADER_DEV void face_fluxes(const V* u, const V* ub, V* f, bool* ok) const {
#pragma unroll
        for (int k = 0; k < N; ++k) f[k] = flux<D>(u[k], gm1);
#pragma unroll
        for (int s = 0; s < M; ++s) ok[s] = physical_state(ub[s], gm1);
    }
    template <int N>
    ADER_DEV void sources(const V* u, const Src<R>& src, V* s) const {
#pragma unroll
        for (int k = 0; k < N; ++k) s[k] = source_at(u[k], src);
    }
};

#ifdef __CUDACC__
template <int NV_, class R_>
struct WarpTeam {
    static constexpr int NV = NV_, NL = 1;
    using R = R_;
    using V = Vec<1, R>;
    R gm1, cx, cy, cz;
    R* sh;               // this lane's column of the exchange buffer: value j at sh[j * 32]
    int v;               // the warp's variable

    __device__ __forceinline__ int var(int) const { return v; }
    __device__ __forceinline__ bool lead() const { return v == 0; }
    __device__ __forceinline__ Vec<NV, R> load(int at) const {
        Vec<NV, R> u;
#pragma unroll
        for (int c = 0; c < NV; ++c) u[c] = sh[(at + c) * 32];
        return u;
    }
    __device__ __forceinline__ void store(int at, const Vec<NV, R>& u) const {
#pragma unroll
        for (int c = 0; c < NV; ++c) sh[(at + c) * 32] = u[c];
    }
    __device__ __forceinline__ R zone_max(R x) const {
        __syncthreads();
        sh[v * 32] = x;
        __syncthreads();
        R m = sh[0];
#pragma unroll
        for (int c = 1; c < NV; ++c) m = fmax(m, sh[c * 32]);
        return m;
    }
    __device__ __forceinline__ bool any(bool x) const { return __syncthreads_or(x) != 0; }
    static __device__ __forceinline__ bool waits(bool done) { return done; }

    // A node's slot holds its NV values; the warp that evaluates the node replaces them with its fluxes.
    template <int N, int A, bool SC>
    __device__ __forceinline__ void fluxes(const V* u, V* f, V* g, V* h) const {
        constexpr int AX = N * 3 * NV;
        __syncthreads();                    // the last exchange has been read
#pragma unroll
        for (int k = 0; k < N; ++k) sh[(k * 3 * NV + v) * 32] = u[k][0];
#pragma unroll
        for (int k = 0; k < 3 * A; ++k) sh[(AX + k * NV + v) * 32] = u[N + k][0];
        __syncthreads();
#pragma unroll 1
        for (int k = v; k < N + 3 * A; k += NV) {
            if (k < N) {
                const int at = k * 3 * NV;
                const Vec<NV, R> x = load(at);
                const Prim<NV, R> q = primitives(x, gm1);
                Vec<NV, R> fx, fy, fz;
                fluxes_from(x, q, fx, fy, fz);
                store(at, SC ? scale(cx, fx) : fx);
                store(at + NV, SC ? scale(cy, fy) : fy);
                store(at + 2 * NV, SC ? scale(cz, fz) : fz);
            } else if (A > 0) {
                const int at = AX + (k - N) * NV, d = (k - N) / (A > 0 ? A : 1);
                const Vec<NV, R> x = load(at);
                if (d == 0) store(at, SC ? flux_scaled<0>(x, gm1, cx) : flux<0>(x, gm1));
                else if (d == 1) store(at, SC ? flux_scaled<1>(x, gm1, cy) : flux<1>(x, gm1));
                else store(at, SC ? flux_scaled<2>(x, gm1, cz) : flux<2>(x, gm1));
            }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < N; ++k) {
            f[k][0] = sh[(k * 3 * NV + v) * 32];
            g[k][0] = sh[(k * 3 * NV + NV + v) * 32];
            h[k][0] = sh[(k * 3 * NV + 2 * NV + v) * 32];
        }
#pragma unroll
        for (int k = 0; k < A; ++k) {
            f[N + k][0] = sh[(AX + k * NV + v) * 32];
            g[N + k][0] = sh[(AX + (A + k) * NV + v) * 32];
            h[N + k][0] = sh[(AX + (2 * A + k) * NV + v) * 32];
        }
    }
    __device__ __forceinline__ V axis_differences(const V* u, R k) const {
        __syncthreads();
#pragma unroll
        for (int n = 0; n < 4; ++n) sh[(n * NV + v) * 32] = u[n][0];
        __syncthreads();
        // direction d at node 0, into the slot 4 + d, and at node 1 + d, in place
        if constexpr (NV == 5) {
            // node 0's three fluxes in one warp, for their common pressure (409 us a 56^3 step at second order, FP64,
            // against 414 with a warp for each; a sum of Euler's flux has one product, so that it rounds as it does alone)
            if (v < 4) {
                const Vec<NV, R> x = load(v * NV);
                if (v == 0) {
                    store(4 * NV, flux<0>(x, gm1));
                    store(5 * NV, flux<1>(x, gm1));
                    store(6 * NV, flux<2>(x, gm1));
                } else if (v == 1) store(NV, flux<0>(x, gm1));
                else if (v == 2) store(2 * NV, flux<1>(x, gm1));
                else store(3 * NV, flux<2>(x, gm1));
            }
        } else if (v < 6) {
            // MHD: the same instructions for both, so that equal states give equal fluxes (see alone)
            const int d = v < 3 ? v : v - 3, at = v < 3 ? 0 : (1 + d) * NV, to = v < 3 ? (4 + d) * NV : at;
            const Vec<NV, R> x = load(at);
            if (d == 0) store(to, flux<0>(x, gm1));
            else if (d == 1) store(to, flux<1>(x, gm1));
            else store(to, flux<2>(x, gm1));
        }
        __syncthreads();
        V r;
        r[0] = k * cx * (sh[(4 * NV + v) * 32] - sh[(NV + v) * 32]) + k * cy * (sh[(5 * NV + v) * 32] - sh[(2 * NV + v) * 32]) +
               k * cz * (sh[(6 * NV + v) * 32] - sh[(3 * NV + v) * 32]);
        return r;
    }
    template <int D, int N, int M>
    __device__ __forceinline__ void face_fluxes(const V* u, const V* ub, V* f, bool* ok) const {
        __syncthreads();
#pragma unroll
        for (int k = 0; k < N; ++k) sh[(k * NV + v) * 32] = u[k][0];
#pragma unroll
        for (int s = 0; s < M; ++s) sh[((N + s) * NV + v) * 32] = ub[s][0];
        __syncthreads();
#pragma unroll 1
        for (int k = v; k < N + M; k += NV) {
            const Vec<NV, R> x = load(k * NV);
            if (k < N) store(k * NV, flux<D>(x, gm1));
            else sh[k * NV * 32] = physical_state(x, gm1) ? R(1) : R(0);
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < N; ++k) f[k][0] = sh[(k * NV + v) * 32];
#pragma unroll
        for (int s = 0; s < M; ++s) ok[s] = sh[(N + s) * NV * 32] > R(0);
    }
    template <int N>
    __device__ __forceinline__ void sources(const V* u, const Src<R>& src, V* s) const {
        __syncthreads();
#pragma unroll
        for (int k = 0; k < N; ++k) sh[(k * NV + v) * 32] = u[k][0];
        __syncthreads();
#pragma unroll 1
        for (int k = v; k < N; k += NV) store(k * NV, source_at(load(k * NV), src));
        __syncthreads();
#pragma unroll
        for (int k = 0; k < N; ++k) s[k][0] = sh[(k * NV + v) * 32];
    }
};
#endif

// values a lane's column of the exchange buffer holds: the largest exchange of the order
template <int ORDER, int NV>
constexpr int team_values() {
    // nodes: 6 axis nodes at order 2, 13 in three directions at order 3, 21 at order 4; faces: two sides' nodes and
    // their two barycentre states
    const int nodes = (ORDER == 4 ? 63 : (ORDER == 3 ? 39 : 6)) * NV;
    const int faces = (2 * (ORDER == 4 ? (NV == 8 ? 24 : 12) : (ORDER == 3 ? 10 : 5)) + 2) * NV;
    return nodes > faces ? nodes : faces;
}

}  // namespace ader
