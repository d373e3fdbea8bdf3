// Instantiates the predictor + face kernel for one (order, variable count,
// precision); included by the small step_o*_*.cu translation units so that
// the build compiles them in parallel.  Expects ADER_ORDER, ADER_NV, ADER_REAL;
// with ADER_SPLIT_VARIANTS the unit holds only the dispatch and the kernel
// variants come from units that also define ADER_FORM and ADER_SRC.
#include "step_kernels.cuh"
#include "zone_o2.cuh"
#include "zone_o3.cuh"
#include "zone_o4.cuh"

namespace ader {

#define ADER_ZONEOPS(O)                                                                                             \
    template <> struct ZoneOps<O> {                                                                                 \
        template <bool SRC, class T>                                                                                \
        static ADER_DEV void predict_modal(const T& t, typename T::V* m, PredCtl& n, const Src<typename T::R>* s,   \
                                           typename T::V* sdt) {                                                    \
            o##O::predict_modal<T, SRC>(t, m, n, s, sdt);                                                           \
        }                                                                                                           \
        template <bool SRC, class T>                                                                                \
        static ADER_DEV void predict_nodal(const T& t, typename T::V* m, PredCtl& n, const Src<typename T::R>* s,   \
                                           typename T::V* sdt) {                                                    \
            o##O::predict_nodal<T, SRC>(t, m, n, s, sdt);                                                           \
        }                                                                                                           \
        static constexpr int FACE_NODES = o##O::FACE_NODES, MEAN_NODES = o##O::MEAN_NODES;                          \
        static ADER_DEV constexpr int mean_node(int k) { return o##O::mean_node(k); }                               \
        template <bool ALL, class V> static ADER_DEV void face_states(const V* p, V& ub, V& avg, V* t) {            \
            o##O::face_states<ALL>(p, ub, avg, t);                                                                  \
        }                                                                                                           \
        template <class F> static ADER_DEV auto face_mean(const F& f) { return o##O::face_mean(f); }                \
        template <class V> static ADER_DEV void edge_fluxes(const V* f, int s, V& plus, V& minus) {                 \
            o##O::edge_fluxes(f, s, plus, minus);                                                                   \
        }                                                                                                           \
        template <class V> static ADER_DEV void edge_states(const V* p, const V& ub, const V& avg, V* e) {          \
            o##O::edge_states(p, ub, avg, e);                                                                       \
        }                                                                                                           \
    };

#ifndef ADER_ZONEOPS_DEFINED
#define ADER_ZONEOPS_DEFINED
ADER_ZONEOPS(2)
ADER_ZONEOPS(3)
ADER_ZONEOPS(4)
#endif

#ifndef ADER_BOTH_FACES_DEFINED
#define ADER_BOTH_FACES_DEFINED
template <int D, class R>
ADER_DEV void both_faces_o2(const Vec<5, R>* m, R gm1, Vec<5, R>* ub, Vec<5, R>* avg, Vec<5, R>* Fa) {
    Vec<5, R> p[6];
    to_face_frame<2, D, +1>(m, p);
    o2::face<D>(p, gm1, ub[0], avg[0], Fa[0]);
    to_face_frame<2, D, -1>(m, p);
    o2::face<D>(p, gm1, ub[1], avg[1], Fa[1]);
}
template <int D, class R>
ADER_DEV void both_faces_o3(const Vec<5, R>* m, R gm1, Vec<5, R>* ub, Vec<5, R>* avg, Vec<5, R>* Fa) {
    Vec<5, R> p[16];
    to_face_frame<3, D, +1>(m, p);
    o3::face_pair<D>(p, gm1, ub, avg, Fa);
}
#endif

#ifdef ADER_ORDER
#ifdef ADER_FORM
// a translation unit of one kernel variant (ADER_FORM, ADER_SRC)
template void launch_pf_variant<ADER_ORDER, ADER_FORM, ADER_NV, ADER_REAL, ADER_SRC>(const StepArgs&, const double*,
                                                                                     cudaStream_t);
#else
#ifdef ADER_SPLIT_VARIANTS
// the variants are compiled in their own translation units (step_o*_*_<form>_<src>.cu)
extern template void launch_pf_variant<ADER_ORDER, FORM_MODAL, ADER_NV, ADER_REAL, false>(const StepArgs&,
                                                                                          const double*, cudaStream_t);
extern template void launch_pf_variant<ADER_ORDER, FORM_NODAL, ADER_NV, ADER_REAL, false>(const StepArgs&,
                                                                                          const double*, cudaStream_t);
extern template void launch_pf_variant<ADER_ORDER, FORM_MODAL, ADER_NV, ADER_REAL, true>(const StepArgs&,
                                                                                         const double*, cudaStream_t);
extern template void launch_pf_variant<ADER_ORDER, FORM_NODAL, ADER_NV, ADER_REAL, true>(const StepArgs&,
                                                                                         const double*, cudaStream_t);
#endif
template int launch_predict_faces_nv<ADER_ORDER, ADER_NV, ADER_REAL>(const StepArgs&, const double*, cudaStream_t);
#endif
#endif

}  // namespace ader
