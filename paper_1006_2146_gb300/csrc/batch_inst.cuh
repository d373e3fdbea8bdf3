// Instantiates the batched phases for one (order, variable count) in FP32
// bulk; included by the small batch_o*_*.cu translation units.  Expects
// ADER_BORDER and ADER_BNV.
#include "batch.cuh"
#include "step_inst.cuh"

namespace ader {

template <int ORDER, int NV>
int batch_phase(int ph, const BatchGroupDev& g, int form, int solver, int threads, int blocks, cudaStream_t st,
                bool launch, const void** fn) {
    using R = float;
    const void* k = nullptr;
    size_t smem = 0;
    bool team = false;
    switch (ph) {
        case PH_TO_F32: k = (const void*)kb_to_f32; break;
        case PH_FACE_B:
            if constexpr (NV == 8) k = (const void*)kb_face_b<ORDER, R>;
            break;
        case PH_WENO1D: k = (const void*)kb_weno1d<ORDER, NV, R>; break;
        case PH_CROSS1:
            if constexpr (ORDER >= 3) k = (const void*)kb_cross1<ORDER, NV, R>;
            break;
        case PH_CROSS2:
            if constexpr (ORDER == 4) k = (const void*)kb_cross2<NV, R>;
            break;
        case PH_PREDICT:
            if (form == FORM_NODAL) {
                if constexpr (uses_team<ORDER, FORM_NODAL, NV, R>()) {
                    k = (const void*)kb_team_predict_faces<ORDER, FORM_NODAL, NV, R>;
                    team = true;
                } else {
                    k = (const void*)kb_predict_faces<ORDER, FORM_NODAL, NV, R>;
                }
            } else if constexpr (uses_team<ORDER, FORM_MODAL, NV, R>()) {
                k = (const void*)kb_team_predict_faces<ORDER, FORM_MODAL, NV, R>;
                team = true;
            } else {
                k = (const void*)kb_predict_faces<ORDER, FORM_MODAL, NV, R>;
            }
            if (team) {                                 // 32 zones per block, whatever `threads` says
                threads = NV * 32;
                blocks = (int)((g.total + 31) / 32);
                smem = team_smem<ORDER, NV, R>();
                if (launch && cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
                    return -1;
            }
            break;
        case PH_FACES:
            if constexpr (NV == 8)
                k = solver == SOLVER_LINEARIZED ? (const void*)kb_mhd_faces<SOLVER_LINEARIZED, R>
                                                : (const void*)kb_mhd_faces<SOLVER_HLL, R>;
            break;
        case PH_UPDATE:
            k = solver == SOLVER_LINEARIZED ? (const void*)kb_flux_update<SOLVER_LINEARIZED, NV, R>
                                            : (const void*)kb_flux_update<SOLVER_HLL, NV, R>;
            break;
        case PH_EMF:
            if constexpr (NV == 8) k = (const void*)kb_emf<R>;
            break;
        case PH_CT:
            if constexpr (NV == 8) k = (const void*)kb_ct<R>;
            break;
        default: break;
    }
    if (fn) *fn = k;
    if (!k) return 0;
    if (!launch) return team ? 2 : 1;
    void* args[] = {(void*)&g};
    return cudaLaunchKernel(k, dim3((unsigned)blocks), dim3((unsigned)threads), args, smem, st) == cudaSuccess ? 1 : -1;
}

template int batch_phase<ADER_BORDER, ADER_BNV>(int, const BatchGroupDev&, int, int, int, int, cudaStream_t, bool,
                                                const void**);

}  // namespace ader
