// Order-3 Euler predictor + face kernel in F32, modal form, with a source (see step_inst.cuh).
#define ADER_ORDER 3
#define ADER_NV 5
#define ADER_REAL float
#define ADER_FORM FORM_MODAL
#define ADER_SRC true
#include "step_inst.cuh"
