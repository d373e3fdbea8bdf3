// Order-3 Euler predictor + face kernel in F64 (see step_inst.cuh): the dispatch; each
// kernel variant is compiled in its own unit, step_o3_euler_f64_<form>_<source>.cu.
#define ADER_ORDER 3
#define ADER_NV 5
#define ADER_REAL double
#define ADER_SPLIT_VARIANTS 1
#include "step_inst.cuh"
