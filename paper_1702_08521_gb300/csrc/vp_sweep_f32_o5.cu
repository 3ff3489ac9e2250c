// vp_sweep_f32_o5.cu -- the sweeps of vp_sweep.cu in FP32 of order 5.
#define VP_SWEEP_ORDER 5
#define VP_SWEEP_REAL float
#define VP_UNIT(name) name##_f32_o5
#include "vp_sweep.cu"
