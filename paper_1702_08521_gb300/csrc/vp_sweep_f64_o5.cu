// vp_sweep_f64_o5.cu -- the sweeps of vp_sweep.cu in FP64 of order 5.
#define VP_SWEEP_ORDER 5
#define VP_SWEEP_REAL double
#define VP_UNIT(name) name##_f64_o5
#include "vp_sweep.cu"
