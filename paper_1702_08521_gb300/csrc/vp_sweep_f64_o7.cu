// vp_sweep_f64_o7.cu -- the sweeps of vp_sweep.cu in FP64 of order 7.
#define VP_SWEEP_ORDER 7
#define VP_SWEEP_REAL double
#define VP_UNIT(name) name##_f64_o7
#include "vp_sweep.cu"
