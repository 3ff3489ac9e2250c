// vp_sweep_f64.cu -- the FP64 sweeps of vp_sweep.cu in a translation unit of
// their own: the two precisions compile in parallel.
#define VP_SWEEP_UNIT_F64
#include "vp_sweep.cu"
