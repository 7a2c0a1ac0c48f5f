// Compile-time-geometry FP32 passes for 108^3 grids.
#define HFX_CT_N 108
#include "hfx_ct.inl"
