// Compile-time-geometry FP32 passes for 120^3 grids.
#define HFX_CT_N 120
#include "hfx_ct.inl"
