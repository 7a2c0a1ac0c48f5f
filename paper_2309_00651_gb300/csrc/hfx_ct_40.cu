// Compile-time-geometry FP32 passes for 40^3 grids.
#define HFX_CT_N 40
#include "hfx_ct.inl"
