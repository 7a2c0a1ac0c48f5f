// Compile-time-geometry FP32 passes for 54^3 grids.
#define HFX_CT_N 54
#include "hfx_ct.inl"
