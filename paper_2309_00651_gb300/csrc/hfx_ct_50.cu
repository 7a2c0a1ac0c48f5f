// Compile-time-geometry FP32 passes for 50^3 grids.
#define HFX_CT_N 50
#include "hfx_ct.inl"
