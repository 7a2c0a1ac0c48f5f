// Compile-time-geometry FP32 passes for 36^3 grids.
#define HFX_CT_N 36
#include "hfx_ct.inl"
