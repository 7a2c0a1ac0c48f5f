// Compile-time-geometry FP32 passes for 100^3 grids.
#define HFX_CT_N 100
#include "hfx_ct.inl"
