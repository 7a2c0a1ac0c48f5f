// Compile-time-geometry FP32 passes for 60^3 grids.
#define HFX_CT_N 60
#include "hfx_ct.inl"
