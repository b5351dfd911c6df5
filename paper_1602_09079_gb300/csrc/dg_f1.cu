// Fused FP32-mixed stage kernel of the degree-1 modal DG basis (order 2).
#define DG_K 1
#include "dg_fused_inst.cuh"
