// Fused reaction pass, FP32, d = 2 (see sgk_pencil.cuh).
#include "sgk_pencil.cuh"

SGK_PENCIL_DISPATCH(pencil_f32_d2, float, false, SGK_PENCIL_D2)
SGK_PENCIL_DISPATCH(pencil_f32_d2_jac, float, true, SGK_PENCIL_D2)
