// Fused reaction pass, FP32, d = 3 and 4, F (see sgk_pencil.cuh).
#include "sgk_pencil.cuh"

SGK_PENCIL_DISPATCH(pencil_f32_d34, float, false, SGK_PENCIL_D34)
