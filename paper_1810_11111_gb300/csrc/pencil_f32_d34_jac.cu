// Fused reaction pass, FP32, d = 3 and 4, Jacobian products (see sgk_pencil.cuh).
#include "sgk_pencil.cuh"

SGK_PENCIL_DISPATCH(pencil_f32_d34_jac, float, true, SGK_PENCIL_D34)
