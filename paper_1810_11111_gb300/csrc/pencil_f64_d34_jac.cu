// Fused reaction pass, FP64, d = 3 and 4, Jacobian products (see sgk_pencil.cuh).
#include "sgk_pencil.cuh"

SGK_PENCIL_DISPATCH(pencil_f64_d34_jac, double, true, SGK_PENCIL_D34)
