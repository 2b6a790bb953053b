// Fused reaction pass, FP64, d = 2 (see sgk_pencil.cuh).
#include "sgk_pencil.cuh"

SGK_PENCIL_DISPATCH(pencil_f64_d2, double, false, SGK_PENCIL_D2)
SGK_PENCIL_DISPATCH(pencil_f64_d2_jac, double, true, SGK_PENCIL_D2)
