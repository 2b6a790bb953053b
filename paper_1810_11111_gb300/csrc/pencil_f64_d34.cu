// Fused reaction pass, FP64, d = 3 and 4, F (see sgk_pencil.cuh).
#include "sgk_pencil.cuh"

SGK_PENCIL_DISPATCH(pencil_f64_d34, double, false, SGK_PENCIL_D34)
