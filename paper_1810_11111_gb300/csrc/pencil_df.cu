// Fused reaction pass, double-float F (see sgk_pencil.cuh).
#include "sgk_pencil.cuh"

SGK_PENCIL_DISPATCH(pencil_df_d2, df2, false, SGK_PENCIL_DF_D2)
SGK_PENCIL_DISPATCH(pencil_df_d34, df2, false, SGK_PENCIL_DF_D34)
