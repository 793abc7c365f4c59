// Tangential-trace stage kernel: degree 2, float fields, right-hand side.
#define DGM_P 2
#define DGM_REAL float
#define DGM_MODE MODE_RHS
#define DGM_LAUNCH launch_t_p2_f32_rhs
#include "dgm_tkern_impl.cuh"
