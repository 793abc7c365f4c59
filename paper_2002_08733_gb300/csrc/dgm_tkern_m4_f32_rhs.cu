// Tangential-trace stage kernel, mixed orders: E of degree 4, H of degree 3,
// float fields, right-hand side.
#define DGM_P 4
#define DGM_REAL float
#define DGM_MODE MODE_RHS
#define DGM_MIXED
#define DGM_LAUNCH launch_t_m4_f32_rhs
#include "dgm_tkern_impl.cuh"
