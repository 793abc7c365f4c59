// Tangential-trace stage kernel, mixed orders: E of degree 2, H of degree 1,
// double fields, right-hand side.
#define DGM_P 2
#define DGM_REAL double
#define DGM_MODE MODE_RHS
#define DGM_MIXED
#define DGM_LAUNCH launch_t_m2_f64_rhs
#include "dgm_tkern_impl.cuh"
