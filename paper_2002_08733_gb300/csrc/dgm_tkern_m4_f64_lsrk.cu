// Tangential-trace stage kernel, mixed orders: E of degree 4, H of degree 3,
// double fields, LSRK4 stage.
#define DGM_P 4
#define DGM_REAL double
#define DGM_MODE MODE_LSRK
#define DGM_MIXED
#define DGM_LAUNCH launch_t_m4_f64_lsrk
#include "dgm_tkern_impl.cuh"
