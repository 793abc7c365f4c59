// Tangential-trace stage kernel, mixed orders: E of degree 3, H of degree 2,
// double fields, LSRK4 stage.
#define DGM_P 3
#define DGM_REAL double
#define DGM_MODE MODE_LSRK
#define DGM_MIXED
#define DGM_LAUNCH launch_t_m3_f64_lsrk
#include "dgm_tkern_impl.cuh"
