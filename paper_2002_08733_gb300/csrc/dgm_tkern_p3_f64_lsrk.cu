// Tangential-trace stage kernel: degree 3, double fields, LSRK4 stage.
#define DGM_P 3
#define DGM_REAL double
#define DGM_MODE MODE_LSRK
#define DGM_LAUNCH launch_t_p3_f64_lsrk
#include "dgm_tkern_impl.cuh"
