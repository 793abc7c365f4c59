// Tangential-trace stage kernel: degree 2, double fields, LSRK4 stage.
#define DGM_P 2
#define DGM_REAL double
#define DGM_MODE MODE_LSRK
#define DGM_LAUNCH launch_t_p2_f64_lsrk
#include "dgm_tkern_impl.cuh"
