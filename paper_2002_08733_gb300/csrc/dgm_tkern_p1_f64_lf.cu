// Tangential-trace stage kernel: degree 1, double fields, leapfrog half steps.
#define DGM_P 1
#define DGM_REAL double
#define DGM_MODE MODE_LF_E
#define DGM_LAUNCH2 launch_t_p1_f64_lfh
#define DGM_LAUNCH launch_t_p1_f64_lf
#include "dgm_tkern_impl.cuh"
