// Tangential-trace stage kernel: degree 2, double fields, right-hand side.
#define DGM_P 2
#define DGM_REAL double
#define DGM_MODE MODE_RHS
#define DGM_LAUNCH launch_t_p2_f64_rhs
#include "dgm_tkern_impl.cuh"
