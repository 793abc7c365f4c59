// Tangential-trace stage kernel: degree 2, float fields, LSRK4 stage, tile variant 1
// (32 columns, 8 threads per column) for the autotuner.
#define DGM_P 2
#define DGM_REAL float
#define DGM_MODE MODE_LSRK
#define DGM_TE 32
#define DGM_NG 8
#define DGM_MINB 3
#define DGM_LAUNCH launch_t_p2_f32_lsrk_v1
#include "dgm_tkern_impl.cuh"
