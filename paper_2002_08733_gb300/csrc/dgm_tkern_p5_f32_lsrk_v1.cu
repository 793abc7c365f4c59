// Tangential-trace stage kernel: degree 5, float fields, LSRK4 stage, tile variant 1
// (32 columns, 4 threads per column) for the autotuner.
#define DGM_P 5
#define DGM_REAL float
#define DGM_MODE MODE_LSRK
#define DGM_TE 32
#define DGM_NG 4
#define DGM_MINB 2
#define DGM_LAUNCH launch_t_p5_f32_lsrk_v1
#include "dgm_tkern_impl.cuh"
