// Tangential-trace stage kernel: degree 4, float fields, LSRK4 stage, tile variant 2
// (16 columns, 8 threads per column) for the autotuner.
#define DGM_P 4
#define DGM_REAL float
#define DGM_MODE MODE_LSRK
#define DGM_TE 16
#define DGM_NG 8
#define DGM_MINB 3
#define DGM_LAUNCH launch_t_p4_f32_lsrk_v2
#include "dgm_tkern_impl.cuh"
