// Leapfrog half steps of plans with receivers: degree 3, float fields.
#define DGM_P 3
#define DGM_REAL float
#define DGM_LF 1
#define DGM_LAUNCH launch_p3_f32_lfe
#define DGM_LAUNCH2 launch_p3_f32_lfh
#include "dgm_kern_impl.cuh"
