// Leapfrog half steps of plans with receivers: degree 5, float fields.
#define DGM_P 5
#define DGM_REAL float
#define DGM_LF 1
#define DGM_LAUNCH launch_p5_f32_lfe
#define DGM_LAUNCH2 launch_p5_f32_lfh
#include "dgm_kern_impl.cuh"
