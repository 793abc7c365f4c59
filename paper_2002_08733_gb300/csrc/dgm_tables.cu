// Dispatch tables over the per-(degree, precision, mode) kernel modules.
//
// tang_kernel (dgm_tang.cuh) is the default; FP32 LSRK variants for the
// autotuner: 0 = the shape measured best (by the number of tiles, see few_tiles), 1 = 32 columns x 8 threads per column
// (p >= 4: x 4), 2 = 16 columns x 8, p >= 4: 3 = 32 x 8 with more registers; up to
// p = 3 (where 64 columns of pairs fit in shared memory) 3 = paired kernel with
// packed FP32x2 arithmetic, 4 = paired kernel with scalar arithmetic; at p = 2, 3
// also 5 = tensor-core variant (64 columns x 512 threads, curl and lift on tcgen05).
//
// FP32 plans created for receivers (max_receivers > 0) and without the penalty
// (prm.recorded) run stage_kernel (dgm_stage.cuh) in the LSRK mode and lf_kernel
// (dgm_lf.cuh) in the leapfrog modes: receiver records and the adjoint's gradients
// are FP64 results formed from FP32 fields, and what was recorded before stays
// reproducible to FP64 accuracy only if the fields keep their rounding.  stage_kernel's
// variants: 0 = 32 columns x 384 threads, 1 = 32 x 192, 2 = 16 x 192, p >= 4:
// 3 = 32 x 512.
#include "dgm_internal.h"
#include "dgmax.h"

namespace dgm {

int launch_t_p1_f32_lsrk(const StageParams&, void*);
int launch_t_p1_f32_rhs(const StageParams&, void*);
int launch_t_p1_f32_lf(const StageParams&, void*);
int launch_t_p1_f32_lfh(const StageParams&, void*);
int launch_p1_f32_raw(const StageParams&, void*);
int launch_t_p1_f32_lsrk_v1(const StageParams&, void*);
int launch_t_p1_f32_lsrk_v2(const StageParams&, void*);
int launch_p1_f32_lsrk(const StageParams&, void*);
int launch_p1_f32_lfe(const StageParams&, void*);
int launch_p1_f32_lfh(const StageParams&, void*);
int launch_p1_f32_lsrk_v1(const StageParams&, void*);
int launch_p1_f32_lsrk_v2(const StageParams&, void*);
int launch_p1_f32_lsrk_v3(const StageParams&, void*);
int launch_p1_f32_lsrk_v4(const StageParams&, void*);
int launch_p1_f32_adj(const AdjParams&, void*);
int launch_t_p1_f64_lsrk(const StageParams&, void*);
int launch_t_p1_f64_rhs(const StageParams&, void*);
int launch_t_p1_f64_lf(const StageParams&, void*);
int launch_t_p1_f64_lfh(const StageParams&, void*);
int launch_p1_f64_raw(const StageParams&, void*);
int launch_p1_f64_adj(const AdjParams&, void*);
int launch_t_p2_f32_lsrk(const StageParams&, void*);
int launch_t_p2_f32_rhs(const StageParams&, void*);
int launch_t_p2_f32_lf(const StageParams&, void*);
int launch_t_p2_f32_lfh(const StageParams&, void*);
int launch_p2_f32_raw(const StageParams&, void*);
int launch_t_p2_f32_lsrk_v1(const StageParams&, void*);
int launch_t_p2_f32_lsrk_v2(const StageParams&, void*);
int launch_p2_f32_lsrk(const StageParams&, void*);
int launch_p2_f32_lfe(const StageParams&, void*);
int launch_p2_f32_lfh(const StageParams&, void*);
int launch_p2_f32_lsrk_v1(const StageParams&, void*);
int launch_p2_f32_lsrk_v2(const StageParams&, void*);
int launch_p2_f32_lsrk_v3(const StageParams&, void*);
int launch_p2_f32_lsrk_v4(const StageParams&, void*);
int launch_p2_f32_lsrk_v5(const StageParams&, void*);
int launch_p2_f32_adj(const AdjParams&, void*);
int launch_t_p2_f64_lsrk(const StageParams&, void*);
int launch_t_p2_f64_rhs(const StageParams&, void*);
int launch_t_p2_f64_lf(const StageParams&, void*);
int launch_t_p2_f64_lfh(const StageParams&, void*);
int launch_p2_f64_raw(const StageParams&, void*);
int launch_p2_f64_adj(const AdjParams&, void*);
int launch_t_p3_f32_lsrk(const StageParams&, void*);
int launch_t_p3_f32_rhs(const StageParams&, void*);
int launch_t_p3_f32_lf(const StageParams&, void*);
int launch_t_p3_f32_lfh(const StageParams&, void*);
int launch_p3_f32_raw(const StageParams&, void*);
int launch_t_p3_f32_lsrk_v1(const StageParams&, void*);
int launch_t_p3_f32_lsrk_v2(const StageParams&, void*);
int launch_p3_f32_lsrk(const StageParams&, void*);
int launch_p3_f32_lfe(const StageParams&, void*);
int launch_p3_f32_lfh(const StageParams&, void*);
int launch_p3_f32_lsrk_v1(const StageParams&, void*);
int launch_p3_f32_lsrk_v2(const StageParams&, void*);
int launch_p3_f32_lsrk_v3(const StageParams&, void*);
int launch_p3_f32_lsrk_v4(const StageParams&, void*);
int launch_p3_f32_lsrk_v5(const StageParams&, void*);
int launch_p3_f32_adj(const AdjParams&, void*);
int launch_t_p3_f64_lsrk(const StageParams&, void*);
int launch_t_p3_f64_rhs(const StageParams&, void*);
int launch_t_p3_f64_lf(const StageParams&, void*);
int launch_t_p3_f64_lfh(const StageParams&, void*);
int launch_p3_f64_raw(const StageParams&, void*);
int launch_p3_f64_adj(const AdjParams&, void*);
int launch_t_p4_f32_lsrk(const StageParams&, void*);
int launch_t_p4_f32_rhs(const StageParams&, void*);
int launch_t_p4_f32_lf(const StageParams&, void*);
int launch_t_p4_f32_lfh(const StageParams&, void*);
int launch_p4_f32_raw(const StageParams&, void*);
int launch_t_p4_f32_lsrk_v1(const StageParams&, void*);
int launch_t_p4_f32_lsrk_v2(const StageParams&, void*);
int launch_t_p4_f32_lsrk_v3(const StageParams&, void*);
int launch_p4_f32_lsrk(const StageParams&, void*);
int launch_p4_f32_lfe(const StageParams&, void*);
int launch_p4_f32_lfh(const StageParams&, void*);
int launch_p4_f32_lsrk_v1(const StageParams&, void*);
int launch_p4_f32_lsrk_v2(const StageParams&, void*);
int launch_p4_f32_lsrk_v3(const StageParams&, void*);
int launch_p4_f32_adj(const AdjParams&, void*);
int launch_t_p4_f64_lsrk(const StageParams&, void*);
int launch_t_p4_f64_rhs(const StageParams&, void*);
int launch_t_p4_f64_lf(const StageParams&, void*);
int launch_t_p4_f64_lfh(const StageParams&, void*);
int launch_p4_f64_raw(const StageParams&, void*);
int launch_p4_f64_adj(const AdjParams&, void*);
int launch_t_p5_f32_lsrk(const StageParams&, void*);
int launch_t_p5_f32_rhs(const StageParams&, void*);
int launch_t_p5_f32_lf(const StageParams&, void*);
int launch_t_p5_f32_lfh(const StageParams&, void*);
int launch_p5_f32_raw(const StageParams&, void*);
int launch_t_p5_f32_lsrk_v1(const StageParams&, void*);
int launch_t_p5_f32_lsrk_v2(const StageParams&, void*);
int launch_t_p5_f32_lsrk_v3(const StageParams&, void*);
int launch_p5_f32_lsrk(const StageParams&, void*);
int launch_p5_f32_lfe(const StageParams&, void*);
int launch_p5_f32_lfh(const StageParams&, void*);
int launch_p5_f32_lsrk_v1(const StageParams&, void*);
int launch_p5_f32_lsrk_v2(const StageParams&, void*);
int launch_p5_f32_lsrk_v3(const StageParams&, void*);
int launch_p5_f32_adj(const AdjParams&, void*);

// mixed orders (E of degree p, H of degree p - 1)
int launch_t_m2_f32_lsrk(const StageParams&, void*);
int launch_t_m2_f32_rhs(const StageParams&, void*);
int launch_t_m2_f64_lsrk(const StageParams&, void*);
int launch_t_m2_f64_rhs(const StageParams&, void*);
int launch_t_m3_f32_lsrk(const StageParams&, void*);
int launch_t_m3_f32_rhs(const StageParams&, void*);
int launch_t_m3_f64_lsrk(const StageParams&, void*);
int launch_t_m3_f64_rhs(const StageParams&, void*);
int launch_t_m4_f32_lsrk(const StageParams&, void*);
int launch_t_m4_f32_rhs(const StageParams&, void*);
int launch_t_m4_f64_lsrk(const StageParams&, void*);
int launch_t_m4_f64_rhs(const StageParams&, void*);

namespace {

// FP32 LSRK4 stages of few tiles of 32 columns.  No more of them than SMs (p = 4: than two
// per SM): the CTAs run side by side, and eight threads per column fill the SMs better than
// four, which win once more CTAs queue.  us per stage, four | eight threads: 137 tiles p = 1
// 3.99 | 3.28, p = 2 5.10 | 4.71 (PML 9.05 | 7.35), p = 3 9.26 | 7.86, p = 4 19.7 | 15.3;
// 274 tiles p = 4 20.0 | 17.0 (PML 27.6 | 23.1); 324 tiles p = 1 4.06 | 4.24, p = 2
// 5.40 | 5.51, p = 4 19.0 | 23.9.  (The penalty and p = 5 always run eight.)
bool few_tiles(const StageParams& prm, int per_sm = 1) {
    constexpr int64_t kSMs = 152;
    return prm.hs == nullptr && (prm.K_active * prm.S + 31) / 32 <= per_sm * kSMs;
}

int launch_p1_f32(const StageParams& prm, int mode, void* st) {
    const bool rec = prm.recorded != 0;
    switch (mode) {
        case MODE_RHS: return launch_t_p1_f32_rhs(prm, st);
        case MODE_LSRK:
            switch (prm.variant) {
                case 1: return rec ? launch_p1_f32_lsrk_v1(prm, st) : launch_t_p1_f32_lsrk_v1(prm, st);
                case 2: return rec ? launch_p1_f32_lsrk_v2(prm, st) : launch_t_p1_f32_lsrk_v2(prm, st);
                case 3: return launch_p1_f32_lsrk_v3(prm, st);
                case 4: return launch_p1_f32_lsrk_v4(prm, st);
                default:
                    return rec              ? launch_p1_f32_lsrk(prm, st)
                           : few_tiles(prm) ? launch_t_p1_f32_lsrk_v1(prm, st)
                                            : launch_t_p1_f32_lsrk(prm, st);
            }
        case MODE_LF_E: return rec ? launch_p1_f32_lfe(prm, st) : launch_t_p1_f32_lf(prm, st);
        case MODE_LF_H: return rec ? launch_p1_f32_lfh(prm, st) : launch_t_p1_f32_lfh(prm, st);
        case MODE_RAW: return launch_p1_f32_raw(prm, st);
        default: return DGM_EINVAL;
    }
}

int launch_p1_f64(const StageParams& prm, int mode, void* st) {
    switch (mode) {
        case MODE_RHS: return launch_t_p1_f64_rhs(prm, st);
        case MODE_LSRK: return launch_t_p1_f64_lsrk(prm, st);
        case MODE_LF_E: return launch_t_p1_f64_lf(prm, st);
        case MODE_LF_H: return launch_t_p1_f64_lfh(prm, st);
        case MODE_RAW: return launch_p1_f64_raw(prm, st);
        default: return DGM_EINVAL;
    }
}

int launch_p2_f32(const StageParams& prm, int mode, void* st) {
    const bool rec = prm.recorded != 0;
    switch (mode) {
        case MODE_RHS: return launch_t_p2_f32_rhs(prm, st);
        case MODE_LSRK:
            switch (prm.variant) {
                case 1: return rec ? launch_p2_f32_lsrk_v1(prm, st) : launch_t_p2_f32_lsrk_v1(prm, st);
                case 2: return rec ? launch_p2_f32_lsrk_v2(prm, st) : launch_t_p2_f32_lsrk_v2(prm, st);
                case 3: return launch_p2_f32_lsrk_v3(prm, st);
                case 4: return launch_p2_f32_lsrk_v4(prm, st);
                case 5: return launch_p2_f32_lsrk_v5(prm, st);
                default:
                    return rec              ? launch_p2_f32_lsrk(prm, st)
                           : few_tiles(prm) ? launch_t_p2_f32_lsrk_v1(prm, st)
                                            : launch_t_p2_f32_lsrk(prm, st);
            }
        case MODE_LF_E: return rec ? launch_p2_f32_lfe(prm, st) : launch_t_p2_f32_lf(prm, st);
        case MODE_LF_H: return rec ? launch_p2_f32_lfh(prm, st) : launch_t_p2_f32_lfh(prm, st);
        case MODE_RAW: return launch_p2_f32_raw(prm, st);
        default: return DGM_EINVAL;
    }
}

int launch_p2_f64(const StageParams& prm, int mode, void* st) {
    switch (mode) {
        case MODE_RHS: return launch_t_p2_f64_rhs(prm, st);
        case MODE_LSRK: return launch_t_p2_f64_lsrk(prm, st);
        case MODE_LF_E: return launch_t_p2_f64_lf(prm, st);
        case MODE_LF_H: return launch_t_p2_f64_lfh(prm, st);
        case MODE_RAW: return launch_p2_f64_raw(prm, st);
        default: return DGM_EINVAL;
    }
}

int launch_p3_f32(const StageParams& prm, int mode, void* st) {
    const bool rec = prm.recorded != 0;
    switch (mode) {
        case MODE_RHS: return launch_t_p3_f32_rhs(prm, st);
        case MODE_LSRK:
            switch (prm.variant) {
                case 1: return rec ? launch_p3_f32_lsrk_v1(prm, st) : launch_t_p3_f32_lsrk_v1(prm, st);
                case 2: return rec ? launch_p3_f32_lsrk_v2(prm, st) : launch_t_p3_f32_lsrk_v2(prm, st);
                case 3: return launch_p3_f32_lsrk_v3(prm, st);
                case 4: return launch_p3_f32_lsrk_v4(prm, st);
                case 5: return launch_p3_f32_lsrk_v5(prm, st);
                default:
                    return rec              ? launch_p3_f32_lsrk(prm, st)
                           : few_tiles(prm) ? launch_t_p3_f32_lsrk_v1(prm, st)
                                            : launch_t_p3_f32_lsrk(prm, st);
            }
        case MODE_LF_E: return rec ? launch_p3_f32_lfe(prm, st) : launch_t_p3_f32_lf(prm, st);
        case MODE_LF_H: return rec ? launch_p3_f32_lfh(prm, st) : launch_t_p3_f32_lfh(prm, st);
        case MODE_RAW: return launch_p3_f32_raw(prm, st);
        default: return DGM_EINVAL;
    }
}

int launch_p3_f64(const StageParams& prm, int mode, void* st) {
    switch (mode) {
        case MODE_RHS: return launch_t_p3_f64_rhs(prm, st);
        case MODE_LSRK: return launch_t_p3_f64_lsrk(prm, st);
        case MODE_LF_E: return launch_t_p3_f64_lf(prm, st);
        case MODE_LF_H: return launch_t_p3_f64_lfh(prm, st);
        case MODE_RAW: return launch_p3_f64_raw(prm, st);
        default: return DGM_EINVAL;
    }
}

int launch_p4_f32(const StageParams& prm, int mode, void* st) {
    const bool rec = prm.recorded != 0;
    switch (mode) {
        case MODE_RHS: return launch_t_p4_f32_rhs(prm, st);
        case MODE_LSRK:
            switch (prm.variant) {
                case 1: return rec ? launch_p4_f32_lsrk_v1(prm, st) : launch_t_p4_f32_lsrk_v1(prm, st);
                case 2: return rec ? launch_p4_f32_lsrk_v2(prm, st) : launch_t_p4_f32_lsrk_v2(prm, st);
                case 3: return rec ? launch_p4_f32_lsrk_v3(prm, st) : launch_t_p4_f32_lsrk_v3(prm, st);
                default:
                    return rec              ? launch_p4_f32_lsrk(prm, st)
                           : few_tiles(prm, 2) ? launch_t_p4_f32_lsrk_v3(prm, st)
                                            : launch_t_p4_f32_lsrk(prm, st);
            }
        case MODE_LF_E: return rec ? launch_p4_f32_lfe(prm, st) : launch_t_p4_f32_lf(prm, st);
        case MODE_LF_H: return rec ? launch_p4_f32_lfh(prm, st) : launch_t_p4_f32_lfh(prm, st);
        case MODE_RAW: return launch_p4_f32_raw(prm, st);
        default: return DGM_EINVAL;
    }
}

int launch_p4_f64(const StageParams& prm, int mode, void* st) {
    switch (mode) {
        case MODE_RHS: return launch_t_p4_f64_rhs(prm, st);
        case MODE_LSRK: return launch_t_p4_f64_lsrk(prm, st);
        case MODE_LF_E: return launch_t_p4_f64_lf(prm, st);
        case MODE_LF_H: return launch_t_p4_f64_lfh(prm, st);
        case MODE_RAW: return launch_p4_f64_raw(prm, st);
        default: return DGM_EINVAL;
    }
}

int launch_p5_f32(const StageParams& prm, int mode, void* st) {
    const bool rec = prm.recorded != 0;
    switch (mode) {
        case MODE_RHS: return launch_t_p5_f32_rhs(prm, st);
        case MODE_LSRK:
            switch (prm.variant) {
                case 1: return rec ? launch_p5_f32_lsrk_v1(prm, st) : launch_t_p5_f32_lsrk_v1(prm, st);
                case 2: return rec ? launch_p5_f32_lsrk_v2(prm, st) : launch_t_p5_f32_lsrk_v2(prm, st);
                case 3: return rec ? launch_p5_f32_lsrk_v3(prm, st) : launch_t_p5_f32_lsrk_v3(prm, st);
                default: return rec ? launch_p5_f32_lsrk(prm, st) : launch_t_p5_f32_lsrk(prm, st);
            }
        case MODE_LF_E: return rec ? launch_p5_f32_lfe(prm, st) : launch_t_p5_f32_lf(prm, st);
        case MODE_LF_H: return rec ? launch_p5_f32_lfh(prm, st) : launch_t_p5_f32_lfh(prm, st);
        case MODE_RAW: return launch_p5_f32_raw(prm, st);
        default: return DGM_EINVAL;
    }
}

int launch_m2_f32(const StageParams& prm, int mode, void* st) {
    if (mode == MODE_RHS) return launch_t_m2_f32_rhs(prm, st);
    if (mode == MODE_LSRK) return launch_t_m2_f32_lsrk(prm, st);
    return DGM_EUNSUP;
}

int launch_m2_f64(const StageParams& prm, int mode, void* st) {
    if (mode == MODE_RHS) return launch_t_m2_f64_rhs(prm, st);
    if (mode == MODE_LSRK) return launch_t_m2_f64_lsrk(prm, st);
    return DGM_EUNSUP;
}

int launch_m3_f32(const StageParams& prm, int mode, void* st) {
    if (mode == MODE_RHS) return launch_t_m3_f32_rhs(prm, st);
    if (mode == MODE_LSRK) return launch_t_m3_f32_lsrk(prm, st);
    return DGM_EUNSUP;
}

int launch_m3_f64(const StageParams& prm, int mode, void* st) {
    if (mode == MODE_RHS) return launch_t_m3_f64_rhs(prm, st);
    if (mode == MODE_LSRK) return launch_t_m3_f64_lsrk(prm, st);
    return DGM_EUNSUP;
}

int launch_m4_f32(const StageParams& prm, int mode, void* st) {
    if (mode == MODE_RHS) return launch_t_m4_f32_rhs(prm, st);
    if (mode == MODE_LSRK) return launch_t_m4_f32_lsrk(prm, st);
    return DGM_EUNSUP;
}

int launch_m4_f64(const StageParams& prm, int mode, void* st) {
    if (mode == MODE_RHS) return launch_t_m4_f64_rhs(prm, st);
    if (mode == MODE_LSRK) return launch_t_m4_f64_lsrk(prm, st);
    return DGM_EUNSUP;
}

}  // namespace

extern const KernelTable kernels_p1_f32 = {launch_p1_f32, 4, launch_p1_f32_adj, 5};
extern const KernelTable kernels_p1_f64 = {launch_p1_f64, 8, launch_p1_f64_adj, 1};
extern const KernelTable kernels_p2_f32 = {launch_p2_f32, 4, launch_p2_f32_adj, 6};
extern const KernelTable kernels_p2_f64 = {launch_p2_f64, 8, launch_p2_f64_adj, 1};
extern const KernelTable kernels_p3_f32 = {launch_p3_f32, 4, launch_p3_f32_adj, 6};
extern const KernelTable kernels_p3_f64 = {launch_p3_f64, 8, launch_p3_f64_adj, 1};
extern const KernelTable kernels_p4_f32 = {launch_p4_f32, 4, launch_p4_f32_adj, 4};
extern const KernelTable kernels_p4_f64 = {launch_p4_f64, 8, launch_p4_f64_adj, 1};
extern const KernelTable kernels_p5_f32 = {launch_p5_f32, 4, launch_p5_f32_adj, 4};

// Kernels of mixed-order plans: E degree pE = 2..4 (H degree pE - 1).
const KernelTable* kernel_table_mixed(int pE, int precision) {
    static const KernelTable f32[] = {{launch_m2_f32, 4, nullptr, 1}, {launch_m3_f32, 4, nullptr, 1}, {launch_m4_f32, 4, nullptr, 1}};
    static const KernelTable f64[] = {{launch_m2_f64, 8, nullptr, 1}, {launch_m3_f64, 8, nullptr, 1}, {launch_m4_f64, 8, nullptr, 1}};
    if (pE < 2 || pE > 4) return nullptr;
    return precision == DGM_FP64 ? &f64[pE - 2] : (precision == DGM_FP32 ? &f32[pE - 2] : nullptr);
}

}  // namespace dgm
