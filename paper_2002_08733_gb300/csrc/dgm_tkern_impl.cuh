// Body of one translation unit of the tangential-trace stage kernel: instantiates
// tang_kernel for one polynomial degree (DGM_P), one field precision (DGM_REAL)
// and one mode (DGM_MODE; MODE_LF_E with DGM_LAUNCH2 also instantiates
// MODE_LF_H; DGM_MIXED: E of degree DGM_P, H of
// DGM_P - 1), and exports its launchers.  Included by the
// dgm_tkern_p<P>_<precision>_<mode>.cu files; one mode per file keeps the
// heavily unrolled kernels compiling in parallel.
#include <cuda_runtime.h>

#include "dgm_internal.h"
#include "dgm_tang.cuh"
#include "dgmax.h"

namespace dgm {
namespace {

constexpr int kP = DGM_P;
using Real = DGM_REAL;
// Tile shape of tang_kernel: threads side by side (columns per CTA), threads per
// column, and resident CTAs per SM asked of the register allocator (DGM_TE /
// DGM_NG / DGM_MINB select an autotuner variant).
template <int MODE, bool SIP, bool PML>
struct Shape {
    static constexpr bool kLF = MODE == MODE_LF_E || MODE == MODE_LF_H, kF64 = sizeof(Real) == 8;
#ifdef DGM_TE
    static constexpr int TE = DGM_TE, NG = DGM_NG, MINB = DGM_MINB;
#else
    // FP32: four threads per column while a thread's rows (half of them) and a
    // trace's coefficients fit its registers, eight from p = 5 on, and at p = 4
    // with the penalty's facet values besides.  (p = 4 with a PML, LSRK4, us, eight
    // threads on 80 registers | four on 168: 250 tiles of 32 columns 47.4 | 27.9, 768 tiles
    // 118 | 62.7; right-hand side of 999 tiles 110 | 64.7)
    // FP64 (bound by the FP64 pipe, which few warps saturate): full warps of 32
    // columns, so that no warp runs two faces or row parts in turn.
    static constexpr int TE = 32;
    static constexpr int NG = kLF ? (kF64 ? 4 : kP <= 4 ? 4 : 8)
                                  : kF64 || SIP || kP == 5 ? 8 : 4;
    static constexpr int MINB =
        kF64 ? (kLF ? (kP <= 3 ? 2 : 1) : kP <= 3 ? 2 : 1)
        : SIP ? (kP <= 3 ? 3 : 2)
        : kP == 1 ? 8 : kP == 2 ? (PML ? 6 : 7) : kP == 3 ? (kLF ? 5 : 4)
        : kP == 4 ? 3 : 2;
#endif
};

// the interior penalty runs in the default shape
#ifdef DGM_MIXED
constexpr bool kMX = true;   // E of degree kP, H of degree kP - 1
#else
constexpr bool kMX = false;
#endif
#if !defined(DGM_TE) && !defined(DGM_MIXED)
constexpr bool kSIP = true;
#else
constexpr bool kSIP = false;
#endif

// Most tiles (of 32 columns) for which the cluster form is taken: two of its CTAs per
// SM (8 x 38 = 2 x 152; three would wait for one another's FP64 pipes).
constexpr unsigned kClusterTiles = 38;

template <int MODE, typename IX, bool SIP, bool PML>
int launch_ix(const StageParams& q, unsigned grid, cudaStream_t st) {
    using Sh = Shape<MODE, SIP, PML>;
    constexpr size_t smem = tang_smem_bytes<kP, Real, Sh::TE, kMX>();
    static bool configured = false;
    auto k = tang_kernel<kP, Real, Sh::TE, Sh::NG, MODE, IX, SIP, PML, kMX, Sh::MINB>;
    if (!configured) {
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)) !=
            cudaSuccess)
            return DGM_ECUDA;
        configured = true;
    }
    return launch_ex(k, grid, Sh::TE * Sh::NG, smem, st, q.pdl != 0, 1, q) == cudaSuccess ? DGM_OK : DGM_ECUDA;
}

// true when every index the kernel forms for this plan is below 2^32: field
// rows (6N x C), auxiliaries (6N x npml S), geometry (G_COUNT x K), the constant
// table (TG_ROWS x K), incident jump terms (3 NF per boundary face)
bool fits_32bit(const StageParams& p) {
    const uint64_t lim = uint64_t(1) << 32;
    const uint64_t K = uint64_t(p.K), C = K * uint64_t(p.S);
    const uint64_t N = uint64_t(nmodes(kP)), NF = uint64_t(nfmodes(kP));
    return 6 * N * C < lim && 6 * N * uint64_t(p.npml) * uint64_t(p.S) < lim &&
           uint64_t(G_COUNT) * K < lim && uint64_t(TG_ROWS) * K < lim && 12 * NF * K < lim;
}

// FP64 meshes of few tiles: a cluster of eight CTAs per tile (see tang_kernel).
// With a tile per CTA the launch takes as long as one SM's FP64 pipe needs for one
// tile, however few there are; a cluster spreads a tile over eight SMs.  us per launch
// of 12 tiles, one CTA | cluster: leapfrog p = 2 15.1 | 7.0; with clusters of
// one-warp CTAs p = 3 37 | 23, LSRK4 p = 4 140 | 90, and from 65 tiles on no gain.
template <int MODE>
int launch_cluster(const StageParams& q, unsigned tiles, cudaStream_t st) {
    constexpr size_t smem = tang_smem_bytes<kP, Real, 32, false>();
    static bool configured = false;
    auto k = tang_kernel<kP, Real, 32, 8, MODE, uint32_t, false, true, false, 1, 8>;
    if (!configured) {
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)) != cudaSuccess)
            return DGM_ECUDA;
        configured = true;
    }
    return launch_ex(k, 8 * tiles, 32 * CLW, smem, st, q.pdl != 0, 8, q) == cudaSuccess ? DGM_OK : DGM_ECUDA;
}

template <int MODE>
int launch_mode(const StageParams& prm, cudaStream_t st) {
    const int64_t C = prm.K_active * prm.S;   // columns updated
    if (C <= 0) return DGM_OK;
    constexpr int kTE = Shape<MODE, false, false>::TE;   // (the same for every shape of a mode)
    const unsigned grid = unsigned((C + kTE - 1) / kTE);
    StageParams q = prm;
    q.dt_f = float(prm.dt);
    q.a_f = float(prm.a);
    q.b_f = float(prm.b);
    const bool i32 = !q.force_index64 && fits_32bit(q);
    // the tile's bulk copy: the plan's tensor-map set of this tile width and the
    // map of this stage's input
    q.tm_u = -1;
    if (q.tmaps != nullptr) {
        constexpr int kSet = kTE == tmap_columns(0) ? 0 : 1;
        static_assert(kTE == tmap_columns(kSet), "a tensor-map set of this tile width");
        q.tmaps = static_cast<const char*>(q.tmaps) + size_t(kSet) * TMAP_COUNT * TMAP_BYTES;
        q.tm_u = q.u == q.tm_f0 ? TM_U0
                 : q.u == q.tm_f1 ? TM_U1
                 : (q.tm_fw != nullptr && q.u == q.tm_fw) ? TM_UW : -1;
    }
    if (q.hs != nullptr) {   // interior penalty
        if constexpr (kSIP && (MODE == MODE_LSRK || MODE == MODE_RHS)) {
            return i32 ? launch_ix<MODE, uint32_t, true, false>(q, grid, st) : launch_ix<MODE, int64_t, true, false>(q, grid, st);
        } else {
            return DGM_EUNSUP;
        }
    }
    if constexpr (sizeof(Real) == 8 && !kMX && MODE != MODE_RHS) {
        if (i32 && grid <= kClusterTiles) return launch_cluster<MODE>(q, grid, st);
    }
    // (64-bit indices: the PML instantiation serves plans without a layer too)
    if (!i32) return launch_ix<MODE, int64_t, false, !kMX>(q, grid, st);
    if constexpr (!kMX) {
        if (q.pml != nullptr && q.npml > 0) return launch_ix<MODE, uint32_t, false, true>(q, grid, st);
    }
    return launch_ix<MODE, uint32_t, false, false>(q, grid, st);
}

}  // namespace

int DGM_LAUNCH(const StageParams& prm, void* stream) {
    return launch_mode<DGM_MODE>(prm, static_cast<cudaStream_t>(stream));
}
#ifdef DGM_LAUNCH2
int DGM_LAUNCH2(const StageParams& prm, void* stream) {
    return launch_mode<MODE_LF_H>(prm, static_cast<cudaStream_t>(stream));
}
#endif

}  // namespace dgm
