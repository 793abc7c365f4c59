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
    // 118 | 62.7, 12,000 tiles 2405 | 1079; right-hand side of 999 tiles 110 | 64.7)
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

#ifdef DGM_MIXED
constexpr bool kMX = true;   // E of degree kP, H of degree kP - 1
#else
constexpr bool kMX = false;
#endif
// not an autotuner variant: all modes, the interior penalty, the rules for few tiles
#ifdef DGM_TE
constexpr bool kDefault = false;
#else
constexpr bool kDefault = true;
#endif

// the tensor map of this stage's input for the tile's bulk copy (TmapIndex), or -1
int tile_map(const StageParams& q) {
    if (q.tmaps == nullptr) return -1;
    return q.u == q.tm_f0 ? TM_U0 : q.u == q.tm_f1 ? TM_U1 : (q.tm_fw != nullptr && q.u == q.tm_fw) ? TM_UW : -1;
}

template <int TE, int NG, int MODE, typename IX, bool SIP, bool PML, int MINB, int CL = 1>
int launch_shape(StageParams& q, int64_t columns, cudaStream_t st) {
    constexpr size_t smem = tang_smem_bytes<kP, Real, TE, kMX>();
    static OncePerDevice once;
    auto k = tang_kernel<kP, Real, TE, NG, MODE, IX, SIP, PML, kMX, MINB, CL>;
    if (!opt_in_smem(k, smem, once)) return DGM_ECUDA;
    // the plan's tensor-map set of this tile width
    constexpr int kSet = TE == tmap_columns(0) ? 0 : 1;
    static_assert(TE == tmap_columns(kSet), "a tensor-map set of this tile width");
    q.tm_u = tile_map(q);
    if (q.tm_u >= 0) q.tmaps = static_cast<const char*>(q.tmaps) + size_t(kSet) * TMAP_COUNT * TMAP_BYTES;
    const unsigned tiles = unsigned((columns + TE - 1) / TE);
    return launch_ex(k, CL * tiles, CL > 1 ? TE * CLW : TE * NG, smem, st, q.pdl != 0, CL, q) == cudaSuccess
               ? DGM_OK : DGM_ECUDA;
}

template <int MODE, typename IX, bool SIP, bool PML>
int launch_ix(StageParams& q, int64_t columns, cudaStream_t st) {
    using Sh = Shape<MODE, SIP, PML>;
    return launch_shape<Sh::TE, Sh::NG, MODE, IX, SIP, PML, Sh::MINB>(q, columns, st);
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

// Rules for few tiles (of 32 columns; one CTA of the ordinary shape works on each).
//
// FP64.  The launch takes as long as one SM's FP64 pipe needs for one tile, however few
// there are.  LSRK4 and leapfrog up to kClusterTiles: a cluster of eight CTAs spreads a tile
// over eight SMs (see tang_kernel; two of its CTAs per SM, 8 x 38 = 2 x 152; three would
// wait for one another's FP64 pipes).  us per launch of 12 tiles, one CTA | cluster: leapfrog
// p = 2 15.1 | 7.0; with clusters of one-warp CTAs p = 3 37 | 23, LSRK4 p = 4 140 | 90.
// LSRK4 beyond and right-hand sides, up to kHalfTiles: tiles of 16 columns, which still find
// an SM each.  65 tiles, 32 columns | 16: LSRK4 p = 1 10.0 | 7.3, with a PML 25.9 | 16.1, p = 4
// with a PML 178 | 111; right-hand side p = 1 with a PML 25.2 | 16.7.  At 94 tiles 9.9 | 9.9
// and 178 | 223.
//
// FP32 right-hand sides: eight threads per column instead of four while their CTAs run side
// by side, at p = 3 up to one tile per SM, at p = 4 up to two (us, four | eight: p = 3 41 tiles
// 8.8 | 8.2, 137 tiles 10.6 | 9.1, 375 tiles 10.9 | 15.5; p = 4 41 tiles 13.0 | 10.9, 137 tiles
// 16.9 | 14.9, 274 tiles 18.7 | 16.7, 375 tiles 19.0 | 25.4).
// FP32 leapfrog at p = 4, without a layer as the right-hand side (137 tiles 17.5 | 13.4, 274
// tiles 18.5 | 14.5, 375 tiles 16.9 | 23.0), with one up to one tile per pair of SMs (41
// tiles 15.2 | 14.1, 94 tiles 18.2 | 19.1).
// FP32 at p = 5, penalty and right-hand side up to one tile per pair of SMs, the penalty on
// rows without a bulk copy up to one per SM: 255 registers per thread instead of 128, and all
// gathers in flight at once (penalty 41 tiles 27.5 | 20.7, 94 tiles 31.6 | 33.4, 137 tiles without
// a bulk copy 41.7 | 35.2; right-hand side with a PML 41 tiles 25.1 | 23.2, 137 tiles 29.2 |
// 28.9).  (The code exceeds the instruction cache, and from one tile per pair on the two SMs of
// a pair share the way it comes.)
constexpr int64_t kSMs = 152, kClusterTiles = kSMs / 4, kHalfTiles = kSMs / 2;

template <int MODE>
int launch_mode(const StageParams& prm, cudaStream_t st) {
    const int64_t C = prm.K_active * prm.S;   // columns updated
    if (C <= 0) return DGM_OK;
    const int64_t tiles = (C + 31) / 32;
    StageParams q = prm;
    q.dt_f = float(prm.dt);
    q.a_f = float(prm.a);
    q.b_f = float(prm.b);
    const bool i32 = !q.force_index64 && fits_32bit(q);
    const bool layer = q.pml != nullptr && q.npml > 0;
    constexpr bool kLF = MODE == MODE_LF_E || MODE == MODE_LF_H;
    if (q.hs != nullptr) {   // interior penalty
        if constexpr (kDefault && !kMX && !kLF) {
            if constexpr (sizeof(Real) == 4 && kP == 5) {
                if (i32 && tiles <= (tile_map(q) < 0 ? kSMs : kSMs / 2))
                    return launch_shape<32, 8, MODE, uint32_t, true, false, 1>(q, C, st);
            }
            return i32 ? launch_ix<MODE, uint32_t, true, false>(q, C, st) : launch_ix<MODE, int64_t, true, false>(q, C, st);
        } else {
            return DGM_EUNSUP;
        }
    }
    if constexpr (sizeof(Real) == 8 && !kMX) {
        if constexpr (MODE != MODE_RHS) {
            if (i32 && tiles <= kClusterTiles) return launch_shape<32, 8, MODE, uint32_t, false, true, 1, 8>(q, C, st);
        }
        if constexpr (!kLF) {
            if (i32 && tiles <= kHalfTiles) return launch_shape<16, 8, MODE, uint32_t, false, true, 1>(q, C, st);
        }
    }
    if constexpr (sizeof(Real) == 4 && !kMX && MODE == MODE_RHS && kP >= 3) {
        constexpr int64_t kTiles = kP == 3 ? kSMs : kP == 4 ? 2 * kSMs : kSMs / 2;
        constexpr int kMinB = kP == 5 ? 1 : 2;
        if (i32 && tiles <= kTiles)
            return layer ? launch_shape<32, 8, MODE, uint32_t, false, true, kMinB>(q, C, st)
                         : launch_shape<32, 8, MODE, uint32_t, false, false, kMinB>(q, C, st);
    }
    if constexpr (sizeof(Real) == 4 && !kMX && kLF && kP == 4) {
        if (i32 && !layer && tiles <= 2 * kSMs) return launch_shape<32, 8, MODE, uint32_t, false, false, 2>(q, C, st);
        if (i32 && layer && tiles <= kSMs / 2) return launch_shape<32, 8, MODE, uint32_t, false, true, 2>(q, C, st);
    }
    // (64-bit indices: the PML instantiation serves plans without a layer too)
    if (!i32) return launch_ix<MODE, int64_t, false, !kMX>(q, C, st);
    if constexpr (!kMX) {
        if (layer) return launch_ix<MODE, uint32_t, false, true>(q, C, st);
    }
    return launch_ix<MODE, uint32_t, false, false>(q, C, st);
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
