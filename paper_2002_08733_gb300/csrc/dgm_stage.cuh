// Fused DG right-hand-side / stage-update kernel (SIMT, FP64 or FP32).
//
// One CTA owns a tile of TE consecutive columns (column = element * S +
// source) and evaluates, for each of them, the whole semi-discrete right-hand
// side of Secs. III-IV in the strong form
//
//   d u_E/dt = B_eps [ s_T curl_ref(u_H) + sum_f R_f^T g_E,f - w_src g(t) ]
//              - A^T eta A^-T u_E - p / eps
//   d u_H/dt = B_mu  [-s_T curl_ref(u_E) + sum_f R_f^T g_H,f ]
//              - A^T eta A^-T u_H - q / mu
//   d p/dt   = -A^T Sigma A^-T p + eps A^T xi A^-T u_E   (likewise q)
//
// where u are covariant modal coefficients (Eq. (mapped_eh)),
// curl_ref uses the geometry-free derivative matrices S_a (Eq.
// (matrix_free_curl); the Piola map, Eq. (piola_transf), leaves only the
// orientation sign s_T = sign det A), B = (A^T A) / (material |det A|) is the
// inverse of the at-most 3x3 block mass matrix (Sec. II), R_f are the
// geometry-free trace matrices onto face f, and g_f = 2|F| A^-1 flux_f are the
// face-mode coefficients of the numerical flux pulled back to the element:
//   flux_E = c_E n x dH - b_E n x (n x dE),  flux_H = c_H n x dE + b_H n x (n x dH)
// with dX = X+ - X- the jump of the physical traces (X = A^-T x_ref per side),
// central (c = 1/2, b = 0, Eqs. (uwc)/(cwc)) or upwind coefficients, and the
// PEC ghost state e+ = -e-, h+ = h- on boundary faces.  The kernel evaluates
// g in the element's reference frame (face_constants_ref), where the pull-back
// cancels the own side's A^-T and, on the three axis faces, leaves the flux
// two components.
//
// Phases (separated by __syncthreads):
//   1 load the tile's coefficients, element constants and the precomputed
//     face constants (neighbour map, flux coefficients; face_consts_kernel)
//     into shared memory
//   2 own traces (4 faces x 6 components) from shared memory, neighbour traces
//     from global memory (the neighbour's coefficients are usually L2 hits)
//   3 numerical flux per (face, face mode) in the reference frame
//   4 right-hand side per component: volume curl + lift (+ source)
//   5 3x3 mass-block inverse, PML terms, and the stage update
// The reference operators are straight-line code with literal coefficients
// (generated at build time, dgm_refgen.cpp) that visits only the non-zero
// entries: S_a[l][m] = 0 unless deg(l) < deg(m), R_f[m][l] = 0 unless
// deg(m) <= deg(l) (hierarchical orthonormal bases), and many more entries
// vanish exactly for the collapsed basis (e.g. on the face x = 0 each mode
// has a single face mode).
#pragma once

#include <cstdint>

#include "dgm_internal.h"
#include "dgm_ops_gen.cuh"
#include "dgm_bulk.cuh"
#include "dgm_tc.cuh"

namespace dgm {

// Tile visited by this CTA.  With G > 1 groups CTAs b = 0, 1, 2, ... take tiles
// from G nearly equal segments in turn (the first n % G hold one tile more), so that
// tiles far apart in the column numbering run at the same time: meshes whose
// neighbours are numbered in G blocks (a Kuhn grid numbered type by type has
// its face neighbours in other type blocks) then find their neighbours'
// coefficients in L1 and L2.  Any order gives the same results.
__device__ __forceinline__ unsigned tile_index(int groups) {
    const unsigned b = blockIdx.x, n = gridDim.x;
    if (groups <= 1) return b;
    const unsigned g = unsigned(groups), seg = b % g, rest = n % g;
    return seg * (n / g) + (seg < rest ? seg : rest) + b / g;
}

// offset of the first mode of total degree d (3-D) and (2-D)
__host__ __device__ constexpr int off3(int d) { return d <= 0 ? 0 : nmodes(d - 1); }
__host__ __device__ constexpr int off2(int d) { return d <= 0 ? 0 : nfmodes(d - 1); }

constexpr int FG = 18;   // face constants per (face, column)
enum FaceConst {
    FC_N = 0,     // unit outward normal (3)
    FC_AITN = 3,  // neighbour A^-T (9), own A^-T on PEC faces
    FC_CE = 12, FC_BE = 13, FC_CH = 14, FC_BH = 15,
    FC_TWOF = 16, // 2 |F|
    FC_BND = 17   // 1 on a PEC face
};
constexpr int EG = 16;   // element constants per column (same slots as G_*)
constexpr int NBS = 4;   // neighbour codes per column staged in shared memory

// Face constants of the stage kernel, whose flux works in the element's
// reference frame (see face_constants_ref), per (face, column).
constexpr int FGR = 15;
enum FaceConstRef {
    FR_Q = 0,     // Q = A^T A_n^-T (9, row major): neighbour reference components -> own
    FR_NAE = 9,   // -alpha_E: -1 on an interior face, -2 on a PEC face (e+ = -e-)
    FR_NAH = 10,  // -alpha_H: -1 on an interior face, 0 on a PEC face (h+ = h-),
                  // -2 on an incident face (h+ = -h-; there alpha_E = 0)
    FR_CE = 11,   // s_T c_E
    FR_BE = 12,   // b_E / (|det A| |A^-T m_f|)
    FR_CH = 13,   // s_T c_H
    FR_BH = 14    // b_H / (|det A| |A^-T m_f|)
};
constexpr int GM = 6;    // metric A^T A per column: entries 00, 01, 02, 11, 12, 22

template <int P, typename R, int TE, bool TC = false>
__host__ __device__ constexpr size_t stage_smem_bytes() {
    // + an mbarrier (phase-1 bulk copies; the tensor-core variant's MMAs) and the
    // tensor-memory base (the operator image lives in the neighbour-trace array,
    // dead after phase 3)
    return sizeof(R) * size_t(TE) *
               (6 * nmodes(P) + 48 * nfmodes(P) + 4 * FGR + EG + GM + NBS) +
           size_t(32);
}

// Reference operators: straight-line code with literal coefficients generated
// at build time from the library's own reference matrices (dgm_refgen.cpp),
// visiting only the entries that are not zero.
template <int P, typename R, int F>
__device__ __forceinline__ void trace_face(const R (&v)[nmodes(P)], R (&acc)[nfmodes(P)]) {
    TraceOp<P, F>::template apply<R>(v, acc);
}

template <int P, typename R>
__device__ __forceinline__ void trace_any(int f, const R (&v)[nmodes(P)], R (&acc)[nfmodes(P)]) {
    switch (f) {
        case 0: trace_face<P, R, 0>(v, acc); break;
        case 1: trace_face<P, R, 1>(v, acc); break;
        case 2: trace_face<P, R, 2>(v, acc); break;
        default: trace_face<P, R, 3>(v, acc); break;
    }
}

template <typename R>
__device__ __forceinline__ void cross3(const R a[3], const R b[3], R o[3]) {
    o[0] = a[1] * b[2] - a[2] * b[1];
    o[1] = a[2] * b[0] - a[0] * b[2];
    o[2] = a[0] * b[1] - a[1] * b[0];
}

// source time function g(t) = sin(2 pi f0 (t - t0)) exp(-(t - t0)^2 / (2 s^2)), s = 1/(2 pi bw)
__device__ __forceinline__ double source_time(double t, double f0, double bw, double t0) {
    const double twopi = 6.283185307179586476925286766559;
    const double s = 1.0 / (twopi * bw);
    const double tau = t - t0;
    return sin(twopi * f0 * tau) * exp(-tau * tau / (2.0 * s * s));
}

// Face constants of face f of one element for the physical-frame flux (the
// adjoint kernel's; the stage kernel uses face_constants_ref), written to
// fc[k * TE]: unit outward normal, the neighbour's A^-T (own on a PEC face),
// flux coefficients, 2|F|, PEC flag.  2|F| n = |det A| A^-T m_f with m_f = 2|F_hat| n_hat of the
// reference face: (1,1,1), (-1,0,0), (0,-1,0), (0,0,-1).  The neighbour's A^-T
// and impedance come from the per-face neighbour table (own values on a
// boundary face), so every input is one coalesced load.
template <typename R, int TE>
__device__ __forceinline__ void face_constants_tab(int f, const R (&ait)[9], R det, R epsm, R mum,
                                                   bool has_nbr, const R (&aitn)[9], R zn,
                                                   int upwind, R* fc) {
    const R m0 = R(f == 0 ? 1 : (f == 1 ? -1 : 0));
    const R m1 = R(f == 0 ? 1 : (f == 2 ? -1 : 0));
    const R m2 = R(f == 0 ? 1 : (f == 3 ? -1 : 0));
    R vn[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) vn[r] = ait[3 * r + 0] * m0 + ait[3 * r + 1] * m1 + ait[3 * r + 2] * m2;
    const R fs = sqrt(vn[0] * vn[0] + vn[1] * vn[1] + vn[2] * vn[2]);
#pragma unroll
    for (int r = 0; r < 3; ++r) fc[(FC_N + r) * TE] = vn[r] / fs;
    fc[FC_TWOF * TE] = fabs(det) * fs;
    const R zm = sqrt(mum / epsm);
    const R zp = has_nbr ? zn : zm;
#pragma unroll
    for (int k = 0; k < 9; ++k) fc[(FC_AITN + k) * TE] = aitn[k];
    fc[FC_BND * TE] = has_nbr ? R(0) : R(1);
    if (upwind) {
        const R ym = R(1) / zm, yp = R(1) / zp;
        fc[FC_CE * TE] = zp / (zm + zp);
        fc[FC_BE * TE] = R(1) / (zm + zp);
        fc[FC_CH * TE] = yp / (ym + yp);
        fc[FC_BH * TE] = R(1) / (ym + yp);
    } else {
        fc[FC_CE * TE] = R(0.5);
        fc[FC_BE * TE] = R(0);
        fc[FC_CH * TE] = R(0.5);
        fc[FC_BH * TE] = R(0);
    }
}

// Face constants of the reference-frame flux of face f (written to fc[k * TE],
// TE the row stride) and, when gm is not null, the element's metric A^T A
// (gm[k * TE]).
//
// With M = A^-T, the reference traces x of both sides, Q = M^-1 M_n = A^T A_n^-T
// and the reference jump dx = Q x+ - alpha x- (alpha: 1, or the PEC ghost
// state), the physical jump is M dx.  The identity (M a) x (M b) =
// det M M^-T (a x b) and n = M m_f / |M m_f| give
//   A^-1 (n x M y)         = (det M / |M m_f|) m_f x y,
//   A^-1 (n x (n x M y))   = (det M / |M m_f|)^2 m_f x (A^T A (m_f x y)),
// so the pulled-back fluxes g = 2|F| A^-1 flux, 2|F| = |det A| |M m_f|, are
//   g_E =  s_T c_E m_f x dh - b_E / (|det A| |M m_f|) m_f x (A^T A (m_f x de))
//   g_H = -s_T c_H m_f x de - b_H / (|det A| |M m_f|) m_f x (A^T A (m_f x dh))
// with no transformation of the traces on the element's own side.  On the
// faces x = 0, y = 0, z = 0 (m_f = -e_a) the cross products only permute
// components, component a of g vanishes, and component a of the own trace
// is not needed.
// incident: a boundary face through which an incident field enters (ghost state
// e+ = e- + 2 E_inc, h+ = -h-, Z+ = Z-; the E_inc part is added by flux_face).
template <typename R>
__device__ __forceinline__ void face_constants_ref(int f, const R (&ait)[9], R det, R epsm, R mum,
                                                   bool has_nbr, const R (&aitn)[9], R zn,
                                                   int upwind, R* fc, R* gm, bool incident,
                                                   int64_t TE) {
    // A^T = det A adj(A^-T), row major
    R at[9];
    at[0] = ait[4] * ait[8] - ait[5] * ait[7];
    at[1] = ait[2] * ait[7] - ait[1] * ait[8];
    at[2] = ait[1] * ait[5] - ait[2] * ait[4];
    at[3] = ait[5] * ait[6] - ait[3] * ait[8];
    at[4] = ait[0] * ait[8] - ait[2] * ait[6];
    at[5] = ait[2] * ait[3] - ait[0] * ait[5];
    at[6] = ait[3] * ait[7] - ait[4] * ait[6];
    at[7] = ait[1] * ait[6] - ait[0] * ait[7];
    at[8] = ait[0] * ait[4] - ait[1] * ait[3];
#pragma unroll
    for (int k = 0; k < 9; ++k) at[k] *= det;
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
        for (int k = 0; k < 3; ++k)
            fc[(FR_Q + 3 * j + k) * TE] =
                at[3 * j] * aitn[k] + at[3 * j + 1] * aitn[3 + k] + at[3 * j + 2] * aitn[6 + k];
    const R m0 = R(f == 0 ? 1 : (f == 1 ? -1 : 0));
    const R m1 = R(f == 0 ? 1 : (f == 2 ? -1 : 0));
    const R m2 = R(f == 0 ? 1 : (f == 3 ? -1 : 0));
    R vn[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) vn[r] = ait[3 * r + 0] * m0 + ait[3 * r + 1] * m1 + ait[3 * r + 2] * m2;
    const R fs = sqrt(vn[0] * vn[0] + vn[1] * vn[1] + vn[2] * vn[2]);
    const R st = det < R(0) ? R(-1) : R(1);
    const R kb = R(1) / (fabs(det) * fs);
    const R zm = sqrt(mum / epsm);
    const R zp = has_nbr ? zn : zm;
    R ce = R(0.5), be = R(0), ch = R(0.5), bh = R(0);
    if (upwind) {
        const R ym = R(1) / zm, yp = R(1) / zp;
        ce = zp / (zm + zp);
        be = R(1) / (zm + zp);
        ch = yp / (ym + yp);
        bh = R(1) / (ym + yp);
    }
    fc[FR_NAE * TE] = has_nbr ? R(-1) : (incident ? R(0) : R(-2));
    fc[FR_NAH * TE] = has_nbr ? R(-1) : (incident ? R(-2) : R(0));
    fc[FR_CE * TE] = st * ce;
    fc[FR_BE * TE] = kb * be;
    fc[FR_CH * TE] = st * ch;
    fc[FR_BH * TE] = kb * bh;
    if (gm != nullptr) {
        gm[0 * TE] = at[0] * at[0] + at[1] * at[1] + at[2] * at[2];
        gm[1 * TE] = at[0] * at[3] + at[1] * at[4] + at[2] * at[5];
        gm[2 * TE] = at[0] * at[6] + at[1] * at[7] + at[2] * at[8];
        gm[3 * TE] = at[3] * at[3] + at[4] * at[4] + at[5] * at[5];
        gm[4 * TE] = at[3] * at[6] + at[4] * at[7] + at[5] * at[8];
        gm[5 * TE] = at[6] * at[6] + at[7] * at[7] + at[8] * at[8];
    }
}

// The stage kernel's face constants, computed once per plan (again when the
// materials or the boundary codes change) for every element, stride K, in the
// kernel's precision: rows f FGR + k, then the metric A^T A.  The same function and inputs as a computation inside the
// stage kernel, so the same bits.
static_assert(4 * FGR + GM == FC_ROWS, "precomputed face-constant rows");
static_assert(EG == TM_ROWS_EG && FGR == TM_ROWS_FC && GM == TM_ROWS_GM, "bulk-copy boxes match the shared-memory rows");
template <typename R>
__global__ void face_consts_kernel(const StageParams prm, R* __restrict__ out) {
    const int64_t K = prm.K;
    const int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (e >= K) return;
    const R* gr = static_cast<const R*>(prm.geo_r);
    R ait[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) ait[k] = gr[int64_t(G_AIT + k) * K + e];
    const R det = gr[int64_t(G_DET) * K + e];
    const R epsm = gr[int64_t(G_EPS) * K + e];
    const R mum = gr[int64_t(G_MU) * K + e];
    for (int f = 0; f < 4; ++f) {
        const R* fn = static_cast<const R*>(prm.fnb_r) + int64_t(f * FNB_COUNT) * K + e;
        const int32_t code = prm.nbr[int64_t(f) * K + e];
        R aitn[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) aitn[k] = fn[int64_t(FNB_AIT + k) * K];
        const R zn = fn[int64_t(FNB_Z) * K];
        face_constants_ref<R>(f, ait, det, epsm, mum, code >= 0 && (code >> 2) < K, aitn, zn, prm.upwind,
                              out + int64_t(f * FGR) * K + e, f == 0 ? out + int64_t(4 * FGR) * K + e : nullptr,
                              code <= -2 && prm.inc != nullptr, K);
    }
}

// index of (i, j) in the six stored entries of a symmetric 3x3 matrix
__host__ __device__ constexpr int sym3(int i, int j) {
    return i > j ? sym3(j, i) : (i == 0 ? j : (i == 1 ? 2 + j : 5));
}

// Numerical flux of modes [m0, m1) of face F (compile time) in the reference
// frame (face_constants_ref): reads both sides' reference traces, overwrites
// the own traces with the pulled-back fluxes g.  On an axis face only the two
// non-zero components of g are written.  FULL: the own trace has all three
// components and the physical jumps M dx are stored for the adjoint.
template <int F, int NF, typename R, int TE, int MODE, typename IX>
__device__ __forceinline__ void flux_face(int m0, int m1, int c, R* trO, const R* trN,
                                          const R* fg, const R* gm, const R* eg, R* jumps,
                                          IX C, IX col, bool active, int32_t code,
                                          const void* incp) {
    constexpr bool FULL = (MODE == MODE_RAW);
    constexpr int A = F == 0 ? -1 : F - 1;       // axis of m_f = -e_A
    constexpr int B = F % 3, CC = (F + 1) % 3;   // the other two axes, (A, B, CC) cyclic
    const R* d = fg + F * FGR * TE + c;
    R q[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) q[k] = (FULL || k / 3 != A) ? d[(FR_Q + k) * TE] : R(0);
    const R nae = d[FR_NAE * TE], nah = d[FR_NAH * TE];
    const R cE = d[FR_CE * TE], bE = d[FR_BE * TE], cH = d[FR_CH * TE], bH = d[FR_BH * TE];
    // A^T A, entries 00, 01, 02, 11, 12, 22 (named, so that they stay in registers)
    const R g00 = gm[0 * TE + c], g01 = gm[1 * TE + c], g02 = gm[2 * TE + c];
    const R g11 = gm[3 * TE + c], g12 = gm[4 * TE + c], g22 = gm[5 * TE + c];
    R ait[9];
    if (FULL) {
#pragma unroll
        for (int k = 0; k < 9; ++k) ait[k] = eg[(G_AIT + k) * TE + c];
    }
    // entries of A^T A used on an axis face: (CC, B), (CC, CC), (B, B)
    auto gsym = [&](int i, int j) -> R {
        const int k = sym3(i, j);
        return k == 0 ? g00 : k == 1 ? g01 : k == 2 ? g02 : k == 3 ? g11 : k == 4 ? g12 : g22;
    };
    const R gcb = gsym(CC, B), gcc = gsym(CC, CC), gbb = gsym(B, B);
    const R kEcb = bE * gcb, kEcc = bE * gcc, kEbb = bE * gbb;
    const R kHcb = bH * gcb, kHcc = bH * gcc, kHbb = bH * gbb;
    // incident face (e+ = e- + 2 E_inc): the E jump is the incident term alone
    const R* inc = (code <= -2 && incp != nullptr && active)
                       ? static_cast<const R*>(incp) + IX(-code - 2) * NF * 3
                       : nullptr;
    // not unrolled: four copies of an unrolled loop (one per face) cost more in
    // instruction fetch than the loop overhead they save
#pragma unroll 1
    for (int m = m0; m < m1; ++m) {
        R* own = trO + (F * 6 * NF + m) * TE + c;
        const R* nbt = trN + (F * 6 * NF + m) * TE + c;
        R de[3] = {0, 0, 0}, dh[3] = {0, 0, 0};   // reference-frame jumps
        {
            R tp[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) tp[k] = nbt[k * NF * TE];
#pragma unroll
            for (int r = 0; r < 3; ++r)
                if (FULL || r != A)
                    de[r] = q[3 * r] * tp[0] + q[3 * r + 1] * tp[1] + q[3 * r + 2] * tp[2] +
                            nae * own[r * NF * TE];
        }
        if (inc != nullptr) {
#pragma unroll
            for (int r = 0; r < 3; ++r)
                if (FULL || r != A) de[r] += inc[m * 3 + r];
        }
        {
            R tp[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) tp[k] = nbt[(3 + k) * NF * TE];
#pragma unroll
            for (int r = 0; r < 3; ++r)
                if (FULL || r != A)
                    dh[r] = q[3 * r] * tp[0] + q[3 * r + 1] * tp[1] + q[3 * r + 2] * tp[2] +
                            nah * own[(3 + r) * NF * TE];
        }
        if (FULL && active) {
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                jumps[IX((F * 6 + r) * NF + m) * C + col] =
                    ait[3 * r] * de[0] + ait[3 * r + 1] * de[1] + ait[3 * r + 2] * de[2];
                jumps[IX((F * 6 + 3 + r) * NF + m) * C + col] =
                    ait[3 * r] * dh[0] + ait[3 * r + 1] * dh[1] + ait[3 * r + 2] * dh[2];
            }
        }
        if (F == 0) {
            // m_f = (1, 1, 1): m x y = (y2 - y1, y0 - y2, y1 - y0)
            const R we[3] = {de[2] - de[1], de[0] - de[2], de[1] - de[0]};
            const R wh[3] = {dh[2] - dh[1], dh[0] - dh[2], dh[1] - dh[0]};
            {   // z = b_E A^T A w_e
                const R z0 = bE * (g00 * we[0] + g01 * we[1] + g02 * we[2]);
                const R z1 = bE * (g01 * we[0] + g11 * we[1] + g12 * we[2]);
                const R z2 = bE * (g02 * we[0] + g12 * we[1] + g22 * we[2]);
                own[0 * NF * TE] = cE * wh[0] - (z2 - z1);
                own[1 * NF * TE] = cE * wh[1] - (z0 - z2);
                own[2 * NF * TE] = cE * wh[2] - (z1 - z0);
            }
            {   // z = b_H A^T A w_h
                const R z0 = bH * (g00 * wh[0] + g01 * wh[1] + g02 * wh[2]);
                const R z1 = bH * (g01 * wh[0] + g11 * wh[1] + g12 * wh[2]);
                const R z2 = bH * (g02 * wh[0] + g12 * wh[1] + g22 * wh[2]);
                own[3 * NF * TE] = -cH * we[0] - (z2 - z1);
                own[4 * NF * TE] = -cH * we[1] - (z0 - z2);
                own[5 * NF * TE] = -cH * we[2] - (z1 - z0);
            }
        } else {
            // m_f = -e_A: (m x y)_A = 0, (m x y)_B = y_CC, (m x y)_CC = -y_B
            {
                own[B * NF * TE] = cE * dh[CC] - kEcb * de[CC] + kEcc * de[B];
                own[CC * NF * TE] = -cE * dh[B] + kEbb * de[CC] - kEcb * de[B];
            }
            {
                own[(3 + B) * NF * TE] = -cH * de[CC] - kHcb * dh[CC] + kHcc * dh[B];
                own[(3 + CC) * NF * TE] = cH * de[B] + kHbb * dh[CC] - kHcb * dh[B];
            }
        }
    }
}

// Right-hand side rows [LO, HI) of component `comp` (before the mass inverse):
// volume curl of the other field plus the lift of the pulled-back fluxes.
// FC: components held per face and field pair, 6 (us: both fields) or 3 (us: the
// other field alone, trO: this field's fluxes alone).
template <int P, typename R, int TE, int LO, int HI, int FC = 6>
__device__ __forceinline__ void rhs_rows(int comp, int c, const R* us, const R* trO, R sgn,
                                         R (&acc)[nmodes(P)]) {
    constexpr int N = nmodes(P);
    constexpr int NF = nfmodes(P);
#pragma unroll
    for (int l = 0; l < N; ++l) acc[l] = R(0);
    // curl_x = d_y v_z - d_z v_y, curl_y = d_z v_x - d_x v_z, curl_z = d_x v_y - d_y v_x,
    // of H for the E equation (+s_T) and of E for the H equation (-s_T)
    const int j = comp % 3;
    const int srcf = FC == 6 && comp < 3 ? 3 : 0;
    const R sg = comp < 3 ? sgn : -sgn;
    // The pulled-back flux of face a + 1 (normal -e_a) has no component a, so
    // component j lifts the fluxes of the three other faces only.
    const R* base = us + c;
    const R* g = trO + (FC == 6 ? comp : j) * NF * TE + c;    // face f of this component: g + f * FC * NF * TE
    switch (j) {
        case 0:
            DerivOp<P, 1>::template apply<R, LO, HI>(base + (srcf + 2) * N * TE, TE, R(1), acc);
            DerivOp<P, 2>::template apply<R, LO, HI>(base + (srcf + 1) * N * TE, TE, R(-1), acc);
            break;
        case 1:
            DerivOp<P, 2>::template apply<R, LO, HI>(base + (srcf + 0) * N * TE, TE, R(1), acc);
            DerivOp<P, 0>::template apply<R, LO, HI>(base + (srcf + 2) * N * TE, TE, R(-1), acc);
            break;
        default:
            DerivOp<P, 0>::template apply<R, LO, HI>(base + (srcf + 1) * N * TE, TE, R(1), acc);
            DerivOp<P, 1>::template apply<R, LO, HI>(base + (srcf + 0) * N * TE, TE, R(-1), acc);
            break;
    }
#pragma unroll
    for (int l = LO; l < HI; ++l) acc[l] *= sg;
    // one copy of each lift, skipped by a branch that is uniform over the
    // group (lifts inside the cases above would triple the code of this phase)
    LiftOp<P, 0>::template apply<R, LO, HI>(g + 0 * FC * NF * TE, TE, acc);
    if (j != 0) LiftOp<P, 1>::template apply<R, LO, HI>(g + 1 * FC * NF * TE, TE, acc);
    if (j != 1) LiftOp<P, 2>::template apply<R, LO, HI>(g + 2 * FC * NF * TE, TE, acc);
    if (j != 2) LiftOp<P, 3>::template apply<R, LO, HI>(g + 3 * FC * NF * TE, TE, acc);
}

template <int P, typename R, int TE, int NPART, int FC = 6>
__device__ __forceinline__ void rhs_part(int part, int comp, int c, const R* us, const R* trO,
                                         R sgn, R (&acc)[nmodes(P)]) {
    constexpr int N = nmodes(P);
    static_assert(NPART >= 1 && NPART <= 4, "row partition");
    switch (part) {
        case 0: rhs_rows<P, R, TE, 0, (NPART == 1 ? N : N / NPART), FC>(comp, c, us, trO, sgn, acc); break;
        case 1: rhs_rows<P, R, TE, N / NPART, (NPART == 2 ? N : 2 * N / NPART), FC>(comp, c, us, trO, sgn, acc); break;
        case 2: rhs_rows<P, R, TE, 2 * N / NPART, (NPART == 3 ? N : 3 * N / NPART), FC>(comp, c, us, trO, sgn, acc); break;
        default: rhs_rows<P, R, TE, 3 * N / NPART, N, FC>(comp, c, us, trO, sgn, acc); break;
    }
}

// Two resident CTAs per SM where the registers allow it: FP32 up to p = 3
// (<= 85 registers at 384 threads), FP64 at 192 threads (<= 170 registers).
// IX: type of the element/column/row index arithmetic.  uint32_t when every
// index of the plan fits (the launcher checks), which saves the 64-bit
// address arithmetic that is a large part of this kernel's integer work;
// int64_t otherwise.
//
// TC: tensor-core variant (FP32, p = 2, 3, LSRK4 stages, 64 columns per CTA):
// the volume curl and the lift (phase 4) run as TF32 split products on the
// tensor cores (dgm_tc.cuh, TcShape), with tensor-memory row (field, column);
// phase 5 reads the pre-mass right-hand side from tensor memory.  The other
// phases are shared with the SIMT kernel.
// PML: phase 5 has the layer's terms.  An instantiation without them serves the plans
// without a layer, whose phase 5 the layer's chunked rows slow down (FP32 LSRK4 stage, us,
// 16^3 grid, without the terms | with: p = 4 53.6 | 57.7; p = 5 135 | 150).
template <int P, typename R, int TE, int NT, int MODE, typename IX = int64_t, bool TC = false, bool PML = true>
__global__ void __launch_bounds__(NT, TC ? 1 : ((sizeof(R) == 8 || P <= 3) ? 2 : 1))
stage_kernel(const StageParams prm) {
    static_assert(MODE == MODE_LSRK || MODE == MODE_RAW, "LSRK4 stages and the adjoint's forward quantities");
    constexpr int N = nmodes(P);
    constexpr int NF = nfmodes(P);
    constexpr int NG = NT / TE;                         // column groups working side by side
    constexpr int NPART = NG >= 24 ? 4 : (NG >= 12 ? 2 : 1);  // row parts of phases 4 and 5
    extern __shared__ __align__(16) unsigned char smem_raw[];
    R* us = reinterpret_cast<R*>(smem_raw);      // [6N][TE]
    R* trO = us + 6 * N * TE;                    // [4][6][NF][TE]  own traces -> g
    R* trN = trO + 24 * NF * TE;                 // [4][6][NF][TE]  nbr traces -> rhs [6][N][TE]
    R* fg = trN + 24 * NF * TE;                  // [4][FGR][TE]
    R* eg = fg + 4 * FGR * TE;                  // [EG][TE]
    R* gm = eg + EG * TE;                        // [GM][TE] metric A^T A
    int32_t* nbs = reinterpret_cast<int32_t*>(gm + GM * TE);   // [NBS][TE] neighbour codes
    static_assert(!TC || (sizeof(R) == 4 && TE == 64 && MODE == MODE_LSRK &&
                          (NT / TE) % 2 == 0 && TcShape<P>::FITS),
                  "tensor-core variant: FP32, 64 columns, LSRK, even groups");
    // mbarrier (phase-1 bulk copies; tensor-core variant: its MMAs) and the
    // tensor-memory base address after the tables; the tensor-core variant's
    // operator image goes into the neighbour-trace array in phase 4
    uint64_t* tc_bar = reinterpret_cast<uint64_t*>(
        (reinterpret_cast<uintptr_t>(nbs + NBS * TE) + 7) & ~uintptr_t(7));
    uint32_t* tc_base = reinterpret_cast<uint32_t*>(tc_bar + 1);
    if constexpr (TC) {
        static_assert(TcShape<P>::B_BYTES <= int(sizeof(R)) * 24 * nfmodes(P) * TE,
                      "operator image fits in the neighbour-trace array");
        if (threadIdx.x == 0) tc::mbar_init(tc_bar, 1);
        if (threadIdx.x < 32) {
            tc::tmem_alloc(tc_base, TcShape<P>::TCOLS);
            tc::fence_before();
        }
    }

    const int c = threadIdx.x % TE;
    const int grp = threadIdx.x / TE;
    const IX K = prm.K;
    const int S = prm.S;
    const IX C = K * S;
    const IX col = IX(tile_index(prm.tile_groups)) * TE + c;
    // only the first K_active elements are updated; the others (halo copies of
    // another partition's elements) are read as neighbours
    const bool active = col < IX(prm.K_active) * IX(S);
    const IX e = active ? col / S : 0;
    const int s = active ? int(col - e * S) : 0;
    const R* u = static_cast<const R*>(prm.u);
    const R* gr = static_cast<const R*>(prm.geo_r);
    // stage coefficients in the kernel's precision: FP32 kernels read the FP32
    // copies, so that no conversion runs on the FP64 pipe
    auto coef = [&](double d, float f) { return sizeof(R) == 4 ? R(f) : R(d); };
    for (int r = grp; r < NBS; r += NG) nbs[r * TE + c] = active ? prm.nbr[IX(r) * K + e] : -1;   // neighbour codes

    // ---- phase 1: tile coefficients, element and face constants --------------
    // Every group loads rows of the tile: the coefficients, the element
    // constants, and the face constants and metric that the plan precomputed
    // (face_consts_kernel), each thread's loads in flight together before its
    // shared-memory stores; every group requests the neighbour coefficients of
    // its first two neighbour items and traces the first, so that the global
    // round trips of the tile and the gathers overlap each other and work.
    constexpr int NOWN = 12, NNBR = 24;                 // phase-2 items
    R vn[N];                                            // neighbour coefficients (phase 2)
    // neighbour item ni = (face ni / 6, component ni % 6): request the
    // neighbour's coefficients of that component given the face's code
    auto request_nbr = [&](int ni, int32_t code, R (&dst)[N]) {
        if (ni < NNBR && active && code >= 0 && (code >> 2) < K) {
            const IX ncol = IX(code >> 2) * S + s;
#pragma unroll
            for (int l = 0; l < N; ++l) dst[l] = u[IX((ni % 6) * N + l) * C + ncol];
        }
    };
    // neighbour item ni: the trace of the neighbour's coefficients v on its
    // face (code & 3) into trN (zeros without a neighbour)
    auto nbr_trace = [&](int ni, int32_t code, const R (&v)[N]) {
        if (ni < NNBR) {
            const int nf = ni / 6, ncomp = ni % 6;
            const bool has_nbr = code >= 0 && (code >> 2) < K;
            if (code >= 0 && (code >> 2) >= K) atomicOr(prm.status, ST_BAD_NEIGHBOUR);
            R acc[NF];
            if (has_nbr) {
                trace_any<P, R>(code & 3, v, acc);
            } else {
#pragma unroll
                for (int m = 0; m < NF; ++m) acc[m] = R(0);
            }
            R* dst = trN + ((nf * 6 + ncomp) * NF) * TE + c;
#pragma unroll
            for (int m = 0; m < NF; ++m) dst[m * TE] = acc[m];
        }
    };
    // neighbour codes of this group's items of rounds 0 and 1 (the staged
    // copies in nbs are not visible before the phase-1 barrier)
    const int32_t code0 = (grp < NNBR && active) ? prm.nbr[IX(grp / 6) * K + e] : -1;
    const int32_t code1 = (grp + NG < NNBR && active) ? prm.nbr[IX((grp + NG) / 6) * K + e] : -1;
    R vn1[N];                                           // round-1 neighbour coefficients
    // Tiled bulk copies where the plan has tensor maps for this tile (one column
    // per element, aligned rows; tm_u >= 0): thread 0 issues four copies (the
    // coefficients [6][N][TE], the element constants, the face constants, the
    // metric and A^T) onto an mbarrier and waits for them itself, with a time
    // limit, while every thread gathers and traces neighbour coefficients; the
    // phase-1 barrier then publishes the tile.  Columns past the end arrive as
    // zeros, which only inactive columns see.  Otherwise every thread loads
    // and stores its share of rows.
    constexpr bool BULK_OK = !TC && (TE * int(sizeof(R)) == 128 || (sizeof(R) == 4 && TE == 16));
    const bool bulk = BULK_OK && prm.tm_u >= 0 && (tc::smem_addr(smem_raw) & 127u) == 0;
    if (bulk) {
        constexpr uint32_t BYTES = uint32_t(sizeof(R)) * TE * (6 * N + EG + 4 * FGR + GM);
        // every box dimension within the copy's limit of 256, the byte count
        // within the mbarrier's transaction count (2^20 - 1)
        static_assert(!BULK_OK || (TE <= 256 && N <= 256 && BYTES < (1u << 20)), "bulk-copy boxes");
        if (threadIdx.x == 0) {
            tc::mbar_init(tc_bar, 1);
            bulk::arrive_expect_tx(tc_bar, BYTES);
            const char* tm = static_cast<const char*>(prm.tmaps);
            const int x = int(tile_index(prm.tile_groups)) * TE;
            bulk::load_3d(us, tm + prm.tm_u * TMAP_BYTES, x, 0, 0, tc_bar);
            bulk::load_2d(eg, tm + TM_GEO * TMAP_BYTES, x, 0, tc_bar);
            bulk::load_3d(fg, tm + TM_FC * TMAP_BYTES, x, 0, 0, tc_bar);
            bulk::load_2d(gm, tm + TM_GM * TMAP_BYTES, x, 4 * FGR, tc_bar);
        }
        request_nbr(grp, code0, vn);
        request_nbr(grp + NG, code1, vn1);
    } else {
        // rows q: [0, 6N) coefficients, then EG element constants, 4 FGR face
        // constants and GM metric rows
        constexpr int Q0 = 6 * N, Q1 = Q0 + EG, Q2 = Q1 + 4 * FGR, Q3 = Q2 + GM;
        constexpr int T1 = Q3;
        constexpr int UR = (T1 + NG - 1) / NG;          // rows per thread (at most)
        constexpr int BATCH = UR < 24 ? UR : 16;        // loads in flight per thread (one batch when it fits)
        const R* fcp = static_cast<const R*>(prm.fcp);
        auto load = [&](int q) -> R {
            if (q < Q0) return active ? u[IX(q) * C + col] : R(0);
            if (q < Q1) {
                const int k = q - Q0;
                return active ? gr[IX(k) * K + e] : R(k == G_DET || k == G_EPS || k == G_MU ? 1 : 0);
            }
            if (q < Q2) {
                const int f = (q - Q1) / FGR, k = (q - Q1) % FGR;
                return active ? fcp[IX(f * FGR + k) * K + e] : R(0);
            }
            return active ? fcp[IX(4 * FGR + q - Q2) * K + e] : R(0);
        };
        auto store = [&](int q, R v) {
            if (q < Q0) us[q * TE + c] = v;
            else if (q < Q1) eg[(q - Q0) * TE + c] = v;
            else if (q < Q2) fg[(q - Q1) * TE + c] = v;
            else gm[(q - Q2) * TE + c] = v;
        };
        R tmp[BATCH];
#pragma unroll
        for (int i0 = 0; i0 < UR; i0 += BATCH) {
#pragma unroll
            for (int i = 0; i < BATCH; ++i) {
                const int q = grp + (i0 + i) * NG;
                tmp[i] = (i0 + i < UR && q < T1) ? load(q) : R(0);
            }
            if (i0 == 0) request_nbr(grp, code0, vn);
#pragma unroll
            for (int i = 0; i < BATCH; ++i) {
                const int q = grp + (i0 + i) * NG;
                if (i0 + i < UR && q < T1) store(q, tmp[i]);
            }
        }
        request_nbr(grp + NG, code1, vn1);
    }
    // Round 0 of the neighbour traces before the phase-1 barrier: it needs only
    // registers and writes rows of trN that phase 1 does not touch, so its
    // gathers and arithmetic overlap the copies and the wait for the slowest
    // group.
    nbr_trace(grp, code0, vn);
#pragma unroll
    for (int l = 0; l < N; ++l) vn[l] = vn1[l];
    if (bulk) {
        bool ok = true;
        if (threadIdx.x == 0) ok = tc::mbar_wait(tc_bar, 0, 500000000ull);
        if (!__syncthreads_and(ok)) {
            // the copies did not complete in time: latch the status, give them a
            // second bounded wait (the shared memory stays this CTA's until its
            // last thread exits) and leave the tile untouched
            if (threadIdx.x == 0) {
                atomicOr(prm.status, int32_t(ST_TIMEOUT));
                tc::mbar_wait(tc_bar, 0, 500000000ull);
            }
            return;
        }
    } else {
        __syncthreads();
    }

    // ---- phase 2: traces ------------------------------------------------------
    // Neighbour traces: item (face, component), one per group and round; round
    // 0 ran in phase 1, and the coefficients of round rr + 1 are requested
    // before the arithmetic of round rr (those of round 1 in phase 1), so every
    // gather overlaps work.  Own traces: item (component, pair of faces),
    // sharing one load of the component's coefficients between two faces, in
    // the last rounds.
    {
        constexpr int ROUNDS = (NNBR + NG - 1) / NG;
        constexpr int OWN_ROUNDS = (NOWN + NG - 1) / NG;
        // unrolled so that handing the prefetched coefficients to the next
        // round is register renaming, not copies
#pragma unroll
        for (int rr = 0; rr < ROUNDS; ++rr) {
            const int ni = grp + rr * NG;
            R vnx[N];
            if (rr >= 1 && rr + 1 < ROUNDS && ni + NG < NNBR)
                request_nbr(ni + NG, nbs[((ni + NG) / 6) * TE + c], vnx);
            if (rr >= 1) nbr_trace(ni, ni < NNBR ? nbs[(ni / 6) * TE + c] : -1, vn);
            const int oi = grp + (rr - (ROUNDS - OWN_ROUNDS)) * NG;   // own item of this round
            if (rr >= ROUNDS - OWN_ROUNDS && oi < NOWN) {
                const int ocomp = oi % 6, fp = oi / 6;
                R v[N];
                R acc[NF];
#pragma unroll
                for (int l = 0; l < N; ++l) v[l] = us[(ocomp * N + l) * TE + c];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int f = 2 * fp + h;
                    // the flux on face a + 1 (normal -e_a) does not use component a
                    // of the own trace, except for the adjoint's physical jumps
                    if (MODE != MODE_RAW && f == ocomp % 3 + 1) continue;
                    trace_any<P, R>(f, v, acc);
                    R* dst = trO + ((f * 6 + ocomp) * NF) * TE + c;
#pragma unroll
                    for (int m = 0; m < NF; ++m) dst[m * TE] = acc[m];
                }
            }
            if (rr >= 1) {
#pragma unroll
                for (int l = 0; l < N; ++l) vn[l] = vnx[l];
            }
        }
    }
    __syncthreads();

    // ---- phase 3: numerical flux per (face, chunk of face modes) -------------
    // in the element's reference frame, one code path per face (the face of an
    // item is uniform over its warp-sized group).  Equal chunks per face,
    // although a mode of the slanted face 0 costs more than one of an axis face
    // (66 against 28 operations): chunks sized by that ratio measured slower
    // (more items, so more per-item setup, and no shorter phase).
    {
        constexpr int CHUNKS = NG >= 12 ? (NG / 4) : (NG == 8 ? 2 : 1);   // face-mode chunks per face
        R* jp = static_cast<R*>(prm.jumps);
        for (int it = grp; it < 4 * CHUNKS; it += NG) {
            const int f = it / CHUNKS;
            const int ch = it % CHUNKS;
            const int m0 = ch * NF / CHUNKS, m1 = (ch + 1) * NF / CHUNKS;
            const int32_t fcode = nbs[f * TE + c];
            switch (f) {
                case 0: flux_face<0, NF, R, TE, MODE, IX>(m0, m1, c, trO, trN, fg, gm, eg, jp, C, col, active, fcode, prm.inc); break;
                case 1: flux_face<1, NF, R, TE, MODE, IX>(m0, m1, c, trO, trN, fg, gm, eg, jp, C, col, active, fcode, prm.inc); break;
                case 2: flux_face<2, NF, R, TE, MODE, IX>(m0, m1, c, trO, trN, fg, gm, eg, jp, C, col, active, fcode, prm.inc); break;
                default: flux_face<3, NF, R, TE, MODE, IX>(m0, m1, c, trO, trN, fg, gm, eg, jp, C, col, active, fcode, prm.inc); break;
            }
        }
    }
    // Phase 5 works per (field, row part): one item updates the three
    // components of a field on its rows, so that the 3x3 mass block is applied
    // once per row and each right-hand-side value is read once.  The LSRK
    // residual rows of that item are requested as soon as the thread's flux
    // item is done, so that their latency overlaps the wait at the phase-3
    // barrier and the phase-4 arithmetic.
    constexpr int NP5 = (NG / 2 < N ? NG / 2 : N) > 0 ? (NG / 2 < N ? NG / 2 : N) : 1;   // row parts per field
    constexpr int RP5 = (N + NP5 - 1) / NP5;          // rows per part (at most)
    constexpr bool P5_EVEN = (N % NP5) == 0;          // every part has exactly RP5 rows
    constexpr bool PREFETCH_RES = (MODE == MODE_LSRK);
    R resv[PREFETCH_RES ? 3 : 1][PREFETCH_RES ? RP5 : 1];
    if (PREFETCH_RES && grp < 2 * NP5) {
        const int fb = (grp / NP5) * 3, part = grp % NP5;
        const int lo = part * N / NP5, hi = (part + 1) * N / NP5;
        const bool load = active && coef(prm.a, prm.a_f) != R(0);
        const R* res = static_cast<const R*>(prm.res);
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int i = 0; i < RP5; ++i)
                resv[k][i] = (load && (P5_EVEN || lo + i < hi)) ? res[IX((fb + k) * N + lo + i) * C + col] : R(0);
    }
    __syncthreads();

    // ---- phase 4: volume curl + lift per (component, row part) -----------------
    R* rh = trN;   // [6][N][TE], the neighbour traces are dead now
    // tensor-core variant: per row (field F, column c) stage A_swap = +-s_T times
    // the other field and the pulled-back fluxes A_g of F's three components in
    // tensor memory (TF32 hi/lo), then one thread issues the MMAs
    if constexpr (TC) {
        using TS = TcShape<P>;
        tc::fence_after();   // the allocation's address, written before the phase-1 barrier
        const uint32_t tb = *tc_base;
        // the operator image, the same for every CTA (an L2 hit after the first
        // ones), into the neighbour-trace array (dead since phase 3)
        unsigned char* tc_b = reinterpret_cast<unsigned char*>(trN);
        {
            const uint4* src = static_cast<const uint4*>(prm.tc_b);
            uint4* dst = reinterpret_cast<uint4*>(tc_b);
            for (int i = threadIdx.x; i < TcShape<P>::B_BYTES / 16; i += NT) dst[i] = __ldg(src + i);
            tc::fence_async_smem();
        }
        const int F = grp % 2, tpart = grp / 2;
        const uint32_t row = tb + (uint32_t(F * 64 + (c & ~31)) << 16);   // this warp's lanes
        const R sgn = eg[G_DET * TE + c] < R(0) ? R(-1) : R(1);
        for (int task = tpart; task < 4; task += NG / 2) {   // uniform over each warp
            if (task == 0) {
                const R sF = F == 0 ? sgn : -sgn;
                const int src = F == 0 ? 3 : 0;
#pragma unroll
                for (int k0 = 0; k0 < TS::KC; k0 += 8) {
                    float hi[8], lo[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const int k = k0 + q;
                        const float v = k < 3 * N ? float(sF * us[(src * N + k) * TE + c]) : 0.0f;
                        hi[q] = tc::to_tf32(v);
                        lo[q] = tc::to_tf32(v - hi[q]);
                    }
                    tc::tmem_st8(row + TS::T_SWAP_HI + k0, hi);
                    tc::tmem_st8(row + TS::T_SWAP_LO + k0, lo);
                }
            } else {
                const int j = task - 1, comp = 3 * F + j;
#pragma unroll
                for (int k0 = 0; k0 < TS::KL; k0 += 8) {
                    float hi[8], lo[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const int k = k0 + q, f = k / NF, m = k % NF;
                        // face j + 1 (normal -e_j) has no component j: left out
                        const float v = (k < 4 * NF && f != j + 1)
                                            ? float(trO[((f * 6 + comp) * NF + m) * TE + c]) : 0.0f;
                        hi[q] = tc::to_tf32(v);
                        lo[q] = tc::to_tf32(v - hi[q]);
                    }
                    tc::tmem_st8(row + TS::T_G_HI + j * TS::KL + k0, hi);
                    tc::tmem_st8(row + TS::T_G_LO + j * TS::KL + k0, lo);
                }
            }
        }
        tc::tmem_st_wait();
        tc::fence_before();
        __syncthreads();
        tc::fence_after();
        if (threadIdx.x == 0) {
            const uint32_t bimg = tc::smem_addr(tc_b);
            const uint32_t d = tb + TS::T_D;
            constexpr uint32_t idc = tc::idesc_tf32(128, TS::NC), idl = tc::idesc_tf32(128, TS::NL);
            // three TF32 products per k-step, small ones first: lo hi, hi lo, hi hi
#pragma unroll 1
            for (int ks = 0; ks < TS::KC / 8; ++ks) {
                const uint64_t bh = tc::smem_desc(bimg + ks * 256, 128, TS::SBO_CURL);
                const uint64_t bl = tc::smem_desc(bimg + TS::B_CURL + ks * 256, 128, TS::SBO_CURL);
                tc::mma_tf32_ts(d, tb + TS::T_SWAP_LO + 8 * ks, bh, idc, ks > 0);
                tc::mma_tf32_ts(d, tb + TS::T_SWAP_HI + 8 * ks, bl, idc, true);
                tc::mma_tf32_ts(d, tb + TS::T_SWAP_HI + 8 * ks, bh, idc, true);
            }
#pragma unroll 1
            for (int j = 0; j < 3; ++j)
#pragma unroll 1
                for (int ks = 0; ks < TS::KL / 8; ++ks) {
                    const uint64_t bh = tc::smem_desc(bimg + 2 * TS::B_CURL + ks * 256, 128, TS::SBO_LIFT);
                    const uint64_t bl = tc::smem_desc(bimg + 2 * TS::B_CURL + TS::B_LIFT + ks * 256, 128,
                                                      TS::SBO_LIFT);
                    const uint32_t dj = d + j * TS::NL;
                    tc::mma_tf32_ts(dj, tb + TS::T_G_LO + j * TS::KL + 8 * ks, bh, idl, true);
                    tc::mma_tf32_ts(dj, tb + TS::T_G_HI + j * TS::KL + 8 * ks, bl, idl, true);
                    tc::mma_tf32_ts(dj, tb + TS::T_G_HI + j * TS::KL + 8 * ks, bh, idl, true);
                }
            tc::mma_commit(tc_bar);
        }
        // bounded wait (half a second of wall time, none once another CTA of the
        // launch has given up); on a timeout the status word says so and the
        // stores of phase 5 are skipped
        const bool failed_before = (*reinterpret_cast<volatile int32_t*>(prm.status) & ST_TIMEOUT) != 0;
        const bool done = __syncthreads_and(!failed_before && tc::mbar_wait(tc_bar, 0, 500000000ull));
        if (!done && threadIdx.x == 0) atomicOr(prm.status, int32_t(ST_TIMEOUT));
        tc::fence_after();
        if (!done) {   // leave the outputs alone; release tensor memory once the MMAs
                       // are done (a second bounded wait)
            tc::mbar_wait(tc_bar, 0, 500000000ull);
            tc::fence_before();
            __syncthreads();
            if (threadIdx.x < 32) tc::tmem_dealloc(tb, TS::TCOLS);
            return;
        }
        // D rows (aligned 16-column chunks, shared by the field's groups) into the
        // right-hand-side array of phase 5, with the point source of the E rows
        for (int ch = tpart; ch < TS::NC / 16; ch += NG / 2) {
            float v[16];
            tc::tmem_ld16(row + TS::T_D + 16 * ch, v);
            tc::tmem_ld_wait();
            R gsrc = R(0);
            const double* rec = nullptr;
            if (F == 0 && prm.src != nullptr && active) {
                rec = prm.src + IX(s) * (SRC_HDR + 3 * N);
                if (rec[0] >= 0.0 && IX(rec[0]) == e) {
                    const double tt = prm.tdev ? *prm.tdev + prm.t : prm.t;
                    gsrc = R(source_time(tt, rec[1], rec[2], rec[3]));
                } else {
                    rec = nullptr;
                }
            }
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                const int col16 = 16 * ch + q, j = col16 / TS::NL, l = col16 % TS::NL;
                if (l < N) {
                    R val = R(v[q]);
                    if (rec != nullptr) val -= gsrc * R(rec[SRC_HDR + j * N + l]);
                    rh[((3 * F + j) * N + l) * TE + c] = val;
                }
            }
        }
    }
    for (int it = grp; it < 6 * NPART && !TC; it += NG) {
        const int comp = it / NPART;
        const int part = it % NPART;
        const R sgn = eg[G_DET * TE + c] < R(0) ? R(-1) : R(1);
        R acc[N];
        rhs_part<P, R, TE, NPART>(part, comp, c, us, trO, sgn, acc);
        const int lo = part * N / NPART, hi = (part + 1) * N / NPART;
        if (comp < 3 && prm.src != nullptr && active) {
            const double* rec = prm.src + IX(s) * (SRC_HDR + 3 * N);
            if (rec[0] >= 0.0 && IX(rec[0]) == e) {   // -1 marks a column without a source
                const double tt = prm.tdev ? *prm.tdev + prm.t : prm.t;
                const R g = R(source_time(tt, rec[1], rec[2], rec[3]));
#pragma unroll
                for (int l = 0; l < N; ++l)
                    if (l >= lo && l < hi) acc[l] -= g * R(rec[SRC_HDR + (comp % 3) * N + l]);
            }
        }
#pragma unroll
        for (int l = 0; l < N; ++l)
            if (l >= lo && l < hi) rh[(comp * N + l) * TE + c] = acc[l];
        if (MODE == MODE_RAW && active) {
            R* rw = static_cast<R*>(prm.raw);
#pragma unroll
            for (int l = 0; l < N; ++l)
                if (l >= lo && l < hi) rw[IX(comp * N + l) * C + col] = acc[l];
        }
    }
    if (MODE == MODE_RAW) return;   // forward quantities for the adjoint only
    __syncthreads();

    // ---- phase 5: mass-block inverse, PML, update per (field, row part) --------
    for (int it = grp; it < 2 * NP5; it += NG) {
        const int field = it / NP5;
        const int part = it % NP5;
        if (!active) continue;
        const int fb = 3 * field;   // first component of this field
        const R det = eg[G_DET * TE + c];
        const R mat = field == 0 ? eg[G_EPS * TE + c] : eg[G_MU * TE + c];
        // the 3x3 mass-block inverse A^T A / (mat |det|), symmetric, from the
        // metric that phase 1 stored
        R B[3][3];
        const R inv = R(1) / (mat * fabs(det));
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int k = j; k < 3; ++k) {
                B[j][k] = inv * gm[sym3(j, k) * TE + c];
                B[k][j] = B[j][k];
            }
        // PML: (A^T D A^-T)[j][k] = sum_a A^T[j][a] D_a A^-T[a][k] for D = eta, Sigma, xi
        int32_t pi = -1;
        if (PML && prm.pml != nullptr) pi = prm.pml[e];
        R ETA[3][3], SIG[3][3], XI[3][3];
        R ait[9], AT[3][3], sg3[3], et3[3], xi3[3];   // PML: A^-T, A^T, sigma, eta, xi
        if (PML && pi >= 0) {
#pragma unroll
            for (int k = 0; k < 9; ++k) ait[k] = eg[(G_AIT + k) * TE + c];
            // A^T = adj(A^-T) det A
            AT[0][0] = ait[4] * ait[8] - ait[5] * ait[7];
            AT[0][1] = ait[2] * ait[7] - ait[1] * ait[8];
            AT[0][2] = ait[1] * ait[5] - ait[2] * ait[4];
            AT[1][0] = ait[5] * ait[6] - ait[3] * ait[8];
            AT[1][1] = ait[0] * ait[8] - ait[2] * ait[6];
            AT[1][2] = ait[2] * ait[3] - ait[0] * ait[5];
            AT[2][0] = ait[3] * ait[7] - ait[4] * ait[6];
            AT[2][1] = ait[1] * ait[6] - ait[0] * ait[7];
            AT[2][2] = ait[0] * ait[4] - ait[1] * ait[3];
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int b = 0; b < 3; ++b) AT[a][b] *= det;
            const R sx = eg[(G_SIG + 0) * TE + c], sy = eg[(G_SIG + 1) * TE + c],
                    sz = eg[(G_SIG + 2) * TE + c];
            sg3[0] = sx; sg3[1] = sy; sg3[2] = sz;
            et3[0] = sy + sz - sx; et3[1] = sz + sx - sy; et3[2] = sx + sy - sz;
            xi3[0] = (sx - sy) * (sx - sz); xi3[1] = (sy - sz) * (sy - sx); xi3[2] = (sz - sx) * (sz - sy);
#pragma unroll
            for (int j = 0; j < 3; ++j)
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    ETA[j][k] = R(0);
                    SIG[j][k] = R(0);
                    XI[j][k] = R(0);
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        const R w = AT[j][a] * ait[3 * a + k];
                        ETA[j][k] += w * et3[a];
                        SIG[j][k] += w * sg3[a];
                        XI[j][k] += w * xi3[a];
                    }
                }
        }
        const R imat = R(1) / mat;
        const IX C2 = IX(prm.npml) * S;
        const IX acol = IX(pi) * S + s;
        R* uo = static_cast<R*>(prm.u_out);
        R* res = static_cast<R*>(prm.res);
        const R* aux = static_cast<const R*>(prm.aux);
        R* auxo = static_cast<R*>(prm.aux_out);
        R* auxr = static_cast<R*>(prm.aux_res);
        const R dt = coef(prm.dt, prm.dt_f), ca = coef(prm.a, prm.a_f), cb = coef(prm.b, prm.b_f);
        const int lo = part * N / NP5, hi = (part + 1) * N / NP5;
        const IX gb = IX(fb * N + lo) * C + col;          // (fb, lo) in the fields
        const IX ab = IX(fb * N + lo) * C2 + acol;        // (fb, lo) in the auxiliaries
        // rows l = lo + i with a compile-time i, so that the prefetched residuals
        // stay in registers; in the layer in chunks whose loads are all requested
        // before their arithmetic
        constexpr int CR = RP5 < 2 ? RP5 : 2;
#pragma unroll
        for (int i0 = 0; i0 < RP5; i0 += CR) {
            R av[CR][3], ar[CR][3];
#pragma unroll
            for (int i = 0; i < CR; ++i)
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const bool ok = PML && pi >= 0 && i0 + i < RP5 && (P5_EVEN || lo + i0 + i < hi);
                    const IX aj = ab + IX(k * N + i0 + i) * C2;
                    av[i][k] = ok ? aux[aj] : R(0);
                    ar[i][k] = ok && ca != R(0) ? auxr[aj] : R(0);
                }
#pragma unroll
            for (int i = 0; i < CR; ++i) {
                const int l = lo + i0 + i;
                if (i0 + i >= RP5 || (!P5_EVEN && l >= hi)) break;
                R r[3], uv[3], du[3];
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    r[k] = rh[((fb + k) * N + l) * TE + c];
                    uv[k] = us[((fb + k) * N + l) * TE + c];
                }
#pragma unroll
                for (int k = 0; k < 3; ++k) du[k] = B[k][0] * r[0] + B[k][1] * r[1] + B[k][2] * r[2];
                if (PML && pi >= 0) {
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        du[k] -= ETA[k][0] * uv[0] + ETA[k][1] * uv[1] + ETA[k][2] * uv[2] + av[i][k] * imat;
                        const R da = -(SIG[k][0] * av[i][0] + SIG[k][1] * av[i][1] + SIG[k][2] * av[i][2]) +
                                     mat * (XI[k][0] * uv[0] + XI[k][1] * uv[1] + XI[k][2] * uv[2]);
                        const IX aj = ab + IX(k * N + i0 + i) * C2;
                        const R rr = (ca == R(0) ? R(0) : ca * ar[i][k]) + dt * da;
                        auxr[aj] = rr;
                        auxo[aj] = av[i][k] + cb * rr;
                    }
                }
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const IX gi = gb + IX(k * N + i0 + i) * C;
                    // resv is 0 when a = 0 (first stage), so no branch on a here
                    const R rr = ca * resv[PREFETCH_RES ? k : 0][PREFETCH_RES ? i0 + i : 0] + dt * du[k];
                    res[gi] = rr;
                    uo[gi] = uv[k] + cb * rr;
                }
            }
        }
    }
    if constexpr (TC) {
        tc::fence_before();
        __syncthreads();
        if (threadIdx.x < 32) tc::tmem_dealloc(*tc_base, TcShape<P>::TCOLS);
    }
}

}  // namespace dgm
