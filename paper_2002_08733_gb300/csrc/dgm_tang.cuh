// Fused DG right-hand-side / stage-update kernel on tangential traces (SIMT,
// FP64 or FP32).  It evaluates the semi-discrete system stated at the head of
// dgm_stage.cuh; this file's form of it has no geometry in the jumps.
//
// Tangential traces.  Only n x X of a trace enters a flux, and for covariant
// coefficients x (X = A^-T x) the tangential part of X on a face is carried by
// the two numbers tau_i = x . t_i, t_i the reference tangents of the face:
//   face 0 (x + y + z = 1): t_1 = e_1 - e_0, t_2 = e_2 - e_0;
//   face a + 1 (x_a = 0):   t_1 = e_b, t_2 = e_c, {b < c} the other two axes.
// A t_i are the face's edges from its lowest vertex, and both elements of a
// face keep their vertices in ascending global id: the edges, their order and
// the parametrisation of the face modes are the same seen from either side.
// So the jump of a face mode is tau_i(+) - tau_i(-), with no matrix between
// the two elements' frames, and a trace costs two components instead of three.
// With sigma_f = -1, +1, -1, +1 for f = 0..3 the identity (M a) x (M b) =
// det M M^-T (a x b), M = A^-T, turns the pulled-back fluxes into two numbers
// per field as well, g = gamma_1 e_b + gamma_2 e_c (face 0: component 0 of g is
// -(gamma_1 + gamma_2)), the same on every face:
//   s_T gE: gamma_1 =  cE dh_2 + e22 de_1 - e12 de_2,  gamma_2 = -cE dh_1 + e11 de_2 - e12 de_1
//  -s_T gH: gamma_1 =  cH de_2 - h22 dh_1 + h12 dh_2,  gamma_2 = -cH de_1 - h11 dh_2 + h12 dh_1
// (de, dh: jumps of tau; cE = sigma c_E, cH = sigma c_H;
// e_ij = s_T b_E (A t_i . A t_j) / (|det A| |M m_f|), h_ij with b_H).  The
// signs s_T are moved into the mass block:
//   du_E = A^T A / (eps det) [curl u_H + lift(s_T gE)]
//   du_H = -A^T A / (mu det) [curl u_E + lift(-s_T gH)].
//
// One CTA owns TE consecutive columns with NG threads per column.
//   phase A: a thread takes one face (NG = 4) or one face and field (NG = 8) of
//     its column: own trace from the tile in shared memory, neighbour trace
//     from its gathered coefficients, both into the same sums; then the flux,
//     written to shared memory.
//   phase B: a thread takes one field and one part of the rows: curl and lift
//     of all three components in registers, then the mass block, the PML terms
//     and the stage update, so the right-hand side never leaves the registers.
// One barrier between the two (and one before phase A for the tile).
//
// What bounds it.  FP64: the FP64 pipe (84 % of its rate at 48,000 elements,
// p = 3); the tangential form needs 6.1 k operations per element-stage instead of
// about 10 k, and with full warps of 32 columns no warp runs two row parts in
// turn: 22.8 -> 11.9 ms per LSRK4 step of the 32^3 grid.  FP32: instruction issue
// and latency (IPC 0.47 per SM quarter at 14 warps; long-scoreboard, instruction
// fetch and barrier stalls); 372 warp instructions per 32 element-stages against
// 669: 0.882 -> 0.598 ms per step of the 32^3 grid at p = 3 (0.285 ms at the
// measured HBM rate), 6.64 -> 4.63 ms on the 40^3 grid at p = 4 with a PML.
// Two columns per thread in packed FP32x2 instructions (half the instructions) was
// slower, 0.673 ms: twice the registers per thread left half the columns in
// flight.
#pragma once

#include <cstdint>
#include <type_traits>

#include "dgm_internal.h"
#include "dgm_ops_gen.cuh"
#include "dgm_bulk.cuh"
#include "dgm_stage.cuh"

namespace dgm {

// Face and element constants of this kernel, one row per constant, [TG_ROWS][K]
// in the plan's precision (tang_consts_kernel).
enum TangConst {
    TG_CE = 0, TG_CH = 1, TG_E11 = 2, TG_NE12 = 3, TG_E22 = 4, TG_NH11 = 5, TG_H12 = 6, TG_NH22 = 7,
    TG_FACE = 8,                  // rows per face
    TG_METRIC = 4 * TG_FACE,      // A^T A: 00, 01, 02, 11, 12, 22
    TG_IE = TG_METRIC + 6,        // 1 / (eps det A)
    TG_IH = TG_METRIC + 7         // -1 / (mu det A)
};
static_assert(TG_IH + 1 == TG_ROWS, "rows of the tangential face-constant table");
// interior penalty, a table of its own, per face (TG_SIPF rows): KS, A t_1 (3), A t_2 (3)

// component of tangent i of face f (face 0: minus component 0)
__host__ __device__ constexpr int tang_comp(int f, int i) { return f == 2 ? 2 * i : (f == 3 ? i : 1 + i); }

// One thread per element, from the FP64 geometry (once per plan, again when the
// materials or the boundary codes change); rounded to the plan's precision last.
template <typename R>
__global__ void tang_consts_kernel(const StageParams prm, bool sip, R* __restrict__ out) {
    const int64_t K = prm.K;
    const int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (e >= K) return;
    double M[9], at[9];
    for (int k = 0; k < 9; ++k) M[k] = prm.geo[int64_t(G_AIT + k) * K + e];
    const double det = prm.geo[int64_t(G_DET) * K + e];
    const double eps = prm.geo[int64_t(G_EPS) * K + e], mu = prm.geo[int64_t(G_MU) * K + e];
    // A^T = det A adj(A^-T), row major: row j is the edge A e_j
    at[0] = M[4] * M[8] - M[5] * M[7];
    at[1] = M[2] * M[7] - M[1] * M[8];
    at[2] = M[1] * M[5] - M[2] * M[4];
    at[3] = M[5] * M[6] - M[3] * M[8];
    at[4] = M[0] * M[8] - M[2] * M[6];
    at[5] = M[2] * M[3] - M[0] * M[5];
    at[6] = M[3] * M[7] - M[4] * M[6];
    at[7] = M[1] * M[6] - M[0] * M[7];
    at[8] = M[0] * M[4] - M[1] * M[3];
    for (int k = 0; k < 9; ++k) at[k] *= det;
    const double zm = sqrt(mu / eps);
    for (int f = 0; f < 4; ++f) {
        double T[2][3], vn[3];
        for (int i = 0; i < 2; ++i)
            for (int r = 0; r < 3; ++r)
                T[i][r] = at[3 * tang_comp(f, i) + r] - (f == 0 ? at[r] : 0.0);
        const double m[3] = {f == 0 ? 1.0 : (f == 1 ? -1.0 : 0.0), f == 0 ? 1.0 : (f == 2 ? -1.0 : 0.0),
                             f == 0 ? 1.0 : (f == 3 ? -1.0 : 0.0)};
        for (int r = 0; r < 3; ++r) vn[r] = M[3 * r] * m[0] + M[3 * r + 1] * m[1] + M[3 * r + 2] * m[2];
        const double kb = 1.0 / (det * sqrt(vn[0] * vn[0] + vn[1] * vn[1] + vn[2] * vn[2]));   // s_T / (|det| |M m|)
        const int32_t code = prm.nbr[int64_t(f) * K + e];
        const bool has = code >= 0 && (code >> 2) < K;
        const int64_t en = has ? int64_t(code >> 2) : e;
        const double mun = prm.geo[int64_t(G_MU) * K + en];
        const double zp = has ? sqrt(mun / prm.geo[int64_t(G_EPS) * K + en]) : zm;
        double ce = 0.5, ch = 0.5, be = 0.0, bh = 0.0;
        if (prm.upwind) {
            ce = zp / (zm + zp);
            be = 1.0 / (zm + zp);
            ch = zm / (zm + zp);
            bh = zm * zp / (zm + zp);
        }
        const double sg = (f & 1) ? 1.0 : -1.0;
        const double t11 = T[0][0] * T[0][0] + T[0][1] * T[0][1] + T[0][2] * T[0][2];
        const double t12 = T[0][0] * T[1][0] + T[0][1] * T[1][1] + T[0][2] * T[1][2];
        const double t22 = T[1][0] * T[1][0] + T[1][1] * T[1][1] + T[1][2] * T[1][2];
        const double v[TG_FACE] = {sg * ce, sg * ch, kb * be * t11, -kb * be * t12, kb * be * t22,
                                   -kb * bh * t11, kb * bh * t12, -kb * bh * t22};
        for (int k = 0; k < TG_FACE; ++k) out[int64_t(f * TG_FACE + k) * K + e] = R(v[k]);
        if (sip) {
            const int32_t sf = prm.sfid[int64_t(f) * K + e];
            const double ks = (sf >= 0 && (sf & 1)) ? prm.sip_alpha / (0.5 * (mu + mun)) * kb : 0.0;
            R* o = const_cast<R*>(static_cast<const R*>(prm.fcp)) + int64_t(f * TG_SIPF) * K + e;
            o[0] = R(ks);
            for (int i = 0; i < 2; ++i)
                for (int r = 0; r < 3; ++r) o[int64_t(1 + 3 * i + r) * K] = R(T[i][r]);
        }
    }
    int k = TG_METRIC;
    for (int i = 0; i < 3; ++i)
        for (int j = i; j < 3; ++j, ++k)
            out[int64_t(k) * K + e] = R(at[3 * i] * at[3 * j] + at[3 * i + 1] * at[3 * j + 1] + at[3 * i + 2] * at[3 * j + 2]);
    out[int64_t(TG_IE) * K + e] = R(1.0 / (eps * det));
    out[int64_t(TG_IH) * K + e] = R(-1.0 / (mu * det));
}

// Mixed orders (MX): E of degree P, H of degree P - 1.  The bases are hierarchical,
// so H's operators are those of degree P - 1, the curl of H tested against E is the
// degree P - 1 curl, the curl of E tested against H the rows of the degree-P one,
// and an E jump enters the H flux with its first face modes.
// Field rows: E component k, mode l at k N + l, H at 3 N + k N_H + l.
template <int P, bool MX> __host__ __device__ constexpr int deg_h() { return MX ? P - 1 : P; }
template <int P, bool MX> __host__ __device__ constexpr int field_rows() {
    return 3 * (nmodes(P) + nmodes(deg_h<P, MX>()));
}

// shared memory: the tile's coefficients [rows][TE], the face quantities
// [face][field][tangent][NF][TE] (jumps, then fluxes), an mbarrier
template <int P, typename R, int TE, bool MX = false>
__host__ __device__ constexpr size_t tang_smem_bytes() {
    return sizeof(R) * size_t(TE) * (field_rows<P, MX>() + 16 * nfmodes(P)) + 16;
}

// minus the own trace of face f of the row block at v (row stride TE), less that at v0 on face 0
template <int P, typename R, int TE>
__device__ __forceinline__ void own_trace(int f, const R* v, const R* v0, R (&acc)[nfmodes(P)]) {
    switch (f) {
        case 0: TraceOp<P, 0>::template own<true>(v, v0, TE, acc); break;
        case 1: TraceOp<P, 1>::template own<false>(v, v0, TE, acc); break;
        case 2: TraceOp<P, 2>::template own<false>(v, v0, TE, acc); break;
        default: TraceOp<P, 3>::template own<false>(v, v0, TE, acc); break;
    }
}

// acc += trace of v on face f
template <int P, typename R>
__device__ __forceinline__ void jump_trace(int f, const R (&v)[nmodes(P)], R (&acc)[nfmodes(P)]) {
    switch (f) {
        case 0: TraceOp<P, 0>::jump(v, acc); break;
        case 1: TraceOp<P, 1>::jump(v, acc); break;
        case 2: TraceOp<P, 2>::jump(v, acc); break;
        default: TraceOp<P, 3>::jump(v, acc); break;
    }
}

// Tuning of the two phases; FP32 figures are ms per LSRK4 step of the 32^3 (p = 3)
// and 24^3 grids, the alternatives measured on the same box.
//
// NG = 4: the larger row part of phase B goes to the threads of faces 1 and 2,
// whose phase A is the shortest (20 and 50 trace entries at p = 3 against 142
// and 125), so that the four warps of a CTA, one per SM quarter, have the same
// amount to do: p = 3 0.602 with rows [0, 13) | [13, 20), 0.631 with equal parts in
// group order.  With a PML phase B outweighs phase A, and equal parts are as good.
template <int P, typename R, bool PML>
__host__ __device__ constexpr bool tang_balance() { return sizeof(R) == 4 && !PML && (P == 3 || P == 4); }
template <int P, typename R, bool PML>
__host__ __device__ constexpr int tang_split(int np, int k) {
    if (np > 4) return k * nmodes(P) / np;
    if (np == 2 && tang_balance<P, R, PML>() && P == 3) return k == 0 ? 0 : k == 1 ? 13 : nmodes(P);
    return row_split(P, np, k);
}
// Residual rows held in registers from before the curl and lift on, in bytes per
// thread: hides their latency where it fits (p = 3 0.602 against 0.673), spills
// where it does not (p = 4 with a PML 0.99 against 1.15).
template <int P, typename R, bool PML>
__host__ __device__ constexpr int tang_early_bytes() {
    return sizeof(R) == 8 ? 144 : P >= 4 && PML ? 0 : P == 5 ? 0 : PML ? 144 : 180;
}

// A thread's column: id, element, source; active: updated by this launch.
template <typename IX>
struct Column {
    IX C, col, e;
    int s;
    bool active;
};

// Phase B of one thread: rows [LO, HI) of the three components of field F
// (0: E, 1: H) of degree P, the other field of degree PO.  us, gs: shared memory
// at this thread's column; r0, ro: first field rows of this and the other field;
// NF: face modes per row group of gs.
template <int P, int PO, int NF, typename R, int TE, int MODE, typename IX, bool PML, int LO, int HI>
__device__ __forceinline__ void tang_rows(const StageParams& prm, int F, const R* us, const R* gs,
                                          const Column<IX>& id, int r0, int ro) {
    constexpr int N = nmodes(P), NR = HI - LO;
    constexpr bool LF = MODE == MODE_LF_E || MODE == MODE_LF_H;
    // residual rows requested before the arithmetic where the registers allow it
    constexpr bool EARLY = MODE == MODE_LSRK && 3 * NR * int(sizeof(R)) <= tang_early_bytes<P, R, PML>();
    auto coef = [&](double d, float f) { return sizeof(R) == 4 ? R(f) : R(d); };
    const IX K = prm.K, C = id.C;
    const bool active = id.active;
    const R ca = coef(prm.a, prm.a_f), cb = coef(prm.b, prm.b_f), dt = coef(prm.dt, prm.dt_f);
    const IX gb = IX(r0 + LO) * C + id.col;
    const R* resi = static_cast<const R*>(prm.res);   // written below, by the same thread after it has read
    const bool ld = active && ca != R(0);
    R rv[EARLY ? NR : 1][3];
    if constexpr (EARLY) {
#pragma unroll
        for (int i = 0; i < NR; ++i)
#pragma unroll
            for (int k = 0; k < 3; ++k) rv[i][k] = ld ? resi[gb + IX(k * N + i) * C] : R(0);
    }
    // a row of a per-element table at the thread's elements
    auto table = [&](const void* base, int row) -> R {
        const R* b = static_cast<const R*>(base) + IX(row) * K;
        return b[id.e];
    };
    const R g00 = table(prm.fct, TG_METRIC), g01 = table(prm.fct, TG_METRIC + 1), g02 = table(prm.fct, TG_METRIC + 2);
    const R g11 = table(prm.fct, TG_METRIC + 3), g12 = table(prm.fct, TG_METRIC + 4), g22 = table(prm.fct, TG_METRIC + 5);
    const R im = table(prm.fct, TG_IE + F);   // 1 / (eps det) or -1 / (mu det)

    R a0[N], a1[N], a2[N];
#pragma unroll
    for (int l = LO; l < HI; ++l) a1[l] = a2[l] = R(0);
    const R* g = gs + 2 * F * NF * TE;    // this field's gamma_1 of face 0; face f at + 4 f NF TE
    LiftOp<P, 0>::template apply<R, LO, HI>(g, TE, a1);
    LiftOp<P, 0>::template apply<R, LO, HI>(g + NF * TE, TE, a2);
#pragma unroll
    for (int l = LO; l < HI; ++l) a0[l] = (a1[l] + a2[l]) * R(-1);
    CurlOp<PO>::template apply<R, LO, HI>(us + ro * TE, nmodes(PO) * TE, TE, a0, a1, a2);
    LiftOp<P, 1>::template apply<R, LO, HI>(g + 4 * NF * TE, TE, a1);
    LiftOp<P, 1>::template apply<R, LO, HI>(g + 5 * NF * TE, TE, a2);
    LiftOp<P, 2>::template apply<R, LO, HI>(g + 8 * NF * TE, TE, a0);
    LiftOp<P, 2>::template apply<R, LO, HI>(g + 9 * NF * TE, TE, a2);
    LiftOp<P, 3>::template apply<R, LO, HI>(g + 12 * NF * TE, TE, a0);
    LiftOp<P, 3>::template apply<R, LO, HI>(g + 13 * NF * TE, TE, a1);
    if (!active) return;

    if (F == 0 && prm.src != nullptr) {
        const double* rec = prm.src + IX(id.s) * (SRC_HDR + 3 * N);   // (E's N)
        if (rec[0] >= 0.0 && IX(rec[0]) == id.e) {   // -1 marks a column without a source
            const double tt = prm.tdev ? *prm.tdev + prm.t : prm.t;
            // the rows carry the factor s_T = sign of det A
            const R gt = (im < R(0) ? R(1) : R(-1)) * R(source_time(tt, rec[1], rec[2], rec[3]));
#pragma unroll
            for (int l = LO; l < HI; ++l) {
                a0[l] = fmaa(gt, R(rec[SRC_HDR + l]), a0[l]);
                a1[l] = fmaa(gt, R(rec[SRC_HDR + N + l]), a1[l]);
                a2[l] = fmaa(gt, R(rec[SRC_HDR + 2 * N + l]), a2[l]);
            }
        }
    }
    R* res = static_cast<R*>(prm.res);
    R* uo = static_cast<R*>(prm.u_out);
    // the mass block; outside the right-hand-side mode scaled by the step
    const R sc = MODE == MODE_RHS ? im : im * dt;
    const R b00 = sc * g00, b01 = sc * g01, b02 = sc * g02, b11 = sc * g11, b12 = sc * g12, b22 = sc * g22;
#pragma unroll
    for (int l = LO; l < HI; ++l) {
        const R r0 = a0[l], r1 = a1[l], r2 = a2[l];
        a0[l] = fmaa(b02, r2, fmaa(b01, r1, b00 * r0));
        a1[l] = fmaa(b12, r2, fmaa(b11, r1, b01 * r0));
        a2[l] = fmaa(b22, r2, fmaa(b12, r1, b02 * r0));
    }
    if constexpr (PML) {
        const int32_t pi = prm.pml != nullptr ? prm.pml[id.e] : -1;
        if (pi >= 0) {
            // PML: D -> A^T D A^-T for D = eta, Sigma, xi ; leapfrog works
            // per Cartesian component in the physical frame
            R M[9], AT[3][3];
#pragma unroll
            for (int k = 0; k < 9; ++k) M[k] = table(prm.geo_r, G_AIT + k);
            const R det = table(prm.geo_r, G_DET);
            const R mat = table(prm.geo_r, G_EPS + F);
            const R imat = R(1) / mat;
            const R sx = table(prm.geo_r, G_SIG), sy = table(prm.geo_r, G_SIG + 1), sz = table(prm.geo_r, G_SIG + 2);
            AT[0][0] = det * (M[4] * M[8] - M[5] * M[7]);
            AT[0][1] = det * (M[2] * M[7] - M[1] * M[8]);
            AT[0][2] = det * (M[1] * M[5] - M[2] * M[4]);
            AT[1][0] = det * (M[5] * M[6] - M[3] * M[8]);
            AT[1][1] = det * (M[0] * M[8] - M[2] * M[6]);
            AT[1][2] = det * (M[2] * M[3] - M[0] * M[5]);
            AT[2][0] = det * (M[3] * M[7] - M[4] * M[6]);
            AT[2][1] = det * (M[1] * M[6] - M[0] * M[7]);
            AT[2][2] = det * (M[0] * M[4] - M[1] * M[3]);
            const R sg[3] = {sx, sy, sz};
            const R et[3] = {sy + sz - sx, sz + sx - sy, sx + sy - sz};
            const R xi[3] = {(sx - sy) * (sx - sz), (sy - sz) * (sy - sx), (sz - sx) * (sz - sy)};
            const IX C2 = IX(prm.npml) * IX(prm.S);
            const IX acol = IX(pi) * IX(prm.S) + id.s;
            auto load_aux = [&](const R* p, IX row) -> R { return p[row * C2 + acol]; };
            auto store_aux = [&](R* p, IX row, R v) { p[row * C2 + acol] = v; };
            // The rows run in chunks whose loads are all requested before their
            // arithmetic.  FP32 from p = 4 on the chunks share one loop body, the
            // right-hand side rotating through the registers, because the code far
            // exceeds the instruction cache (249 -> 221 KB; two steps of the 40^3 dipole
            // at p = 4 9.79 -> 9.27 ms).  At p = 3 (130 -> 114 KB) the rotation costs more
            // than the misses (24^3 batch, 16 columns: 21.0 -> 21.9 ms): unrolled, where
            // the rotation is only a renaming.
            constexpr int CH = sizeof(R) == 8 ? 2 : LF ? 4 : 3, NRP = round_up(NR, CH);
            constexpr int UNROLL = P >= 4 && sizeof(R) == 4 ? 1 : NRP / CH;
            R q0[NRP], q1[NRP], q2[NRP];
#pragma unroll
            for (int i = 0; i < NRP; ++i) {
                q0[i] = i < NR ? a0[LO + (i < NR ? i : 0)] : R(0);
                q1[i] = i < NR ? a1[LO + (i < NR ? i : 0)] : R(0);
                q2[i] = i < NR ? a2[LO + (i < NR ? i : 0)] : R(0);
            }
            auto rotate = [&](R (&q)[NRP]) {
                R t[CH];
#pragma unroll
                for (int i = 0; i < CH; ++i) t[i] = q[i];
#pragma unroll
                for (int i = 0; i + CH < NRP; ++i) q[i] = q[i + CH];
#pragma unroll
                for (int i = 0; i < CH; ++i) q[NRP - CH + i] = t[i];
            };
            const IX ab = IX(r0 + LO);   // (both fields of degree P)
            if constexpr (LF) {
                // Leapfrog with the PML terms by the trapezoid rule (Sec. V), X = A^-T x:
                //   X_new = ((1 - dt eta/2) X + dt (A^-T du - A^-T aux / mat)) / (1 + dt eta/2)
                // then the other field's auxiliary, Y = A^-T (other field), mat' its material:
                //   Z_new = ((1 - dt sigma/2) Z + dt mat' xi Y) / (1 + dt sigma/2)
                const R omat = table(prm.geo_r, G_EPS + 1 - F);
                const IX abo = IX(ro + LO);
                R* auxl = static_cast<R*>(prm.aux_out);   // in place: aux_out == aux
                R xx[3], xy[3], za[3], zb[3];
                const R ndi = imat * -dt;
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const R hd = R(0.5) * dt * et[a], hs = R(0.5) * dt * sg[a];
                    const R nx = R(1) + hd, nz = R(1) + hs;
                    xy[a] = R(1) / nx;
                    xx[a] = (R(1) - hd) * xy[a];
                    const R iz = R(1) / nz;
                    za[a] = (R(1) - hs) * iz;
                    zb[a] = iz * dt * omat * xi[a];
                }
#pragma unroll(UNROLL)
                for (int i0 = 0; i0 < NR; i0 += CH) {
                    R av[CH][3], oa[CH][3];
#pragma unroll
                    for (int i = 0; i < CH; ++i) {
                        const bool ok = i0 + i < NR;
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            av[i][k] = ok ? load_aux(auxl, ab + IX(k * N + i0 + i)) : R(0);
                            oa[i][k] = ok ? load_aux(auxl, abo + IX(k * N + i0 + i)) : R(0);
                        }
                    }
#pragma unroll
                    for (int i = 0; i < CH; ++i) {
                        if (i0 + i >= NR) break;
                        const int l = LO + i0 + i;
                        R ov[3], uv[3], Xn[3], Zn[3];
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            uv[k] = us[(r0 + k * N + l) * TE];
                            ov[k] = us[(ro + k * N + l) * TE];
                        }
#pragma unroll
                        for (int a = 0; a < 3; ++a) {
                            auto phys = [&](R p, R q, R r) {
                                return fmaa(M[3 * a + 2], r, fmaa(M[3 * a + 1], q, M[3 * a] * p));
                            };
                            const R y = fmaa(ndi, phys(av[i][0], av[i][1], av[i][2]), phys(q0[i], q1[i], q2[i]));
                            Xn[a] = fmaa(xx[a], phys(uv[0], uv[1], uv[2]), xy[a] * y);
                            Zn[a] = fmaa(za[a], phys(oa[i][0], oa[i][1], oa[i][2]), zb[a] * phys(ov[0], ov[1], ov[2]));
                        }
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            uo[gb + IX(k * N + i0 + i) * C] =
                                fmaa(AT[k][2], Xn[2], fmaa(AT[k][1], Xn[1], AT[k][0] * Xn[0]));
                            store_aux(auxl, abo + IX(k * N + i0 + i),
                                      fmaa(AT[k][2], Zn[2], fmaa(AT[k][1], Zn[1], AT[k][0] * Zn[0])));
                        }
                    }
                    rotate(q0);
                    rotate(q1);
                    rotate(q2);
                }
                return;
            } else {
                // (an auxiliary residual row is read before it is written, by the same thread)
                const R* aux = static_cast<const R*>(prm.aux);
                const R* auxi = static_cast<const R*>(prm.aux_res);
                R* auxo = static_cast<R*>(prm.aux_out);
                R* auxr = static_cast<R*>(prm.aux_res);
                // -eta, -Sigma, mat xi and -1/mat, times the step outside the right-hand-side mode
                const R st = MODE == MODE_RHS ? R(1) : dt;
                const R nst = R(-1) * st, ni = nst * imat;
                R ETA[3][3], SIG[3][3], XI[3][3];
#pragma unroll
                for (int j = 0; j < 3; ++j)
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        const R w0 = AT[j][0] * M[k], w1 = AT[j][1] * M[3 + k], w2 = AT[j][2] * M[6 + k];
                        ETA[j][k] = nst * fmaa(w2, et[2], fmaa(w1, et[1], w0 * et[0]));
                        SIG[j][k] = nst * fmaa(w2, sg[2], fmaa(w1, sg[1], w0 * sg[0]));
                        XI[j][k] = st * mat * fmaa(w2, xi[2], fmaa(w1, xi[1], w0 * xi[0]));
                    }
#pragma unroll(UNROLL)
                for (int i0 = 0; i0 < NR; i0 += CH) {
                    R av[CH][3], ar[CH][3];
#pragma unroll
                    for (int i = 0; i < CH; ++i) {
                        const bool ok = i0 + i < NR;
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            av[i][k] = ok ? load_aux(aux, ab + IX(k * N + i0 + i)) : R(0);
                            ar[i][k] = (MODE == MODE_LSRK && ok && ca != R(0)) ? load_aux(auxi, ab + IX(k * N + i0 + i)) : R(0);
                        }
                    }
#pragma unroll
                    for (int i = 0; i < CH; ++i) {
                        if (i0 + i >= NR) break;
                        const int l = LO + i0 + i;
                        R uv[3], d[3];
#pragma unroll
                        for (int k = 0; k < 3; ++k) uv[k] = us[(r0 + k * N + l) * TE];
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            d[k] = fmaa(ni, av[i][k], fmaa(ETA[k][2], uv[2], fmaa(ETA[k][1], uv[1], ETA[k][0] * uv[0])));
                            const R da = fmaa(SIG[k][2], av[i][2], fmaa(SIG[k][1], av[i][1], fmaa(SIG[k][0], av[i][0],
                                         fmaa(XI[k][2], uv[2], fmaa(XI[k][1], uv[1], XI[k][0] * uv[0])))));
                            const IX row = ab + IX(k * N + i0 + i);
                            if (MODE == MODE_RHS) {
                                store_aux(auxo, row, da);
                            } else {
                                const R rr = fmaa(ca, ar[i][k], da);
                                store_aux(auxr, row, rr);
                                store_aux(auxo, row, fmaa(cb, rr, av[i][k]));
                            }
                        }
                        q0[i] += d[0];
                        q1[i] += d[1];
                        q2[i] += d[2];
                    }
                    rotate(q0);
                    rotate(q1);
                    rotate(q2);
                }
#pragma unroll
                for (int i = 0; i < NR; ++i) {
                    a0[LO + i] = q0[i];
                    a1[LO + i] = q1[i];
                    a2[LO + i] = q2[i];
                }
            }
        }
    }
    // update; residual rows in chunks when they were not requested early
    constexpr int CH = EARLY ? NR : int(32 / sizeof(R));
#pragma unroll
    for (int i0 = 0; i0 < NR; i0 += CH) {
        R rc[CH][3];
        if constexpr (MODE == MODE_LSRK) {
#pragma unroll
            for (int i = 0; i < CH; ++i) {
                if (i0 + i >= NR) break;
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    if constexpr (EARLY) rc[i][k] = rv[i][k];
                    else rc[i][k] = ld ? resi[gb + IX(k * N + i0 + i) * C] : R(0);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < CH; ++i) {
            if (i0 + i >= NR) break;
            const int l = LO + i0 + i;
            const R du[3] = {a0[l], a1[l], a2[l]};
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const IX gi = gb + IX(k * N + i0 + i) * C;
                if (MODE == MODE_RHS) {
                    uo[gi] = du[k];
                } else if (MODE == MODE_LSRK) {
                    const R rr = fmaa(ca, rc[i][k], du[k]);
                    res[gi] = rr;
                    uo[gi] = fmaa(cb, rr, us[(r0 + k * N + l) * TE]);
                } else {
                    uo[gi] = us[(r0 + k * N + l) * TE] + du[k];
                }
            }
        }
    }
}

template <int P, int PO, int NF, typename R, int TE, int MODE, typename IX, bool PML, int NPART, int K0 = 0>
__device__ __forceinline__ void tang_parts(const StageParams& prm, int F, int part, const R* us, const R* gs,
                                           const Column<IX>& id, int r0, int ro) {
    if (part == K0)
        tang_rows<P, PO, NF, R, TE, MODE, IX, PML, tang_split<P, R, PML>(NPART, K0),
                  tang_split<P, R, PML>(NPART, K0 + 1)>(prm, F, us, gs, id, r0, ro);
    else if constexpr (K0 + 1 < NPART)
        tang_parts<P, PO, NF, R, TE, MODE, IX, PML, NPART, K0 + 1>(prm, F, part, us, gs, id, r0, ro);
}

// one code path for both fields where their degrees are equal
template <int P, typename R, int TE, int MODE, typename IX, bool PML, bool MX, int NPART>
__device__ __forceinline__ void tang_part(const StageParams& prm, int F, int part, const R* us, const R* gs,
                                          const Column<IX>& id) {
    constexpr int PH = deg_h<P, MX>(), N = nmodes(P), NF = nfmodes(P);
    if constexpr (!MX) {
        tang_parts<P, P, NF, R, TE, MODE, IX, PML, NPART>(prm, F, part, us, gs, id, 3 * F * N, 3 * (1 - F) * N);
    } else {
        if (F == 0) tang_parts<P, PH, NF, R, TE, MODE, IX, PML, NPART>(prm, 0, part, us, gs, id, 0, 3 * N);
        else tang_parts<PH, P, NF, R, TE, MODE, IX, PML, NPART>(prm, 1, part, us, gs, id, 3 * N, 0);
    }
}

constexpr int CLW = 4;   // warps of a cluster's CTA

// barrier of all threads of the cluster; shared-memory writes before it, remote
// ones too, are visible after it
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

// IX: type of the element/column/row index arithmetic (uint32_t when every
// index of the plan fits, else int64_t).  MINB: resident CTAs per SM asked of
// the register allocator.  NG = 4: thread groups = faces (both fields), then
// (field, half of the rows); NG = 8: (face, field), then (field, quarter of the
// rows), the two fields of a face in the two halves of a warp (TE = 16) or in
// two neighbouring warps (TE = 32).
// CL = 8 (FP64 on small meshes): a tile of 32 columns takes the eight CTAs of a
// cluster, CTA = the thread group of the face items, four warps each.  An SM's FP64
// pipes work through a warp's instruction in 64 cycles, so that a launch lasts as
// long as its longest warp however few tiles there are: here a warp has a quarter
// of an item's face modes and a sixteenth of a field's rows.  Face values are
// written into every CTA's shared memory, and cluster barriers take the place of
// the CTA's.
template <int P, typename R, int TE, int NG, int MODE, typename IX, bool SIP, bool PML, bool MX, int MINB, int CL = 1>
__global__ void __launch_bounds__(CL > 1 ? TE * CLW : TE * NG, MINB) tang_kernel(const StageParams prm) {
    static_assert(CL == 1 || (CL == 8 && NG == CL && TE == 32 && sizeof(R) == 8 && !SIP && !MX), "cluster shape");
    static_assert((TE == 32 && (NG == 4 || NG == 8)) || (TE == 16 && NG == 8), "tile shape");
    static_assert(!(SIP || MX) || MODE == MODE_LSRK || MODE == MODE_RHS, "interior penalty and mixed-order modes");
    static_assert(!(MX && (SIP || PML)), "mixed orders: no penalty, no PML");
    constexpr int N = nmodes(P), NF = nfmodes(P);
    constexpr int PH = deg_h<P, MX>(), NH = nmodes(PH), NFH = nfmodes(PH), ROWS = field_rows<P, MX>();
    constexpr bool LF = MODE == MODE_LF_E || MODE == MODE_LF_H;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    R* us = reinterpret_cast<R*>(smem_raw);   // [ROWS][TE]
    R* gs = us + ROWS * TE;                   // [4][2][2][NF][TE]
    uint64_t* bar = reinterpret_cast<uint64_t*>(gs + 16 * NF * TE);

    const int c = threadIdx.x % TE;
    const int grp = CL > 1 ? int(blockIdx.x % CL) : threadIdx.x / TE;   // (CL: the rank in the cluster)
    const int sub = CL > 1 ? int(threadIdx.x / TE) : 0;                 // (CL: the warp in the CTA)
    const IX K = prm.K;
    const int S = prm.S;
    const IX x0 = IX(CL > 1 ? blockIdx.x / CL : tile_index(prm.tile_groups)) * TE;
    // no CTA writes into another's shared memory before all of the cluster run
    if constexpr (CL > 1) asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    Column<IX> id;
    id.C = K * S;
    id.col = x0 + c;
    // only the first K_active elements are updated; the others (halo copies of
    // another partition's elements) are read as neighbours
    id.active = id.col < IX(prm.K_active) * IX(S);
    id.e = id.active ? id.col / S : 0;
    id.s = id.active ? int(id.col - id.e * S) : 0;
    const IX C = id.C;
    const bool active = id.active;
    const R* u = static_cast<const R*>(prm.u);   // may alias u_out (leapfrog)
    auto coef = [&](double d, float f) { return sizeof(R) == 4 ? R(f) : R(d); };

    // What no earlier launch of the call writes: the face's code and constants
    const int f = NG == 4 ? grp : grp >> 1;
    const int half = NG == 4 ? 0 : grp & 1;      // field (leapfrog: tangent) of this thread when NG = 8
    auto table = [&](int row) -> R {
        const R* b = static_cast<const R*>(prm.fct) + IX(row) * K;
        return b[id.e];
    };
    const int32_t code = active ? prm.nbr[IX(f) * K + id.e] : -1;
    const R cE = table(f * TG_FACE + TG_CE), cH = table(f * TG_FACE + TG_CH);
    bulk::wait_previous_launch();

    // The tile: one bulk tensor copy of its rows where the plan has a
    // map of u (aligned rows), issued first and waited for by thread 0; columns
    // past the end arrive as zeros.
    const bool bulk = CL == 1 && prm.tm_u >= 0 && (tc::smem_addr(smem_raw) & 127u) == 0;
    if (bulk && threadIdx.x == 0) {
        static_assert(sizeof(R) * TE * ROWS < (1u << 20), "bytes of an mbarrier phase");
        tc::mbar_init(bar, 1);
        bulk::arrive_expect_tx(bar, uint32_t(sizeof(R)) * TE * ROWS);
        bulk::load_3d(us, static_cast<const char*>(prm.tmaps) + prm.tm_u * TMAP_BYTES, int(x0), 0, 0, bar);
    }
    // Otherwise every thread loads its rows: by asynchronous copies, all in flight at once,
    // in a cluster (whose CTAs all take the whole tile) and in the shapes of few tiles, else
    // in batches through registers, which follow one another, each a round trip, but
    // leave the L1 to the gathers (us, batches | copies: right-hand side p = 4, 16 tiles
    // 16.7 | 12.8; LSRK4 p = 5, 768 tiles in random order 203 | 222).  One of the two per
    // instantiation: the choice at run time cost the p = 3 kernel 7 percent.
    constexpr bool ASYNC = CL > 1 || (sizeof(R) == 4 && NG == 8 && TE == 32 && MINB <= 2 &&
                                      (MINB == 1 || P == 3 || (P == 4 && !SIP)));
    if (ASYNC && !bulk) {
        constexpr int STEP = CL > 1 ? CLW : NG;
        const int r0 = CL > 1 ? sub : grp;
        if (active) {
            const R* src = u + (IX(r0) * C + id.col);
            uint32_t dst = tc::smem_addr(us + r0 * TE + c);
#pragma unroll 8
            for (int q = r0; q < ROWS; q += STEP, src += IX(STEP) * C, dst += STEP * TE * uint32_t(sizeof(R)))
                asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" :: "r"(dst), "l"(src), "n"(sizeof(R)) : "memory");
        } else {
            for (int q = r0; q < ROWS; q += STEP) us[q * TE + c] = R(0);
        }
    }
    // ---- phase A: jumps and fluxes of one face -----------------------------------
    const bool bad = code >= 0 && IX(code >> 2) >= K;
    if (bad) atomicOr(prm.status, int32_t(ST_BAD_NEIGHBOUR));
    const bool has = code >= 0 && !bad;
    const int nf = code & 3;                                    // the neighbour's local face
    const IX nc = has ? IX(code >> 2) * S + id.s : 0;           // the neighbour's column
    // items q = 2 field + tangent of this thread
    constexpr int QF = MODE == MODE_LF_E ? 2 : 0;              // leapfrog: only the other field's jumps
    constexpr int QN = LF ? (NG == 4 ? 2 : 1) : (NG == 4 ? 4 : 2);
    const int q0 = QF + (NG == 4 ? 0 : half * QN);
    // ALL: registers for the gathers of both items at once, one round trip instead of two
    // to four (a slanted neighbour face's component 0 serves both)
    constexpr bool ALL = sizeof(R) == 4 && NG == 8 && TE == 32 && MINB == 1;
    constexpr bool AHEAD = ALL || P <= 3 || (P == 4 && PML);   // gathers of a slanted neighbour face in two register sets
    R vn[N], vm[AHEAD ? N : 1], vx[ALL && QN == 2 ? N : 1];
    // first field row of component `comp` of a field
    auto row_of = [&](int fld, int comp) { return fld == 0 ? comp * N : 3 * N + comp * NH; };
    auto fetch = [&](int fld, int comp, R* v) {   // the neighbour's coefficients of one component
        const R* p = u + (IX(row_of(fld, comp)) * C + nc);
        if (!MX || fld == 0) {
#pragma unroll
            for (int l = 0; l < N; ++l) v[l] = p[IX(l) * C];
        } else {
#pragma unroll
            for (int l = 0; l < NH; ++l) v[l] = p[IX(l) * C];
        }
    };
    auto gather = [&](int q) {
        if (!has) return;
        fetch(q >> 1, tang_comp(nf, q & 1), vn);
        if constexpr (AHEAD) {
            if (nf == 0) fetch(q >> 1, 0, vm);
        }
    };
    gather(q0);
    if constexpr (ALL && QN == 2) {
        if (has) fetch(q0 >> 1, tang_comp(nf, 1), vx);
    }
    if (bulk) {
        bool ok = true;
        if (threadIdx.x == 0) ok = tc::mbar_wait(bar, 0, 500000000ull);
        if (!__syncthreads_and(ok)) {
            // the copy did not complete in time: latch the status, give it a
            // second bounded wait (the shared memory stays this CTA's until its
            // last thread exits) and leave the tile untouched
            if (threadIdx.x == 0) {
                atomicOr(prm.status, int32_t(ST_TIMEOUT));
                tc::mbar_wait(bar, 0, 500000000ull);
            }
            return;
        }
    } else if constexpr (ASYNC) {
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        if constexpr (CL > 1) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    } else {
        constexpr int UR = (ROWS + NG - 1) / NG, BATCH = UR < 16 ? UR : 16;
#pragma unroll 1
        for (int i0 = 0; i0 < UR; i0 += BATCH) {
            R tmp[BATCH];
#pragma unroll
            for (int i = 0; i < BATCH; ++i) {
                const int q = grp + (i0 + i) * NG;
                tmp[i] = (active && q < ROWS) ? u[IX(q) * C + id.col] : R(0);
            }
#pragma unroll
            for (int i = 0; i < BATCH; ++i) {
                const int q = grp + (i0 + i) * NG;
                if (q < ROWS) us[q * TE + c] = tmp[i];
            }
        }
        __syncthreads();
    }
    R* gf = gs + f * 4 * NF * TE + c;   // this face's rows: [field][tangent][NF]
    // a face value into the shared memory of the cluster's ranks lo .. lo + n - 1
    const uint32_t sbase = tc::smem_addr(smem_raw);
    uint32_t rbase[CL];
    if constexpr (CL > 1) {
#pragma unroll
        for (int r = 0; r < CL; ++r) asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rbase[r]) : "r"(sbase), "r"(r));
    }
    auto put = [&](R* o, R v, bool pair) {
        if constexpr (CL > 1) {
            const uint32_t off = tc::smem_addr(o) - sbase;
#pragma unroll
            for (int r = 0; r < CL; ++r)
                if (!pair || r / 2 == f)   // pair: the two ranks of this face
                    asm volatile("st.shared::cluster.f64 [%0], %1;" :: "r"(rbase[r] + off), "d"(double(v)) : "memory");
        } else {
            *o = v;
        }
    };
    const bool inc = code <= -2 && prm.inc != nullptr;
    // jump of item q of a field of degree PF: own trace, then the neighbour's
    // (CL: modes of quarter `mq` only; the arithmetic of the others falls away)
    auto item = [&](auto deg, int q, auto mq) {
        constexpr int part = decltype(mq)::value;
        constexpr int PF = decltype(deg)::value, NP = nmodes(PF), NPF = nfmodes(PF);
        const int fld = q >> 1, i = q & 1;
        const R* v0 = us + row_of(fld, 0) * TE + c;
        R acc[NPF];
        own_trace<PF, R, TE>(f, v0 + tang_comp(f, i) * NP * TE, v0, acc);
        if (has) {
            R(&w)[NP] = *reinterpret_cast<R(*)[NP]>(vn);
            if (nf == 0) {   // slanted neighbour face: less component 0
                if constexpr (AHEAD) {
#pragma unroll
                    for (int l = 0; l < NP; ++l) w[l] -= vm[l];
                } else {
                    const R* p0 = u + (IX(row_of(fld, 0)) * C + nc);
#pragma unroll
                    for (int l = 0; l < NP; ++l) w[l] -= p0[IX(l) * C];
                }
            }
            jump_trace<PF, R>(nf, w, acc);
        } else {
            // boundary face, acc = -own: PEC (e+ = -e-, h+ = h-) or incident
            // (e+ = e- + 2 E_inc, h+ = -h-; the E_inc part is added with the flux)
            const R al = ((fld == 0) != inc) ? R(2) : R(0);
#pragma unroll
            for (int m = 0; m < NPF; ++m) acc[m] *= al;
        }
        // central flux of the leapfrog: gamma_1 = c tau_2, gamma_2 = -c tau_1 of the other field
        const R cc = LF ? (MODE == MODE_LF_E ? cE : cH) * R(i ? 1 : -1) : R(1);
        R* o = gf + (LF ? 2 * (1 - fld) + 1 - i : q) * NF * TE;
#pragma unroll
        for (int m = 0; m < NPF; ++m) {
            if (CL > 1 && m * CLW / NPF != part) continue;
            if constexpr (LF) put(o + m * TE, cc * acc[m], false);
            else put(o + m * TE, acc[m], true);   // both threads of the face
        }
    };
#pragma unroll 1
    for (int k = 0; k < QN; ++k) {
        const int q = q0 + k;
        auto quarter = [&](auto mq) {
            if (!MX || (q >> 1) == 0) item(std::integral_constant<int, P>{}, q, mq);
            else item(std::integral_constant<int, PH>{}, q, mq);
        };
        if constexpr (CL > 1) {
            switch (sub) {
                case 0: quarter(std::integral_constant<int, 0>{}); break;
                case 1: quarter(std::integral_constant<int, 1>{}); break;
                case 2: quarter(std::integral_constant<int, 2>{}); break;
                default: quarter(std::integral_constant<int, 3>{}); break;
            }
        } else {
            quarter(std::integral_constant<int, 0>{});
        }
        if constexpr (ALL && QN == 2) {
#pragma unroll
            for (int l = 0; l < N; ++l) vn[l] = vx[l];
        } else {
            if (k + 1 < QN) gather(q + 1);
        }
    }
    if constexpr (!LF) {
        // fluxes in place; with NG = 8 the face's two threads split the modes
        // and first wait for each other's jumps
        if constexpr (CL > 1) {
            cluster_sync();
        } else if (NG == 8) {
            if (TE == 16) __syncwarp();
            else asm volatile("bar.sync %0, 64;" :: "r"(1 + f) : "memory");
        }
        constexpr int MH = NG == 8 ? NF / 2 : NF;
        const int m0 = half * MH, m1 = (NG == 8 && half == 0) ? MH : NF;
        const R e11 = table(f * TG_FACE + TG_E11), ne12 = table(f * TG_FACE + TG_NE12), e22 = table(f * TG_FACE + TG_E22);
        const R nh11 = table(f * TG_FACE + TG_NH11), h12 = table(f * TG_FACE + TG_H12), nh22 = table(f * TG_FACE + TG_NH22);
        const R ncE = cE * R(-1), ncH = cH * R(-1);
        // incident jump terms of this face: covariant components [NF][3]
        const R* ic = inc ? static_cast<const R*>(prm.inc) + IX(-code - 2) * NF * 3 : nullptr;
        // interior penalty: this column's facet field on face f (and, on the
        // owner side, its output and residual), [3][NF][facet][S]
        const R* hsv = nullptr;
        R *hso = nullptr, *hsr = nullptr;
        R T1[3], T2[3], ks = R(0);
        const int64_t fs = int64_t(prm.n_facets) * S;
        const R ca = coef(prm.a, prm.a_f), cb = coef(prm.b, prm.b_f), dt = coef(prm.dt, prm.dt_f);
        const R sig = (f & 1) ? R(1) : R(-1);
        if constexpr (SIP) {
            const int32_t sf = active ? prm.sfid[IX(f) * K + id.e] : -1;
            if (sf >= 0) {
                const int64_t off = int64_t(sf >> 1) * S + id.s;
                hsv = static_cast<const R*>(prm.hs) + off;
                if (sf & 1) {
                    hso = static_cast<R*>(prm.hs_out) + off;
                    hsr = MODE == MODE_LSRK ? static_cast<R*>(prm.hs_res) + off : nullptr;
                }
            }
            const R* ts = static_cast<const R*>(prm.fcp) + IX(f * TG_SIPF) * K + id.e;
            ks = ts[0];
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                T1[r] = ts[IX(1 + r) * K];
                T2[r] = ts[IX(4 + r) * K];
            }
        }
        // the modes in chunks, so that a chunk's facet values arrive together
        constexpr int MC = SIP ? (NF + 3) / 4 : 1, MSTEP = CL > 1 ? CLW : MC;
#pragma unroll(SIP ? 1 : (P <= 3 ? 10 : 3))
        for (int mb = m0 + sub; mb < m1; mb += MSTEP) {
            R hv[SIP ? MC : 1][3], hr[SIP ? MC : 1][3];
            if constexpr (SIP) {
#pragma unroll
                for (int j = 0; j < MC; ++j)
#pragma unroll
                    for (int r = 0; r < 3; ++r) {
                        const int64_t o = int64_t(r * NF + mb + j) * fs;
                        hv[j][r] = (hsv != nullptr && mb + j < m1) ? hsv[o] : R(0);
                        hr[j][r] = (MODE == MODE_LSRK && hsr != nullptr && mb + j < m1) ? hsr[o] : R(0);
                    }
            }
#pragma unroll
            for (int j = 0; j < MC; ++j) {
                const int m = mb + j;
                if (SIP && m >= m1) break;
                R* o = gf + m * TE;
                const bool hm = !MX || m < NFH;   // a mode of H's traces
                R e1 = o[0], e2 = o[NF * TE];
                const R h1 = hm ? o[2 * NF * TE] : R(0), h2 = hm ? o[3 * NF * TE] : R(0);
                if (ic != nullptr) {
                    const R z = f == 0 ? ic[3 * m] : R(0);
                    e1 += ic[3 * m + tang_comp(f, 0)] - z;
                    e2 += ic[3 * m + tang_comp(f, 1)] - z;
                }
                R p1 = fmaa(cE, h2, fmaa(e22, e1, ne12 * e2));
                R p2 = fmaa(ncE, h1, fmaa(e11, e2, ne12 * e1));
                if (hm) {
                    put(o + 2 * NF * TE, fmaa(cH, e2, fmaa(h12, h2, nh22 * h1)), false);
                    put(o + 3 * NF * TE, fmaa(ncH, e1, fmaa(h12, h1, nh11 * h2)), false);
                }
                if constexpr (SIP) {
                    // both sides: gamma += m_f x (A^T h_s); owner: dh_s/dt =
                    // -ks A (m_f x de) = -ks sigma (A t_1 de_2 - A t_2 de_1)
                    if (hsv != nullptr) {
                        p1 += sig * (T2[0] * hv[j][0] + T2[1] * hv[j][1] + T2[2] * hv[j][2]);
                        p2 -= sig * (T1[0] * hv[j][0] + T1[1] * hv[j][1] + T1[2] * hv[j][2]);
                    }
                    if (hso != nullptr) {
#pragma unroll
                        for (int r = 0; r < 3; ++r) {
                            const R d = -ks * sig * (T1[r] * e2 - T2[r] * e1);
                            const int64_t oo = int64_t(r * NF + m) * fs;
                            if (MODE == MODE_RHS) {
                                hso[oo] = d;
                            } else {
                                const R rr = ca * hr[j][r] + dt * d;
                                hsr[oo] = rr;
                                hso[oo] = hv[j][r] + cb * rr;
                            }
                        }
                    }
                }
                put(o, p1, false);
                put(o + NF * TE, p2, false);
            }
        }
    }
    if constexpr (CL > 1) cluster_sync();
    else __syncthreads();

    // ---- phase B: curl, lift, mass block, update ----------------------------------
    if constexpr (LF) {
        // one field.  At p = 5 (eight groups) eight row parts with a layer, four without one,
        // half of the groups idle: of eight every one repeats the curl's reads of the
        // tile (us per half step, four | eight parts: 137 tiles with a PML 41.4 | 37.5; 999 tiles
        // without 87 | 92).
        constexpr int F = MODE == MODE_LF_E ? 0 : 1;
        constexpr int G = CL > 1 ? 16 : P == 5 && !PML ? 4 : NG, NPB = N < G ? N : G;
        if (const int part = CL > 1 ? sub * CL + grp : grp; part < NPB)
            tang_part<P, R, TE, MODE, IX, PML, MX, NPB>(prm, F, part, us + c, gs + c, id);
    } else if constexpr (CL > 1) {
        constexpr int NPB = N < 16 ? N : 16;
        if (const int part = sub * 4 + (grp >> 1); part < NPB)
            tang_part<P, R, TE, MODE, IX, PML, MX, NPB>(prm, grp & 1, part, us + c, gs + c, id);
    } else if constexpr (NG == 4) {
        constexpr bool BAL = tang_balance<P, R, PML>() && !MX;
        const int F = BAL ? grp >> 1 : grp & 1;
        const int part = BAL ? (grp == 1 || grp == 2 ? 0 : 1) : grp >> 1;
        tang_part<P, R, TE, MODE, IX, PML, MX, 2>(prm, F, part, us + c, gs + c, id);
    } else {
        tang_part<P, R, TE, MODE, IX, PML, MX, 4>(prm, grp & 1, grp >> 1, us + c, gs + c, id);
    }
}

}  // namespace dgm
