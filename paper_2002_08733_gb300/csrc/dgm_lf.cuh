// Leapfrog half step of FP32 plans for receivers, on reference-frame traces.
//
// Those plans keep the rounding of stage_kernel (dgm_stage.cuh): receiver
// records are FP64 results formed from FP32 fields.  So every value here is the
// same chain of operations as in stage_kernel, with what a half step does not
// need left out: it advances one field from the jumps of the other, the flux is
// central, no face is incident (those need LSRK4), and the advanced field enters by its
// own rows only.
//
// One CTA owns TE consecutive columns, NG = 12 threads per column:
//   1  tile of the other field; neighbour trace of item (face, component);
//   2  own trace of the same item;
//   3  flux of item (face, third of the face modes), in place of the own traces;
//   4  curl and lift of item (component, quarter of the rows);
//   5  mass block, PML terms and update of one twelfth of the rows, which were
//      requested before phase 4.
// Each phase has twelve items (nine in 2), one per thread group, and shared memory
// holds one field's traces.  As a mode of stage_kernel the half step gave six of
// its twelve groups nothing to do in phases 1, 2, 4 and 5 and held both fields'
// traces, so that one CTA filled an SM at p = 4 (132 KB; 63 KB now, two CTAs): 252 us
// per half step of 82,944 elements with a PML then, 127 us now (25 us at the measured
// HBM rate; latency of the gathers and of the five barriers bounds it).
#pragma once

#include "dgm_bulk.cuh"
#include "dgm_stage.cuh"

namespace dgm {

constexpr int LF_NG = 12;   // threads per column

template <int P, typename R, int TE>
__host__ __device__ constexpr size_t lf_smem_bytes() {
    return sizeof(R) * size_t(TE) * (3 * nmodes(P) + 24 * nfmodes(P) + EG + GM);
}

template <int P, typename R, int TE, int MODE, typename IX>
__global__ void __launch_bounds__(TE * LF_NG, 2) lf_kernel(const StageParams prm) {
    static_assert(MODE == MODE_LF_E || MODE == MODE_LF_H, "leapfrog half steps");
    constexpr int N = nmodes(P), NF = nfmodes(P), NG = LF_NG;
    constexpr int F = MODE == MODE_LF_E ? 0 : 1, O = 1 - F;   // field advanced, field it reads
    extern __shared__ __align__(16) unsigned char smem_raw[];
    R* us = reinterpret_cast<R*>(smem_raw);      // [3N][TE] the other field
    R* trO = us + 3 * N * TE;                    // [4][3][NF][TE] own traces -> g
    R* trN = trO + 12 * NF * TE;                 // [4][3][NF][TE] neighbour traces -> rhs [3][N][TE]
    R* eg = trN + 12 * NF * TE;                  // [EG][TE]
    R* gm = eg + EG * TE;                        // [GM][TE] metric A^T A
    static_assert(N <= 4 * NF, "the right-hand side fits in the neighbour-trace array");

    const int c = threadIdx.x % TE;
    const int grp = threadIdx.x / TE;
    const IX K = prm.K;
    const int S = prm.S;
    const IX C = K * S;
    const IX col = IX(tile_index(prm.tile_groups)) * TE + c;
    const bool active = col < IX(prm.K_active) * IX(S);   // others: halo copies, read as neighbours
    const IX e = active ? col / S : 0;
    const int s = active ? int(col - e * S) : 0;
    const R* u = static_cast<const R*>(prm.u);   // aliases u_out
    const R* gr = static_cast<const R*>(prm.geo_r);
    const R* fcp = static_cast<const R*>(prm.fcp);

    // ---- phase 1: tile, element constants, neighbour traces ----------------------
    const int f = grp / 3, k = grp % 3;          // trace item: face, component
    const int32_t code = active ? prm.nbr[IX(f) * K + e] : -1;
    const bool bad = code >= 0 && IX(code >> 2) >= K;
    if (bad) atomicOr(prm.status, int32_t(ST_BAD_NEIGHBOUR));
    const bool has = code >= 0 && !bad;
    // this thread's flux item (face, third of the modes): its constants
    const int ff = grp / 3, ch = grp % 3;
    R q[9], na = R(0), cc = R(0);
    auto face_const = [&](int r) { return active ? fcp[IX(ff * FGR + r) * K + e] : R(0); };
#pragma unroll
    for (int i = 0; i < 9; ++i) q[i] = face_const(FR_Q + i);
    na = face_const(O == 0 ? FR_NAE : FR_NAH);
    cc = face_const(F == 0 ? FR_CE : FR_CH);
    bulk::wait_previous_launch();
    {
        R vn[N];
        if (has) {
            const R* p = u + (IX((3 * O + k) * N) * C + (IX(code >> 2) * S + s));
#pragma unroll
            for (int l = 0; l < N; ++l) vn[l] = p[IX(l) * C];
        }
        constexpr int T1 = 3 * N + EG + GM, UR = (T1 + NG - 1) / NG;
        R tmp[UR];
#pragma unroll
        for (int i = 0; i < UR; ++i) {
            const int q = grp + i * NG;
            tmp[i] = R(0);
            if (!active || q >= T1) continue;
            tmp[i] = q < 3 * N        ? u[IX(3 * O * N + q) * C + col]
                     : q < 3 * N + EG ? gr[IX(q - 3 * N) * K + e]
                                      : fcp[IX(4 * FGR + q - 3 * N - EG) * K + e];
        }
#pragma unroll
        for (int i = 0; i < UR; ++i) {
            const int q = grp + i * NG;
            if (q < 3 * N) us[q * TE + c] = tmp[i];
            else if (q < T1) eg[(q - 3 * N) * TE + c] = tmp[i];   // (gm follows eg)
        }
        R acc[NF];
        if (has) {
            trace_any<P, R>(code & 3, vn, acc);
        } else {
#pragma unroll
            for (int m = 0; m < NF; ++m) acc[m] = R(0);
        }
#pragma unroll
        for (int m = 0; m < NF; ++m) trN[((f * 3 + k) * NF + m) * TE + c] = acc[m];
    }
    __syncthreads();

    // ---- phase 2: own traces (the flux on face a + 1 does not use component a) ---
    if (f != k + 1) {
        R v[N], acc[NF];
#pragma unroll
        for (int l = 0; l < N; ++l) v[l] = us[(k * N + l) * TE + c];
        trace_any<P, R>(f, v, acc);
#pragma unroll
        for (int m = 0; m < NF; ++m) trO[((f * 3 + k) * NF + m) * TE + c] = acc[m];
    }
    __syncthreads();

    // ---- phase 3: central flux g = +-c (m_f x jump of the other field) ------------
    {
        const R cs = F == 0 ? cc : -cc;
        const int ax = ff - 1;                   // axis of m_f = -e_A; -1 on the slanted face
        for (int m = ch * NF / 3; m < (ch + 1) * NF / 3; ++m) {
            R* own = trO + (ff * 3 * NF + m) * TE + c;
            const R* nbt = trN + (ff * 3 * NF + m) * TE + c;
            R d[3], tp[3];
#pragma unroll
            for (int r = 0; r < 3; ++r) tp[r] = nbt[r * NF * TE];
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                d[r] = R(0);
                if (r == ax) continue;
                d[r] = q[3 * r] * tp[0] + q[3 * r + 1] * tp[1] + q[3 * r + 2] * tp[2] + na * own[r * NF * TE];
            }
            // m_f = (1, 1, 1): m x y = (y2 - y1, y0 - y2, y1 - y0); m_f = -e_A:
            // (m x y)_A = 0 (not stored), (m x y)_B = y_CC, (m x y)_CC = -y_B, (A, B, CC) cyclic
            if (ax < 0) {
                own[0] = cs * (d[2] - d[1]);
                own[NF * TE] = cs * (d[0] - d[2]);
                own[2 * NF * TE] = cs * (d[1] - d[0]);
            } else if (ax == 0) {
                own[NF * TE] = cs * d[2];
                own[2 * NF * TE] = -cs * d[1];
            } else if (ax == 1) {
                own[2 * NF * TE] = cs * d[0];
                own[0] = -cs * d[2];
            } else {
                own[0] = cs * d[1];
                own[NF * TE] = -cs * d[0];
            }
        }
    }
    // the rows this thread updates in phase 5, requested before phase 4
    constexpr int NP = NG < N ? NG : N, RP = (N + NP - 1) / NP;   // row parts, rows of one (at most)
    const int lo = grp * N / NP, hi = (grp + 1) * N / NP;
    const bool upd = active && grp < NP;
    const IX gb = IX(3 * F * N + lo) * C + col;
    const int32_t pi = upd && prm.pml != nullptr ? prm.pml[e] : -1;
    R uv[RP][3];
#pragma unroll
    for (int i = 0; i < RP; ++i)
#pragma unroll
        for (int r = 0; r < 3; ++r) uv[i][r] = (upd && lo + i < hi) ? u[gb + IX(r * N + i) * C] : R(0);
    __syncthreads();

    // ---- phase 4: volume curl + lift per (component, quarter of the rows) ---------
    R* rh = trN;
    {
        const int j = grp % 3, part = grp / 3;
        const R sgn = eg[G_DET * TE + c] < R(0) ? R(-1) : R(1);
        R acc[N];
        rhs_part<P, R, TE, 4, 3>(part, 3 * F + j, c, us, trO, sgn, acc);
        const int l0 = part * N / 4, l1 = (part + 1) * N / 4;
        if (F == 0 && prm.src != nullptr && active) {
            const double* rec = prm.src + IX(s) * (SRC_HDR + 3 * N);
            if (rec[0] >= 0.0 && IX(rec[0]) == e) {   // -1 marks a column without a source
                const double tt = prm.tdev ? *prm.tdev + prm.t : prm.t;
                const R g = R(source_time(tt, rec[1], rec[2], rec[3]));
#pragma unroll
                for (int l = 0; l < N; ++l)
                    if (l >= l0 && l < l1) acc[l] -= g * R(rec[SRC_HDR + j * N + l]);
            }
        }
#pragma unroll
        for (int l = 0; l < N; ++l)
            if (l >= l0 && l < l1) rh[(j * N + l) * TE + c] = acc[l];
    }
    __syncthreads();

    // ---- phase 5: mass block, PML, update ------------------------------------------
    if (!upd) return;
    const R det = eg[G_DET * TE + c];
    const R mat = eg[(G_EPS + F) * TE + c];
    R B[3][3];
    const R inv = R(1) / (mat * fabs(det));
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int t = r; t < 3; ++t) {
            B[r][t] = inv * gm[sym3(r, t) * TE + c];
            B[t][r] = B[r][t];
        }
    const R dt = sizeof(R) == 4 ? R(prm.dt_f) : R(prm.dt);
    R* uo = static_cast<R*>(prm.u_out);
    auto mass = [&](int i, R (&du)[3]) {
        R r[3];
#pragma unroll
        for (int t = 0; t < 3; ++t) r[t] = rh[(t * N + lo + i) * TE + c];
#pragma unroll
        for (int t = 0; t < 3; ++t) du[t] = B[t][0] * r[0] + B[t][1] * r[1] + B[t][2] * r[2];
    };
    if (pi < 0) {
#pragma unroll
        for (int i = 0; i < RP; ++i) {
            if (lo + i >= hi) break;
            R du[3];
            mass(i, du);
#pragma unroll
            for (int t = 0; t < 3; ++t) uo[gb + IX(t * N + i) * C] = uv[i][t] + dt * du[t];
        }
        return;
    }
    // The PML terms by the trapezoid rule, per Cartesian component in the physical
    // frame X = A^-T x:
    //   X_new = ((1 - dt eta/2) X + dt (A^-T du - A^-T aux / mat)) / (1 + dt eta/2)
    // with aux this field's auxiliary; then the other field's auxiliary,
    //   Z_new = gamma Z + dt beta mat' xi Y,  beta = 1/(1 + dt sigma/2),
    //   gamma = (1 - dt sigma/2) beta,  Y = A^-T (other field), mat' its material.
    R ait[9], AT[3][3];
#pragma unroll
    for (int i = 0; i < 9; ++i) ait[i] = eg[(G_AIT + i) * TE + c];
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
    const R sx = eg[(G_SIG + 0) * TE + c], sy = eg[(G_SIG + 1) * TE + c], sz = eg[(G_SIG + 2) * TE + c];
    const R sg3[3] = {sx, sy, sz};
    const R et3[3] = {sy + sz - sx, sz + sx - sy, sx + sy - sz};
    const R xi3[3] = {(sx - sy) * (sx - sz), (sy - sz) * (sy - sx), (sz - sx) * (sz - sy)};
    const R imat = R(1) / mat;
    const R omat = eg[(G_EPS + O) * TE + c];
    const IX C2 = IX(prm.npml) * S;
    const IX acol = IX(pi) * S + s;
    const IX ab = IX(3 * F * N + lo) * C2 + acol;    // this field's rows in the auxiliaries
    const IX abo = IX(3 * O * N + lo) * C2 + acol;   // the other field's
    R* auxl = static_cast<R*>(prm.aux_out);          // in place: aux_out == aux
    // all auxiliary rows requested before the arithmetic
    R av[RP][3], oa[RP][3];
#pragma unroll
    for (int i = 0; i < RP; ++i)
#pragma unroll
        for (int t = 0; t < 3; ++t) {
            const bool ok = lo + i < hi;
            av[i][t] = ok ? auxl[ab + IX(t * N + i) * C2] : R(0);
            oa[i][t] = ok ? auxl[abo + IX(t * N + i) * C2] : R(0);
        }
#pragma unroll
    for (int i = 0; i < RP; ++i) {
        if (lo + i >= hi) break;
        R du[3], ov[3], Xn[3], Zn[3];
        mass(i, du);
#pragma unroll
        for (int t = 0; t < 3; ++t) ov[t] = us[(t * N + lo + i) * TE + c];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const R x = ait[3 * a] * uv[i][0] + ait[3 * a + 1] * uv[i][1] + ait[3 * a + 2] * uv[i][2];
            const R y = ait[3 * a] * du[0] + ait[3 * a + 1] * du[1] + ait[3 * a + 2] * du[2];
            const R z = ait[3 * a] * av[i][0] + ait[3 * a + 1] * av[i][1] + ait[3 * a + 2] * av[i][2];
            const R hd = R(0.5) * dt * et3[a];
            Xn[a] = ((R(1) - hd) * x + dt * (y - z * imat)) / (R(1) + hd);
            const R yo = ait[3 * a] * ov[0] + ait[3 * a + 1] * ov[1] + ait[3 * a + 2] * ov[2];
            const R zo = ait[3 * a] * oa[i][0] + ait[3 * a + 1] * oa[i][1] + ait[3 * a + 2] * oa[i][2];
            const R beta = R(1) / (R(1) + R(0.5) * dt * sg3[a]);
            const R gamma = (R(1) - R(0.5) * dt * sg3[a]) * beta;
            Zn[a] = gamma * zo + dt * beta * omat * xi3[a] * yo;
        }
#pragma unroll
        for (int t = 0; t < 3; ++t) {
            uo[gb + IX(t * N + i) * C] = AT[t][0] * Xn[0] + AT[t][1] * Xn[1] + AT[t][2] * Xn[2];
            auxl[abo + IX(t * N + i) * C2] = AT[t][0] * Zn[0] + AT[t][1] * Zn[1] + AT[t][2] * Zn[2];
        }
    }
}

}  // namespace dgm
