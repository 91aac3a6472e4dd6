// FP32 deviation storage of the FE-LBM step (included by felbm.cu).
//
// The state is split into the macroscopic fields -- C in FP64, p and u in
// FP32 -- and the FP32 deviations of the distributions from their
// equilibria, dpsi_a = psi_a - psi_a^eq(C, p, u), whose zeroth (and, for g,
// first) moments are zero.  The scheme is the same as the FP64 path
// (Sec. II.C of arXiv:1708.04678); only the storage and arithmetic differ:
//  * collision needs no pass of its own: psi_hat = psi^eq + (1 - omega) dpsi;
//  * every gradient and every difference of equilibria is formed from
//    differences of the fields (C differences taken in FP64), so nothing
//    cancels catastrophically in FP32 -- e.g. h^eq_v - h^eq_0 =
//    Gamma_v (C_v - C_0) + C_0 (Gamma_v - Gamma_0), and Gamma_v - Gamma_0 is
//    a polynomial in u_v - u_0;
//  * the chemical potential (double well near C in {0, 1} and the patch
//    Laplacian of C) is evaluated in FP64;
//  * the mass solve runs in FP32 and its last sweep updates the fields (C in
//    FP64) and the deviations in place.
#pragma once

// The deviations are stored in the planes of vec_at: consecutive vertices of
// consecutive triangles are consecutive 16-byte words, so a warp's gather of a
// plane touches 3 or 4 lines.  With one 64-byte row per node each 16-byte load
// of a warp touched 16.

// omega = 1 / (tau + 1/2), 1/tau = C/tau_l + (1-C)/tau_v (Sec. II.A)
__device__ __forceinline__ float omega32(float C, const Phys& c) {
    float inv_tau = C * c.inv_tau_l_f + (1.0f - C) * c.inv_tau_v_f;
    return 1.0f / (1.0f / inv_tau + 0.5f);
}

// Gamma_q(u1) - Gamma_q(u0) as a polynomial in du = u1 - u0, su = u1 + u0.
template <int q>
__device__ __forceinline__ float dgamma32(float dux, float duy, float sux, float suy) {
    float edu = edot<q, float>(dux, duy), esu = edot<q, float>(sux, suy);
    return (float)wq(q) * (3.0f * edu + 4.5f * edu * esu - 1.5f * (dux * sux + duy * suy));
}
template <int q>
__device__ __forceinline__ float gamma32(float ux, float uy, float uu15) {
    float eu = edot<q, float>(ux, uy);
    return (float)wq(q) * (1.0f + 3.0f * eu + 4.5f * eu * eu - uu15);
}

// ------------------------------------------------- chemical potential ------
// The terms of k_mu (FP64), the Laplacian as differences to C_i; FP32 output.
__device__ __forceinline__ void mu32_node(const DevMesh& m, const Phys& c, const Bufs& b, int i) {
    double Ci = b.C[i];
    double lap = 0.0;
    for (int k = m.row_ptr[i]; k < m.row_ptr[i + 1]; ++k) lap += m.lval[k] * (b.C[m.col[k]] - Ci);
    double wall = 0.0;
    for (int k = m.winc_ptr[i]; k < m.winc_ptr[i + 1]; ++k) {
        int e = m.winc_edge[k];
        double Ca = b.C[m.wall_a[e]], Cb = b.C[m.wall_b[e]];
        double s = 0.5 * (Ca + Cb) - (Ca * Ca + Ca * Cb + Cb * Cb) * (1.0 / 3.0);
        wall -= m.wall_phi[e] * m.wall_len[e] * s;
    }
    b.mu32[i] = (float)(2.0 * c.beta * Ci * (Ci - 1.0) * (2.0 * Ci - 1.0) - (c.kappa * lap + wall * m.inv_vol[i]));
}

// kW > 0: the sum over the ELL copy of the row (zero padding), its columns
// and coefficients loaded up front so the gathers of C are issued together;
// kW = 0: CSR, in the difference form of the FP64 path.
template <int kW>
__global__ void __launch_bounds__(kBlock) k_mu32(DevMesh m, Phys c, Bufs b) {
    pdl_release();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m.N) return;
    if constexpr (kW == 0) {
        mu32_node(m, c, b, i);
    } else {
        const int Np = m.Np;
        int col[kW];
        double l[kW];
#pragma unroll
        for (int k = 0; k < kW; ++k) {
            col[k] = m.ell_col[k * Np + i];
            l[k] = m.ell_lval[k * Np + i];
        }
        // The row's coefficients sum to zero (the P1 stiffness rows do), so
        // sum l_k (C_k - C_i) = sum l_k C_k: one FP64 FMA per entry instead
        // of a subtraction and an FMA on this FP64-pipe-bound kernel.  The
        // cancellation costs about 1e-15 absolute in the Laplacian, far below
        // the FP32 rounding of the stored mu.
        const double Ci = b.C[i];
        double lap = 0.0;
#pragma unroll
        for (int k = 0; k < kW; ++k) lap = fma(l[k], b.C[col[k]], lap);
        // 2 beta C (C - 1)(2 C - 1) - kappa lap in five FP64 operations; the wall
        // flux only where there is one: 68 us on 2,082,816 nodes, 71 us with nine
        double mu = fma(Ci * (Ci - 1.0), fma(4.0 * c.beta, Ci, -2.0 * c.beta), -c.kappa * lap);
        const int w0 = m.winc_ptr[i], w1 = m.winc_ptr[i + 1];
        if (w0 < w1) {
            double wall = 0.0;
            for (int k = w0; k < w1; ++k) {
                int e = m.winc_edge[k];
                double Ca = b.C[m.wall_a[e]], Cb = b.C[m.wall_b[e]];
                double s = 0.5 * (Ca + Cb) - (Ca * Ca + Ca * Cb + Cb * Cb) * (1.0 / 3.0);
                wall -= m.wall_phi[e] * m.wall_len[e] * s;
            }
            mu -= wall * m.inv_vol[i];
        }
        b.mu32[i] = (float)mu;
    }
}

__device__ __forceinline__ void gradmu32_tri(const DevMesh& m, const Bufs& b, int t) {
    const int Tp = m.Tp;
    int v0 = m.tri[t], v1 = m.tri[Tp + t], v2 = m.tri[2 * Tp + t];
    float m0 = b.mu32[v0], d1 = b.mu32[v1] - m0, d2 = b.mu32[v2] - m0;
    b.gmu32[t] = d1 * m.grad32[2 * Tp + t] + d2 * m.grad32[4 * Tp + t];
    b.gmu32[Tp + t] = d1 * m.grad32[3 * Tp + t] + d2 * m.grad32[5 * Tp + t];
}

// FELBM_LAPMU_NODAL: nodal Laplacian of mu (patch Laplacian with zero wall
// flux), formed in FP64 from the FP32 mu like the Laplacian of C.
__device__ __forceinline__ void lmu32_node(const DevMesh& m, const Phys& c, const Bufs& b, int i) {
    const double mi = b.mu32[i];
    double lap = 0.0;
    for (int k = m.row_ptr[i]; k < m.row_ptr[i + 1]; ++k) lap += m.lval[k] * ((double)b.mu32[m.col[k]] - mi);
    b.lmu32[i] = (float)(c.lapmu_fac * lap);
}

__global__ void __launch_bounds__(kBlock) k_lmu32(DevMesh m, Phys c, Bufs b) {
    pdl_release();
    pdl_wait();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < m.N) lmu32_node(m, c, b, i);
}

__global__ void __launch_bounds__(kBlock) k_gradmu32(DevMesh m, Bufs b) {
    pdl_release();
    pdl_wait();
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < m.T) gradmu32_tri(m, b, t);
}

// ------------------------------- forces and element residual (FP32) ------
// R_a = A (Phi_a - e_a . grad psi_hat_a), psi_hat = psi^eq + (1 - omega) dpsi,
// gradients formed from differences to vertex 0 (sum of the b_v is zero).
__device__ __forceinline__ void element32_out(const DevMesh& m, const Phys& c, const Bufs& b, int t, float (&out)[18]) {
    const int Tp = m.Tp;
    int v[3];
    float bx[3], by[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        v[k] = m.tri[k * Tp + t];
        bx[k] = m.grad32[(2 * k) * Tp + t];
        by[k] = m.grad32[(2 * k + 1) * Tp + t];
    }
    const float A = m.area32[t];
    const double C0d = b.C[v[0]], C1d = b.C[v[1]], C2d = b.C[v[2]];
    const float dC1 = (float)(C1d - C0d), dC2 = (float)(C2d - C0d);
    const float C0 = (float)C0d;
    const float Cb = C0 + (dC1 + dC2) * (1.0f / 3.0f);
    float p[3], ux[3], uy[3], om1[3];
    float mus = 0.0f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        p[k] = b.p32[v[k]];
        ux[k] = b.ux32[v[k]];
        uy[k] = b.uy32[v[k]];
        mus += b.mu32[v[k]];
    }
    om1[0] = 1.0f - omega32(C0, c);
    om1[1] = 1.0f - omega32(C0 + dC1, c);
    om1[2] = 1.0f - omega32(C0 + dC2, c);
    const float third = 1.0f / 3.0f;
    const float ubx = (ux[0] + ux[1] + ux[2]) * third, uby = (uy[0] + uy[1] + uy[2]) * third;
    const float mub = mus * third;
    const float gCx = dC1 * bx[1] + dC2 * bx[2], gCy = dC1 * by[1] + dC2 * by[2];
    const float dp1 = p[1] - p[0], dp2 = p[2] - p[0];
    const float gpx = dp1 * bx[1] + dp2 * bx[2], gpy = dp1 * by[1] + dp2 * by[2];
    float lapmu = 0.0f;
    if (c.lapmu_nodal) {
        lapmu = (b.lmu32[v[0]] + b.lmu32[v[1]] + b.lmu32[v[2]]) * (1.0f / 3.0f);
    } else {
        const float gmx = b.gmu32[t], gmy = b.gmu32[Tp + t];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            int nb = m.nbr[k * Tp + t];
            if (nb >= 0) lapmu -= (gmx + b.gmu32[nb]) * bx[k] + (gmy + b.gmu32[Tp + nb]) * by[k];
        }
    }
    const float drho = c.drho_f;
    const float rhob = c.rho_v_f + Cb * drho;
    const float f = 3.0f * Cb / rhob;
    const float vhx = gCx - f * (gpx - mub * gCx), vhy = gCy - f * (gpy - mub * gCy);
    // Forces as in k_element: with T = Gamma / w - 1, A Phi_g = w s (P + Q T) and
    // A Phi_h = w A ((e - u).v + M lap mu)(1 + T), the axis weight folded into the vectors.
    const float uub15 = 1.5f * (ubx * ubx + uby * uby);
    const float w1 = 1.0f / 9.0f, Aw = A * w1, P = A * mub, Q = fmaf(A * third, drho, P);
    const float sx = w1 * gCx, sy = w1 * gCy, su = ubx * sx + uby * sy;
    const float vx = Aw * vhx, vy = Aw * vhy, vu = ubx * vx + uby * vy - Aw * (c.mobility_f * lapmu);
    // Differences of the equilibria to vertex 0, k = 1, 2:
    //   h: w ((1 + T_0) dC_k + C_k dT_k),  g: w (dp_k + (drho_k T_0 + rho_k dT_k) / 3),
    //   dT_k = 3 e.du_k + 4.5 (e.du_k)(e.su_k) - 1.5 du_k.su_k, su_k = u_k + u_0
    const float uu0 = 1.5f * (ux[0] * ux[0] + uy[0] * uy[0]);
    const float dC[2] = {dC1, dC2}, dp[2] = {dp1, dp2};
    float dux[2], duy[2], sux[2], suy[2], D[2], Ck[2], rk[2], dr[2], abx[2], aby[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        dux[k] = ux[k + 1] - ux[0];
        duy[k] = uy[k + 1] - uy[0];
        sux[k] = ux[k + 1] + ux[0];
        suy[k] = uy[k + 1] + uy[0];
        D[k] = -1.5f * (dux[k] * sux[k] + duy[k] * suy[k]);
        Ck[k] = C0 + dC[k];
        dr[k] = drho * third * dC[k];
        rk[k] = third * (c.rho_v_f + C0 * drho) + dr[k];
        abx[k] = A * bx[k + 1];
        aby[k] = A * by[k + 1];
    }
    // the post-collision deviations of the three vertices, all loaded first
    // (the rest populations do not enter)
    float pg[3][9], ph[3][9];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            float g4[4], h4[4];
            load_vec(g4, b.dpsi, m.Np, j, v[k]);
            load_vec(h4, b.dpsi, m.Np, 2 + j, v[k]);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                pg[k][1 + 4 * j + e] = g4[e];
                ph[k][1 + 4 * j + e] = h4[e];
            }
        }
    out[0] = -4.0f * su * fmaf(Q, -uub15, P);
    out[9] = -4.0f * fmaf(vu, -uub15, vu);
    // a direction and its opposite together: e.u changes sign, the squares do not
#define FELBM_ELEM32_PAIR(q, fw)                                                                   \
    {                                                                                              \
        const float w = (float)wq(q);                                                              \
        const float eu = edot<q, float>(ubx, uby), t2 = fmaf(4.5f * eu, eu, -uub15);               \
        const float tp = fmaf(3.0f, eu, t2), tm = fmaf(-3.0f, eu, t2);                             \
        const float es = edot<q, float>((fw) * sx, (fw) * sy), ev = edot<q, float>((fw) * vx, (fw) * vy); \
        const float vp = ev - (fw) * vu, vm = -ev - (fw) * vu;                                     \
        float gp = (es - (fw) * su) * fmaf(Q, tp, P), gm = (-es - (fw) * su) * fmaf(Q, tm, P);     \
        float hp = fmaf(vp, tp, vp), hm = fmaf(vm, tm, vm);                                        \
        const float e0 = edot<q, float>(ux[0], uy[0]), z2 = fmaf(4.5f * e0, e0, -uu0);             \
        const float zp = fmaf(3.0f, e0, z2), zm = fmaf(-3.0f, e0, z2);                             \
        const float g0p = om1[0] * pg[0][q], g0m = om1[0] * pg[0][opp(q)];                         \
        const float h0p = om1[0] * ph[0][q], h0m = om1[0] * ph[0][opp(q)];                         \
        _Pragma("unroll") for (int k = 0; k < 2; ++k) {                                            \
            const float ed = edot<q, float>(dux[k], duy[k]), es2 = edot<q, float>(sux[k], suy[k]); \
            const float d2 = fmaf(4.5f * ed, es2, D[k]);                                           \
            const float dTp = fmaf(3.0f, ed, d2), dTm = fmaf(-3.0f, ed, d2);                       \
            const float eb = edot<q, float>(abx[k], aby[k]);                                       \
            const float gqp = fmaf(dTp, rk[k], fmaf(zp, dr[k], dp[k])), gqm = fmaf(dTm, rk[k], fmaf(zm, dr[k], dp[k])); \
            const float hqp = fmaf(dTp, Ck[k], fmaf(zp, dC[k], dC[k])), hqm = fmaf(dTm, Ck[k], fmaf(zm, dC[k], dC[k])); \
            gp = fmaf(-eb, fmaf(w, gqp, fmaf(om1[k + 1], pg[k + 1][q], -g0p)), gp);                \
            gm = fmaf(eb, fmaf(w, gqm, fmaf(om1[k + 1], pg[k + 1][opp(q)], -g0m)), gm);            \
            hp = fmaf(-eb, fmaf(w, hqp, fmaf(om1[k + 1], ph[k + 1][q], -h0p)), hp);                \
            hm = fmaf(eb, fmaf(w, hqm, fmaf(om1[k + 1], ph[k + 1][opp(q)], -h0m)), hm);            \
        }                                                                                          \
        out[q] = gp;                                                                               \
        out[opp(q)] = gm;                                                                          \
        out[9 + (q)] = hp;                                                                         \
        out[9 + opp(q)] = hm;                                                                      \
    }
    FELBM_ELEM32_PAIR(1, 1.0f) FELBM_ELEM32_PAIR(2, 1.0f) FELBM_ELEM32_PAIR(5, 0.25f) FELBM_ELEM32_PAIR(6, 0.25f)
#undef FELBM_ELEM32_PAIR
}

__device__ __forceinline__ void element32_tri(const DevMesh& m, const Phys& c, const Bufs& b, int t) {
    float out[18];
    element32_out(m, c, b, t, out);
    float2* dst = reinterpret_cast<float2*>(b.R32 + (size_t)t * 18);
#pragma unroll
    for (int k = 0; k < 9; ++k) dst[k] = make_float2(out[2 * k], out[2 * k + 1]);
}

// The vertices' 48 deviation values are all loaded (as twelve 16-byte loads)
// before the per-direction arithmetic, so that they are in flight together; 80
// registers (6 blocks of 128 per SM).  Runs where k_force32 does not.
__global__ void __launch_bounds__(128, 6) k_element32(DevMesh m, Phys c, Bufs b) {
    pdl_release();
    pdl_wait();
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < m.T) element32_tri(m, c, b, t);
}

// ------------------------------------------ streaming RHS gather (FP32) ----
// As k_rhs; the wall term needs psi_hat_opp - psi_hat at a node, which in the
// split form is  g: -2 w rho (e.u) + (1-omega)(dg_opp - dg),
//                h: -6 w C (e.u)   + (1-omega)(dh_opp - dh).
// What the weak bounce-back of a wall edge reads at one of its ends.
struct WallEnd {
    float C, ux, uy, om, rho;
    float4 d[4];      // deviations (planes of vec_at)
};
template <int kP0, int kP1>
__device__ __forceinline__ WallEnd wall_end(const Phys& c, const Bufs& b, int Np, int v) {
    WallEnd e;
    e.C = (float)b.C[v];
    e.ux = b.ux32[v];
    e.uy = b.uy32[v];
#pragma unroll
    for (int p = kP0; p < kP1; ++p) e.d[p] = reinterpret_cast<const float4*>(b.dpsi)[(size_t)p * Np + v];
    e.om = 1.0f - omega32(e.C, c);
    e.rho = c.rho_v_f + e.C * c.drho_f;
    return e;
}
// psi_hat_opp - psi_hat of component k of plane p at one end; a direction's
// opposite is two components further in the same plane.
template <int kP, int k>
__device__ __forceinline__ float wall_diff(const WallEnd& e) {
    constexpr int q = 1 + 4 * (kP & 1) + k;
    static_assert(opp(q) == 1 + 4 * (kP & 1) + (k ^ 2), "opposites share a plane");
    const float w = (float)wq(q), eu = edot<q, float>(e.ux, e.uy);
    const float4 d = e.d[kP];
    const float dev = k == 0 ? d.z - d.x : k == 1 ? d.w - d.y : k == 2 ? d.x - d.z : d.y - d.w;
    return (kP < 2 ? -2.0f * w * e.rho * eu : -6.0f * w * e.C * eu) + e.om * dev;
}
// The term of component k of plane p: zero for the outgoing directions.
template <int kP, int k>
__device__ __forceinline__ float wall32(const Phys& c, const WallEnd& i, const WallEnd& o, float L, float nx, float ny) {
    const float en = edot<1 + 4 * (kP & 1) + k, float>(nx, ny);
    if (!(en < 0.0f)) return 0.0f;
    return -c.dt_f * en * (L * (1.0f / 3.0f) * wall_diff<kP, k>(i) + L * (1.0f / 6.0f) * wall_diff<kP, k>(o));
}

// kI > 0: the incident triangles from the incidence ELL (padding: the zero
// residual row T), their ids and gradients loaded up front; kI = 0: CSR.
template <int kI = 0, bool kFirst = true>
__device__ __forceinline__ void rhs32_node(const DevMesh& m, const Phys& c, const Bufs& b, int i, float tau0) {
    const int Np = m.Np;
    float acc[18];
#pragma unroll
    for (int q = 0; q < 18; ++q) acc[q] = 0.0f;
    const float c1 = c.dt3_f, c2 = c.dt2h_f;
    constexpr int kIr = kI > 0 ? kI : 1;
    int tt[kIr];
    float bxx[kIr], byy[kIr];
    if constexpr (kI > 0) {
#pragma unroll
        for (int k = 0; k < kI; ++k) {
            tt[k] = m.iell_tri[k * Np + i];
            bxx[k] = m.iell_bx32[k * Np + i];
            byy[k] = m.iell_by32[k * Np + i];
        }
    }
    const int k0 = kI > 0 ? 0 : m.inc_ptr[i], k1 = kI > 0 ? kI : m.inc_ptr[i + 1];
#pragma unroll(kI > 0 ? kIr : 1)
    for (int k = k0; k < k1; ++k) {
        int t;
        float bxi, byi;
        if constexpr (kI > 0) {
            t = tt[k];
            bxi = bxx[k];
            byi = byy[k];
        } else {
            t = m.inc_tri[k];
            bxi = m.inc_bx32[k];
            byi = m.inc_by32[k];
        }
        const float2* src = reinterpret_cast<const float2*>(b.R32 + (size_t)t * 18);
        float r[18];
#pragma unroll
        for (int s = 0; s < 9; ++s) {
            float2 v2 = src[s];
            r[2 * s] = v2.x;
            r[2 * s + 1] = v2.y;
        }
#define FELBM_RHS32_Q(q)                                        \
        {                                                       \
            float w = c1 + c2 * edot<q, float>(bxi, byi);              \
            acc[q] = fmaf(r[q], w, acc[q]);                     \
            acc[9 + q] = fmaf(r[9 + q], w, acc[9 + q]);         \
        }
        FELBM_RHS32_Q(0) FELBM_RHS32_Q(1) FELBM_RHS32_Q(2) FELBM_RHS32_Q(3) FELBM_RHS32_Q(4)
        FELBM_RHS32_Q(5) FELBM_RHS32_Q(6) FELBM_RHS32_Q(7) FELBM_RHS32_Q(8)
#undef FELBM_RHS32_Q
    }
    for (int k = m.winc_ptr[i]; k < m.winc_ptr[i + 1]; ++k) {
        const int e = m.winc_edge[k];
        const int o = m.wall_a[e] == i ? m.wall_b[e] : m.wall_a[e];
        const float L = (float)m.wall_len[e], nx = (float)m.wall_nx[e], ny = (float)m.wall_ny[e];
        const WallEnd ei = wall_end<0, 4>(c, b, Np, i), eo = wall_end<0, 4>(c, b, Np, o);
#define FELBM_WALL32_P(p)                                                \
        acc[vec_row(p, 0)] += wall32<p, 0>(c, ei, eo, L, nx, ny);        \
        acc[vec_row(p, 1)] += wall32<p, 1>(c, ei, eo, L, nx, ny);        \
        acc[vec_row(p, 2)] += wall32<p, 2>(c, ei, eo, L, nx, ny);        \
        acc[vec_row(p, 3)] += wall32<p, 3>(c, ei, eo, L, nx, ny);
        FELBM_WALL32_P(0) FELBM_WALL32_P(1) FELBM_WALL32_P(2) FELBM_WALL32_P(3)
#undef FELBM_WALL32_P
    }
    float s = m.inv_lumped32[i] * tau0;
    store_all(b.r32, Np, i, acc);
    if (kFirst) {
#pragma unroll
        for (int q = 0; q < 18; ++q) acc[q] *= s;
        store_all(b.e1, Np, i, acc);
    }
}

// at most 64 registers (8 blocks of 128 per SM; 6 % faster than 96 registers)
template <int kI, bool kFirst = true>
__global__ void __launch_bounds__(128, 8) k_rhs32(DevMesh m, Phys c, Bufs b, float tau0) {
    pdl_release();
    pdl_wait();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < m.N) rhs32_node<kI, kFirst>(m, c, b, i, tau0);
}

// -------------------- element residuals and their gather in one kernel ----
// One node block (HostMesh::blk_ptr) per thread block: the residuals of the
// triangles at its nodes go to shared memory, then two threads a node (one per
// class of directions) gather them.  The same arithmetic as k_element32 and
// k_rhs32 in the same order; the residuals, 72 bytes a triangle written and
// gathered back through DRAM by those two, never leave the multiprocessor, for
// about 10 % of the triangles formed twice.  Bound by load latency and L1 (48 %
// of its wavefronts, 34 % of the issue slots, 24 warps at 80 registers, which
// spill 88 to 100 bytes a thread): 337 us
// on 2,082,816 nodes against 237 + 144 us for the two kernels, 31 against 22 +
// 19 us on 131,072 nodes.  Two threads a triangle at 80 or 64 registers: 352
// and 381 us; 256 threads a block: 416 us.  Residual rows hold the planes of
// vec_at one after another, 20 floats apart (16-byte words of consecutive
// triangles in different banks); the row after the last is zero (padding).
constexpr int kForceThreads = 384;
constexpr int kForceRow = 20;
constexpr int kForceTris = 1400;       // two thread blocks' rows fit a multiprocessor's shared memory

__host__ __device__ constexpr size_t force_smem_bytes(int max_tri) { return (size_t)(max_tri + 1) * kForceRow * 4; }

// The gather of the planes kC and kC + 2 (one class of directions of g and of
// h, which share the weights), with the rest populations in class 0.
template <int kC, int kI>
__device__ __forceinline__ void force32_gather(const DevMesh& m, const Phys& c, const Bufs& b, const float* R, int i,
                                               float tau0, int first) {
    const int Np = m.Np;
    const float c1 = c.dt3_f, c2 = c.dt2h_f;
    int tt[kI];
    float bxx[kI], byy[kI];
#pragma unroll
    for (int k = 0; k < kI; ++k) {
        tt[k] = m.iell_loc[k * Np + i];
        bxx[k] = m.iell_bx32[k * Np + i];
        byy[k] = m.iell_by32[k * Np + i];
    }
    const int w0 = m.winc_ptr[i], w1 = m.winc_ptr[i + 1];
    float ag[4] = {0.0f, 0.0f, 0.0f, 0.0f}, ah[4] = {0.0f, 0.0f, 0.0f, 0.0f}, ar[2] = {0.0f, 0.0f};
    constexpr int q0 = 1 + 4 * kC;
#pragma unroll
    for (int k = 0; k < kI; ++k) {
        const float* row = R + tt[k] * kForceRow;
        float rg[4], rh[4];
        load_shared(rg, row + 4 * kC);
        load_shared(rh, row + 8 + 4 * kC);
        const float w[4] = {c1 + c2 * edot<q0, float>(bxx[k], byy[k]), c1 + c2 * edot<q0 + 1, float>(bxx[k], byy[k]),
                            c1 + c2 * edot<q0 + 2, float>(bxx[k], byy[k]), c1 + c2 * edot<q0 + 3, float>(bxx[k], byy[k])};
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            ag[v] = fmaf(rg[v], w[v], ag[v]);
            ah[v] = fmaf(rh[v], w[v], ah[v]);
        }
        if constexpr (kC == 0) {
            float r0[2];
            load_shared(r0, row + 16);
            ar[0] = fmaf(r0[0], c1, ar[0]);
            ar[1] = fmaf(r0[1], c1, ar[1]);
        }
    }
    for (int k = w0; k < w1; ++k) {
        const int e = m.winc_edge[k];
        const int o = m.wall_a[e] == i ? m.wall_b[e] : m.wall_a[e];
        const float L = (float)m.wall_len[e], nx = (float)m.wall_nx[e], ny = (float)m.wall_ny[e];
        const WallEnd ei = wall_end<0, 4>(c, b, Np, i), eo = wall_end<0, 4>(c, b, Np, o);
#define FELBM_FORCE_WALL(v)                                              \
        ag[v] += wall32<kC, v>(c, ei, eo, L, nx, ny);                    \
        ah[v] += wall32<kC + 2, v>(c, ei, eo, L, nx, ny);
        FELBM_FORCE_WALL(0) FELBM_FORCE_WALL(1) FELBM_FORCE_WALL(2) FELBM_FORCE_WALL(3)
#undef FELBM_FORCE_WALL
    }
    store_vec(b.r32, Np, kC, i, ag);
    store_vec(b.r32, Np, kC + 2, i, ah);
    if (kC == 0) store_vec(b.r32, Np, 4, i, ar);
    if (first) {
        const float s = m.inv_lumped32[i] * tau0;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            ag[v] *= s;
            ah[v] *= s;
            if (v < 2) ar[v] *= s;
        }
        store_vec(b.e1, Np, kC, i, ag);
        store_vec(b.e1, Np, kC + 2, i, ah);
        if (kC == 0) store_vec(b.e1, Np, 4, i, ar);
    }
}

template <int kI>
__global__ void __launch_bounds__(kForceThreads, 2) k_force32(DevMesh m, Phys c, Bufs b, float tau0, int first) {
    extern __shared__ __align__(16) float force_rows[];
    float* R = force_rows;
    pdl_release();
    const int blk = (int)blockIdx.x, tid = (int)threadIdx.x;
    const int t0 = m.blk_tri_ptr[blk], nt = m.blk_tri_ptr[blk + 1] - t0;
    const int s0 = m.blk_ptr[blk], ni = m.blk_ptr[blk + 1] - s0;
    if (tid < kForceRow) R[nt * kForceRow + tid] = 0.0f;
    pdl_wait();
    for (int r = tid; r < nt; r += kForceThreads) {
        float out[18];
        element32_out(m, c, b, m.blk_tri[t0 + r], out);
        float* row = R + r * kForceRow;
#pragma unroll
        for (int p = 0; p < 4; ++p)
            *reinterpret_cast<float4*>(row + 4 * p) =
                make_float4(out[vec_row(p, 0)], out[vec_row(p, 1)], out[vec_row(p, 2)], out[vec_row(p, 3)]);
        *reinterpret_cast<float2*>(row + 16) = make_float2(out[0], out[9]);
    }
    __syncthreads();
    for (int w = tid; w < 2 * ni; w += kForceThreads) {
        if (w < ni)
            force32_gather<0, kI>(m, c, b, R, s0 + w, tau0, first);
        else
            force32_gather<1, kI>(m, c, b, R, s0 + w - ni, tau0, first);
    }
}

// ---------------------------- update of fields and deviations (node) ------
// With the increment d = psi^{n+1} - psi_hat of all 18 populations at node i:
//   C' = C + sum d_h (FP64), p' = p + sum d_g, rho' u' = rho u + 3 sum e d_g,
//   dpsi' = (1 - omega) dpsi + d + psi^eq(C, p, u) - psi^eq(C', p', u'),
// the equilibrium difference written through dC, dp, du (no cancellation):
//   h: -(Gamma' dC + C (Gamma' - Gamma)),
//   g: -(w dp + cs2 (drho (Gamma' - w) + rho (Gamma' - Gamma))).
__device__ __forceinline__ void dev32_update(const DevMesh& m, const Phys& c, const Bufs& b, int i,
                                             const float (&d)[18]) {
    const int Np = m.Np;
    const double Cd = b.C[i];
    const float C = (float)Cd;
    const float p = b.p32[i], ux = b.ux32[i], uy = b.uy32[i];
    const float om1 = 1.0f - omega32(C, c);
    float dC = 0.0f, dp = 0.0f;
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        dC += d[9 + q];
        dp += d[q];
    }
    const float jx = (d[1] - d[3]) + (d[5] - d[6]) + (d[8] - d[7]);
    const float jy = (d[2] - d[4]) + (d[5] + d[6]) - (d[7] + d[8]);
    const double Cnd = Cd + (double)dC;
    const float drho_c = c.drho_f;
    const float rho = c.rho_v_f + C * drho_c;
    const float rhon = rho + drho_c * dC;
    const float uxn = (rho * ux + 3.0f * jx) / rhon, uyn = (rho * uy + 3.0f * jy) / rhon;
    const float drho = drho_c * dC;
    const float dux = uxn - ux, duy = uyn - uy, sux = uxn + ux, suy = uyn + uy;
    const float uun15 = 1.5f * (uxn * uxn + uyn * uyn);
    const float third = 1.0f / 3.0f;
    float dev[18];
    load_all(dev, b.dpsi, Np, i);
#define FELBM_UPD32_Q(q)                                                                         \
    {                                                                                            \
        const float w = (float)wq(q);                                                            \
        const float Gn = gamma32<q>(uxn, uyn, uun15);                                            \
        const float dG = dgamma32<q>(dux, duy, sux, suy);                                        \
        dev[q] = om1 * dev[q] + d[q] - (w * dp + third * (drho * (Gn - w) + rho * dG));            \
        dev[9 + q] = om1 * dev[9 + q] + d[9 + q] - (Gn * dC + C * dG);                                     \
    }
    FELBM_UPD32_Q(0) FELBM_UPD32_Q(1) FELBM_UPD32_Q(2) FELBM_UPD32_Q(3) FELBM_UPD32_Q(4)
    FELBM_UPD32_Q(5) FELBM_UPD32_Q(6) FELBM_UPD32_Q(7) FELBM_UPD32_Q(8)
#undef FELBM_UPD32_Q
    store_all(b.dpsi, Np, i, dev);
    b.C[i] = Cnd;
    b.p32[i] = p + dp;
    b.ux32[i] = uxn;
    b.uy32[i] = uyn;
}

// ------------------------------------ conversions to / from full FP64 ------
// stage [18][N] (caller order) <- psi = psi^eq(C, p, u) + dpsi, in FP64
// (one thread per caller-order node o: the 18 stage streams are written
// coalesced, the node's fields and deviation row read at i = iperm[o])
__global__ void k_dev32_to_full(DevMesh m, Phys c, Bufs b, double* stage) {
    const int o = blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= m.N) return;
    const int N = m.N, Np = m.Np, i = m.iperm[o];
    double C = b.C[i], p = b.p32[i], ux = b.ux32[i], uy = b.uy32[i];
    double rho = c.rho_v + C * (c.rho_l - c.rho_v);
    double uu15 = 1.5 * (ux * ux + uy * uy);
    float dev[18];
    load_all(dev, b.dpsi, Np, i);
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        double eu = ex(q) * ux + ey(q) * uy;
        double G = wq(q) * (1.0 + 3.0 * eu + 4.5 * eu * eu - uu15);
        stage[(size_t)q * N + o] = wq(q) * p + rho * (1.0 / 3.0) * (G - wq(q)) + (double)dev[q];
        stage[(size_t)(9 + q) * N + o] = G * C + (double)dev[9 + q];
    }
}

// fields and deviations <- psi (stage [18][N], caller order, FP64)
// (one thread per caller-order node o: the 18 stage streams are read
// coalesced, the node's fields and deviation row written at i = iperm[o])
__global__ void k_full_to_dev32(DevMesh m, Phys c, Bufs b, const double* __restrict__ stage) {
    const int o = blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= m.N) return;
    const int N = m.N, Np = m.Np, i = m.iperm[o];
    double g[9], h[9], C = 0.0, p = 0.0;
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        g[q] = stage[(size_t)q * N + o];
        h[q] = stage[(size_t)(9 + q) * N + o];
        C += h[q];
        p += g[q];
    }
    const double jx = (g[1] - g[3]) + (g[5] - g[6]) + (g[8] - g[7]);
    const double jy = (g[2] - g[4]) + (g[5] + g[6]) - (g[7] + g[8]);
    const double rho = c.rho_v + C * (c.rho_l - c.rho_v);
    // the stored fields (FP32 p, u; FP64 C); deviations are taken relative to
    // the equilibrium of exactly these values
    const float rhof = (float)rho, Cf = (float)C, pf = (float)p;
    const float uxf = 3.0f * (float)jx / rhof, uyf = 3.0f * (float)jy / rhof;
    const double ps = pf;
    const float uu15 = 1.5f * (uxf * uxf + uyf * uyf);
    const float r3 = rhof * (1.0f / 3.0f);
    // g_q - g_q^eq = (g_q - w p) - (rho/3) w T_q and h_q - h_q^eq = (h_q - w C) - w T_q C,
    // T_q = Gamma_q / w_q - 1 = 3 e.u + 4.5 (e.u)^2 - 1.5 u.u: the large differences in
    // FP64, rounded once to FP32; the velocity terms (O(|u|) of the state) in FP32
    float dev[18];
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        const float wf = (float)wq(q);
        const float eu = (float)ex(q) * uxf + (float)ey(q) * uyf;
        const float T = 3.0f * eu + 4.5f * eu * eu - uu15;
        const float dg0 = (float)(g[q] - wq(q) * ps), dh0 = (float)(h[q] - wq(q) * C);
        dev[q] = dg0 - r3 * (wf * T);
        dev[9 + q] = dh0 - (wf * T) * Cf;
    }
    store_all(b.dpsi, Np, i, dev);
    b.C[i] = C;
    b.p32[i] = pf;
    b.ux32[i] = uxf;
    b.uy32[i] = uyf;
}

// Initial state at equilibrium with C0, p0, u0 (the layout of k_init_state):
// the fields are stored and the deviations are zero.
__global__ void k_init_dev32(DevMesh m, Bufs b, const double* __restrict__ stage, int has_p, int has_u) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m.N) return;
    const int o = m.perm[i], N = m.N;
    const double* u = stage + (has_p ? 2 : 1) * (size_t)N;
    b.C[i] = stage[o];
    b.p32[i] = has_p ? (float)stage[N + o] : 0.0f;
    b.ux32[i] = has_u ? (float)u[o] : 0.0f;
    b.uy32[i] = has_u ? (float)u[N + o] : 0.0f;
#pragma unroll
    for (int q = 0; q < 18; ++q) b.dpsi[vec_at(m.Np, q, i)] = 0.0f;
}

__global__ void k_gather_out_f(DevMesh m, const float* __restrict__ src, double* stage) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m.N) return;
    stage[m.perm[i]] = (double)src[i];
}
