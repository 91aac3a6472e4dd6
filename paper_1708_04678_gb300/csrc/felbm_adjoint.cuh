// Adjoint (reverse mode) of one FP64 time step (included by felbm.cu).
//
// Given lambda = dL/dpsi^{n+1} and the state psi^n, the passes below form
// dL/dpsi^n and add dL/dphi_c (per wall edge).  The step (Sec. II.C of
// arXiv:1708.04678) is   psi^{n+1} = psi_hat + M11^{-1} RHS(psi_hat, Phi),
// psi_hat = collide(psi), Phi = forces(moments, mu, lap mu), so in reverse:
//   lambda_RHS = M11^{-1} lambda                       (M11 symmetric: same solve)
//   A:  per triangle  lambda_R = sum_k w(v_k) lambda_RHS(v_k), pulled back
//       through the forces to the nine element scalars (u, C, mu means,
//       grad C, grad p, lap mu)
//   B:  per triangle  lambda of grad mu (own and the neighbours' lap mu terms)
//   D:  per node      gathers over incident triangles: lambda of psi_hat,
//       mu, C, p, u; transpose of the weak bounce-back wall term
//   E:  per node      transpose of mu (double well, patch Laplacian, wetting
//       flux; per-edge dL/dphi_c), of the collision and of the moments ->
//       lambda^n.
// Every pass gathers; none scatters, so there are no atomics and the result
// does not depend on scheduling.
//
// All passes are FP64.  A and E pull lambda back through the forces and the
// collision in reverse, one sweep over the directions each; differentiating
// forward once per scalar (nine and four sweeps of dual numbers) took 108 and
// 42 us on the 128x64 droplet (16,384 triangles) against 20 and 18 us.
#pragma once

// ------------------------------------------------------ adjoint buffers
struct AdjBufs {
    double* lam;     // [18][Np] lambda (in: dL/dpsi^{n+1}; out: dL/dpsi^n)
    double* lamhat;  // [18][Np] dL/dpsi_hat
    double* lamR;    // [T][18]  dL/dR
    double* lamE;    // [T][9]   dL/d(C_bar, mu_bar, ux_bar, uy_bar, gCx, gCy, gpx, gpy, lap mu)
    double* lamG;    // [2][Tp]  dL/d(grad mu)
    double* lamMu;   // [Np]
    double* lamC;    // [Np]
    double* lamP;
    double* lamUx;
    double* lamUy;
    double* dphi;    // [E] dL/dphi_c accumulated per wall edge since the seed
    const double* lamRHS;  // [18][Np] M11^{-1} lambda (the solve's output)
    const double* kval;    // [nnz] P1 stiffness entries (symmetric)
};

// (x, y) += v e_q, additions only
template <int q>
__device__ __forceinline__ void add_along(double& x, double& y, double v) {
    if (ex(q) == 1) x += v;
    if (ex(q) == -1) x -= v;
    if (ey(q) == 1) y += v;
    if (ey(q) == -1) y -= v;
}

// A: element residual adjoint and the adjoint of the forces.  With
// T = Gamma / w - 1 = 3 e.u + 4.5 (e.u)^2 - 1.5 u.u and s = (e - u).grad C,
//   Phi_g = w s (mu + (mu + drho/3) T),  Phi_h = w (1 + T) ((e - u).v + M lap mu),
//   v = (1 + f mu) grad C - f grad p,    f = 3 C / rho.
__global__ void __launch_bounds__(128) k_adj_elem_a(DevMesh m, Phys c, Bufs b, AdjBufs a) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= m.T) return;
    const int Tp = m.Tp, Np = m.Np;
    int v[3];
    double bx[3], by[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        v[k] = m.tri[k * Tp + t];
        bx[k] = m.grad[(2 * k) * Tp + t];
        by[k] = m.grad[(2 * k + 1) * Tp + t];
    }
    const double A = m.area[t];
    const double c1 = c.dt * (1.0 / 3.0), c2 = 0.5 * c.dt * c.dt;
    // lambda_R = sum over the vertices of the RHS weights times lambda_RHS
    double lr[18];
#define FELBM_ADJA_Q(q)                                                               \
    {                                                                                 \
        double sg = 0.0, sh = 0.0;                                                    \
        for (int k = 0; k < 3; ++k) {                                                 \
            double w = c1 + c2 * edot<q, double>(bx[k], by[k]);                       \
            sg += w * a.lamRHS[q * Np + v[k]];                                        \
            sh += w * a.lamRHS[(9 + q) * Np + v[k]];                                  \
        }                                                                             \
        lr[q] = sg;                                                                   \
        lr[9 + q] = sh;                                                               \
    }
    FELBM_ADJA_Q(0) FELBM_ADJA_Q(1) FELBM_ADJA_Q(2) FELBM_ADJA_Q(3) FELBM_ADJA_Q(4)
    FELBM_ADJA_Q(5) FELBM_ADJA_Q(6) FELBM_ADJA_Q(7) FELBM_ADJA_Q(8)
#undef FELBM_ADJA_Q
#pragma unroll
    for (int q = 0; q < 18; ++q) a.lamR[(size_t)t * 18 + q] = lr[q];
    // the nine element scalars, as in k_element
    double Cs = 0, uxs = 0, uys = 0, mus = 0, gCx = 0, gCy = 0, gpx = 0, gpy = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        double Cv = b.C[v[k]], pv = b.p[v[k]];
        Cs += Cv;
        uxs += b.ux[v[k]];
        uys += b.uy[v[k]];
        mus += b.mu[v[k]];
        gCx += Cv * bx[k];
        gCy += Cv * by[k];
        gpx += pv * bx[k];
        gpy += pv * by[k];
    }
    const double third = 1.0 / 3.0;
    double sv[9] = {uxs * third, uys * third, Cs * third, mus * third, gCx, gCy, gpx, gpy, 0.0};
    {
        double gmx = b.gmu[t], gmy = b.gmu[Tp + t], lapmu = 0.0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            int nb = m.nbr[k * Tp + t];
            if (nb >= 0) lapmu -= (gmx + b.gmu[nb]) * bx[k] + (gmy + b.gmu[Tp + nb]) * by[k];
        }
        sv[8] = lapmu;
    }
    // lambda_s = sum_q A lr_q dPhi_q / ds: moments of the adjoints of s (S), of
    // (e - u).v (V) and of T over the directions
    const double ux = sv[0], uy = sv[1], mu = sv[3], drho = c.rho_l - c.rho_v, rho = c.rho_v + sv[2] * drho;
    const double f = 3.0 * sv[2] / rho, hx = gpx - mu * gCx, hy = gpy - mu * gCy;
    const double vx = gCx - f * hx, vy = gCy - f * hy;
    const double u_gC = ux * gCx + uy * gCy, u_v = ux * vx + uy * vy - c.mobility * sv[8];
    const double uu15 = 1.5 * (ux * ux + uy * uy), mud = mu + drho * third;
    double S0 = 0.0, Sx = 0.0, Sy = 0.0, V0 = 0.0, Vx = 0.0, Vy = 0.0, T0 = 0.0, Tx = 0.0, Ty = 0.0, M0 = 0.0;
#define FELBM_ADJF_Q(q)                                                               \
    {                                                                                 \
        const double eu = edot<q>(ux, uy), T = fma(3.0 + 4.5 * eu, eu, -uu15);        \
        const double lg = wq(q) * lr[q], lh = wq(q) * lr[9 + q];                      \
        const double sq = edot<q>(gCx, gCy) - u_gC, vq = edot<q>(vx, vy) - u_v;       \
        const double S = lg * fma(mud, T, mu), V = fma(lh, T, lh), gs = lg * sq;      \
        const double t = fma(gs, mud, lh * vq), te = t * (3.0 + 9.0 * eu);            \
        S0 += S;                                                                      \
        V0 += V;                                                                      \
        T0 += t;                                                                      \
        add_along<q>(Sx, Sy, S);                                                      \
        add_along<q>(Vx, Vy, V);                                                      \
        add_along<q>(Tx, Ty, te);                                                     \
        M0 += fma(gs, T, gs);                                                         \
    }
    FELBM_ADJF_Q(0) FELBM_ADJF_Q(1) FELBM_ADJF_Q(2) FELBM_ADJF_Q(3) FELBM_ADJF_Q(4)
    FELBM_ADJF_Q(5) FELBM_ADJF_Q(6) FELBM_ADJF_Q(7) FELBM_ADJF_Q(8)
#undef FELBM_ADJF_Q
    const double lvx = Vx - ux * V0, lvy = Vy - uy * V0, fm = 1.0 + f * mu;
    // stored as (C_bar, mu_bar, ux_bar, uy_bar, gCx, gCy, gpx, gpy, lap mu)
    double* dst = a.lamE + (size_t)t * 9;
    dst[0] = -A * (hx * lvx + hy * lvy) * (3.0 * c.rho_v / (rho * rho));      // df/dC = 3 rho_v / rho^2
    dst[1] = A * (M0 + f * (gCx * lvx + gCy * lvy));
    dst[2] = A * (Tx - 3.0 * ux * T0 - gCx * S0 - vx * V0);
    dst[3] = A * (Ty - 3.0 * uy * T0 - gCy * S0 - vy * V0);
    dst[4] = A * (Sx - ux * S0 + fm * lvx);
    dst[5] = A * (Sy - uy * S0 + fm * lvy);
    dst[6] = -A * f * lvx;
    dst[7] = -A * f * lvy;
    dst[8] = A * c.mobility * V0;
}

// B: lambda of grad mu_T.  lap mu_T = -sum_k[nb_k] (G_T + G_nb).b_k, so G_T
// receives -lambda_lap(T) b_k(T) from its own edges and -lambda_lap(nb) b_s(nb)
// from each neighbour (s = the shared edge's slot in the neighbour).
__global__ void __launch_bounds__(kBlock) k_adj_elem_b(DevMesh m, AdjBufs a) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= m.T) return;
    const int Tp = m.Tp;
    const double lt = a.lamE[(size_t)t * 9 + 8];
    double gx = 0.0, gy = 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        int nb = m.nbr[k * Tp + t];
        if (nb < 0) continue;
        int sl = m.nbr_slot[k * Tp + t];
        double ln = a.lamE[(size_t)nb * 9 + 8];
        gx -= lt * m.grad[(2 * k) * Tp + t] + ln * m.grad[(2 * sl) * Tp + nb];
        gy -= lt * m.grad[(2 * k + 1) * Tp + t] + ln * m.grad[(2 * sl + 1) * Tp + nb];
    }
    a.lamG[t] = gx;
    a.lamG[Tp + t] = gy;
}

// D: node gathers over the incident triangles and the wall bounce-back term
__global__ void __launch_bounds__(128) k_adj_node_d(DevMesh m, Phys c, AdjBufs a) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m.N) return;
    const int Np = m.Np;
    double lh[18];
#pragma unroll
    for (int q = 0; q < 18; ++q) lh[q] = a.lam[q * Np + i];
    double lmu = 0.0, lC = 0.0, lp = 0.0, lux = 0.0, luy = 0.0;
    const double third = 1.0 / 3.0;
    for (int k = m.inc_ptr[i]; k < m.inc_ptr[i + 1]; ++k) {
        const int t = m.inc_tri[k];
        const double bxi = m.inc_bx[k], byi = m.inc_by[k];
        const double A = m.area[t];
        const double* lr = a.lamR + (size_t)t * 18;
#define FELBM_ADJD_Q(q)                                          \
        {                                                        \
            double eb = A * edot<q, double>(bxi, byi);           \
            lh[q] -= eb * lr[q];                                 \
            lh[9 + q] -= eb * lr[9 + q];                         \
        }
        FELBM_ADJD_Q(1) FELBM_ADJD_Q(2) FELBM_ADJD_Q(3) FELBM_ADJD_Q(4)
        FELBM_ADJD_Q(5) FELBM_ADJD_Q(6) FELBM_ADJD_Q(7) FELBM_ADJD_Q(8)
#undef FELBM_ADJD_Q
        const double* le = a.lamE + (size_t)t * 9;
        lC += le[0] * third + le[4] * bxi + le[5] * byi;
        lmu += le[1] * third + a.lamG[t] * bxi + a.lamG[m.Tp + t] * byi;
        lux += le[2] * third;
        luy += le[3] * third;
        lp += le[6] * bxi + le[7] * byi;
    }
    // weak bounce-back: RHS_q(i) += f [L/3 (psi_opp - psi_q)(i) + L/6 (psi_opp - psi_q)(o)]
    // for incoming q on each wall edge (i, o); its transpose seen from node i:
    for (int k = m.winc_ptr[i]; k < m.winc_ptr[i + 1]; ++k) {
        const int e = m.winc_edge[k];
        const int o = m.wall_a[e] == i ? m.wall_b[e] : m.wall_a[e];
        const double L = m.wall_len[e], nx = m.wall_nx[e], ny = m.wall_ny[e];
#define FELBM_ADJW_Q(q)                                                                            \
        {                                                                                          \
            double en = edot<q, double>(nx, ny);                                                   \
            if (en < 0.0) {                                                                        \
                double f = -c.dt * en;                                                             \
                double cg = f * (L * (1.0 / 3.0) * a.lamRHS[q * Np + i] + L * (1.0 / 6.0) * a.lamRHS[q * Np + o]); \
                double ch = f * (L * (1.0 / 3.0) * a.lamRHS[(9 + q) * Np + i] +                    \
                                 L * (1.0 / 6.0) * a.lamRHS[(9 + q) * Np + o]);                   \
                lh[opp(q)] += cg;                                                                  \
                lh[q] -= cg;                                                                       \
                lh[9 + opp(q)] += ch;                                                              \
                lh[9 + q] -= ch;                                                                   \
            }                                                                                      \
        }
        FELBM_ADJW_Q(1) FELBM_ADJW_Q(2) FELBM_ADJW_Q(3) FELBM_ADJW_Q(4)
        FELBM_ADJW_Q(5) FELBM_ADJW_Q(6) FELBM_ADJW_Q(7) FELBM_ADJW_Q(8)
#undef FELBM_ADJW_Q
    }
#pragma unroll
    for (int q = 0; q < 18; ++q) a.lamhat[q * Np + i] = lh[q];
    a.lamMu[i] = lmu;
    a.lamC[i] = lC;
    a.lamP[i] = lp;
    a.lamUx[i] = lux;
    a.lamUy[i] = luy;
}

// E: transpose of mu, of the collision and of the moments -> lambda^n.
__global__ void __launch_bounds__(128) k_adj_node_e(DevMesh m, Phys c, Bufs b, AdjBufs a) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m.N) return;
    const int Np = m.Np;
    const double C = b.C[i], p = b.p[i], ux = b.ux[i], uy = b.uy[i];
    // mu_i = 2 beta C (C-1)(2C-1) - kappa sum_j l_ij C_j + (1/V_i) sum_e phi_e L_e s(C_a, C_b),
    // l_ij = -2 K_ij / V_i with K symmetric
    double lC = a.lamC[i];
    lC += 2.0 * c.beta * (6.0 * C * C - 6.0 * C + 1.0) * a.lamMu[i];
    double kl = 0.0;
    for (int k = m.row_ptr[i]; k < m.row_ptr[i + 1]; ++k) {
        int j = m.col[k];
        kl += a.kval[k] * a.lamMu[j] * m.inv_vol[j];
    }
    lC += 2.0 * c.kappa * kl;
    for (int k = m.winc_ptr[i]; k < m.winc_ptr[i + 1]; ++k) {
        const int e = m.winc_edge[k];
        const int ia = m.wall_a[e], ib = m.wall_b[e];
        const double Ca = b.C[ia], Cb = b.C[ib];
        const double w = a.lamMu[ia] * m.inv_vol[ia] + a.lamMu[ib] * m.inv_vol[ib];
        const double Co = ia == i ? Cb : Ca;
        const double ds = 0.5 - (2.0 * C + Co) * (1.0 / 3.0);   // d s / d C_i
        lC += m.wall_phi[e] * m.wall_len[e] * ds * w;
        if (ia == i) {   // one owner per edge writes its phi_c contribution
            const double sv = 0.5 * (Ca + Cb) - (Ca * Ca + Ca * Cb + Cb * Cb) * (1.0 / 3.0);
            a.dphi[e] += m.wall_len[e] * sv * w;
        }
    }
    // collision: psi_hat = psi - omega(C) (psi - psi_eq(C, p, u)) with
    // g_eq = w (p + rho T / 3), h_eq = w (1 + T) C: lambda_psi_hat pulled back to
    // C, p and u (psi fixed)
    const double inv_tau = fma(C, c.inv_tau_l - c.inv_tau_v, c.inv_tau_v), half = 1.0 / fma(0.5, inv_tau, 1.0);
    const double omega = inv_tau * half, om1 = 1.0 - omega;
    const double drho = c.rho_l - c.rho_v, rho = c.rho_v + C * drho, inv_rho = 1.0 / rho;
    const double uu15 = 1.5 * (ux * ux + uy * uy), rcs2 = rho * (1.0 / 3.0);
    double lh[18], lom = 0.0, lpe = 0.0, lre = 0.0, lCe = 0.0, T0 = 0.0, Tx = 0.0, Ty = 0.0;
#pragma unroll
    for (int q = 0; q < 18; ++q) lh[q] = a.lamhat[q * Np + i];
#define FELBM_ADJC_Q(q)                                                               \
    {                                                                                 \
        const double eu = edot<q>(ux, uy), T = fma(3.0 + 4.5 * eu, eu, -uu15);        \
        const double wg = wq(q) * lh[q], wh = wq(q) * lh[9 + q];                      \
        lom -= lh[q] * (b.psi[q * Np + i] - wq(q) * fma(rcs2, T, p));                 \
        lom -= lh[9 + q] * (b.psi[(9 + q) * Np + i] - wq(q) * fma(C, T, C));          \
        const double t = fma(rcs2, wg, C * wh), te = t * (3.0 + 9.0 * eu);            \
        lpe += wg;                                                                    \
        lre += wg * T;                                                                \
        lCe += fma(wh, T, wh);                                                        \
        T0 += t;                                                                      \
        add_along<q>(Tx, Ty, te);                                                     \
    }
    FELBM_ADJC_Q(0) FELBM_ADJC_Q(1) FELBM_ADJC_Q(2) FELBM_ADJC_Q(3) FELBM_ADJC_Q(4)
    FELBM_ADJC_Q(5) FELBM_ADJC_Q(6) FELBM_ADJC_Q(7) FELBM_ADJC_Q(8)
#undef FELBM_ADJC_Q
    lC += omega * (lCe + drho * (1.0 / 3.0) * lre) + lom * half * half * (c.inv_tau_l - c.inv_tau_v);
    const double lp = a.lamP[i] + omega * lpe;
    const double lux = a.lamUx[i] + omega * (Tx - 3.0 * ux * T0), luy = a.lamUy[i] + omega * (Ty - 3.0 * uy * T0);
    // moments: C = sum h, p = sum g, u = 3 sum e g / rho(C)
    lC -= (ux * lux + uy * luy) * drho * inv_rho;
    const double gx = 3.0 * inv_rho * lux, gy = 3.0 * inv_rho * luy;
#define FELBM_ADJM_Q(q)                                                               \
    a.lam[q * Np + i] = fma(om1, lh[q], lp + edot<q>(gx, gy));                        \
    a.lam[(9 + q) * Np + i] = fma(om1, lh[9 + q], lC);
    FELBM_ADJM_Q(0) FELBM_ADJM_Q(1) FELBM_ADJM_Q(2) FELBM_ADJM_Q(3) FELBM_ADJM_Q(4)
    FELBM_ADJM_Q(5) FELBM_ADJM_Q(6) FELBM_ADJM_Q(7) FELBM_ADJM_Q(8)
#undef FELBM_ADJM_Q
}
