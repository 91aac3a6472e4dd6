// CUDA implementation of the FE-LBM contact-line step for sm_103a (GB300).
//
// Data layout in HBM (all carved from the caller's workspace):
//  * distributions psi: double [18][Np] -- g_0..g_8 then h_0..h_8, direction
//    major, node stride Np = N rounded up to 64 (coalesced node streams);
//  * nodal fields C, p, ux, uy, mu: double [Np];
//  * triangle tables: vertices int [3][Tp], area [Tp], shape gradients
//    double [6][Tp], edge neighbours int [3][Tp] (structure of arrays);
//  * element residual R: double [T][18] (array of structures: the node gather
//    reads one triangle's 18 values as 9 contiguous 16-byte loads);
//  * the 18 FP32 values a node has in the solve (iterates, right-hand side)
//    and in the deviations of FP32 storage: four planes float4 [Np] and one
//    float2 [Np] (vec_at);
//  * node-node pattern (CSR, and ELL with the diagonal first) with the
//    consistent mass and Laplacian coefficients; node -> triangle and node ->
//    wall-edge incidence (CSR);
//  * per block of at most 512 nodes: the layers of nodes around it, its rows of
//    the mass matrix with 16-bit block-local columns, its triangles.
// Nodes are in compact tiles and blocks (recursive bisection), in reverse
// Cuthill-McKee order inside a block, and triangles are sorted by their lowest
// node, so every gather reads a narrow window of the arrays.
//
// One time step (Sec. II.C of arXiv:1708.04678, D2Q9 form) is six kinds of
// kernels, captured once into a CUDA graph:
//   k_collide   moments (eq:velocity, eq:pressure), collision (eqn::collide)
//   k_mu        chemical potential with the patch Laplacian and the wetting
//               flux (eqn:mp_mu, eqn:lapl_int_mp, eqn:bc2)
//   k_gradmu    P0 gradient of mu per triangle
//   k_element   element Laplacian of mu (Sec. II.D), P0 forces at the
//               barycentre (eq:G, eq:H, eq:intF) and the element residual
//               A_T (Phi - e.grad psi_hat) of eq:galerkin_lbm
//   k_rhs       node-centric gather of the streaming right-hand side with
//               weak bounce-back on walls; first Chebyshev iterate (FP32
//               storage on large meshes: k_force32 does k_element's and k_rhs's
//               work on one block, residuals in shared memory)
//   k_block32   sweeps of the consistent-mass solve with the lumped-mass
//               preconditioner, several per launch (FP32 corrections; k_sweep32
//               and k_cheb32 one at a time, k_cheb in FP64); the last adds the
//               increment
// No floating-point atomics: every sum is a fixed-order loop or tree.  The one
// atomic is an integer counter that picks the block of k_diag_fused32 that
// combines the blocks' partials (in block order, whichever block it is).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <utility>
#include <new>
#include <string>
#include <vector>

#include "felbm_internal.h"

namespace felbm {

// ---------------------------------------------------------------- D2Q9 ----
__host__ __device__ constexpr int ex(int q) {
    return q == 1 || q == 5 || q == 8 ? 1 : (q == 3 || q == 6 || q == 7 ? -1 : 0);
}
__host__ __device__ constexpr int ey(int q) {
    return q == 2 || q == 5 || q == 6 ? 1 : (q == 4 || q == 7 || q == 8 ? -1 : 0);
}
__host__ __device__ constexpr double wq(int q) {
    return q == 0 ? 4.0 / 9.0 : (q <= 4 ? 1.0 / 9.0 : 1.0 / 36.0);
}
__host__ __device__ constexpr int opp(int q) {
    return q == 0 ? 0 : (q <= 4 ? (q + 1) % 4 + 1 : (q - 5 + 2) % 4 + 5);
}
static_assert(opp(1) == 3 && opp(2) == 4 && opp(3) == 1 && opp(4) == 2, "opp");
static_assert(opp(5) == 7 && opp(6) == 8 && opp(7) == 5 && opp(8) == 6, "opp");

// e.v for a compile-time direction: only additions, in the type of v (an
// FP32 caller must not be promoted to FP64 -- GB300 runs FP64 at 1/64 rate)
template <int q, class T>
__device__ __forceinline__ T edot(T vx, T vy) {
    T r = T(0);
    if (ex(q) == 1) r = vx;
    if (ex(q) == -1) r = -vx;
    if (ey(q) == 1) r = r + vy;
    if (ey(q) == -1) r = r - vy;
    return r;
}

// ------------------------------------------------------- device tables ----
struct DevMesh {
    int32_t N, T, E, Np, Tp;
    double period_y;
    const int32_t* tri;       // [3][Tp]
    const double* area;       // [Tp]
    const double* grad;       // [6][Tp]
    const float* area32;      // [Tp]   FP32 copies for the FP32-deviation path
    const float* grad32;      // [6][Tp]
    const int32_t* nbr;       // [3][Tp]
    const int32_t* nbr_slot;  // [3][Tp] local index of the shared edge in the neighbour
    const int32_t* row_ptr;   // [N+1]
    const int32_t* col;       // [nnz]
    const double* mval;       // [nnz] consistent mass
    const double* lval;       // [nnz] -2 K_ij / V_i (patch Laplacian of C)
    const double* inv_lumped; // [Np]
    const float* mval32;      // [nnz] FP32 copy of the mass entries
    int32_t ell_w;            // width of the ELL copy (max row length), 0 = none
    const int32_t* ell_col;   // [ell_w][Np] column-major ELL copy of the pattern
    int32_t n_blocks;         // node blocks (contiguous id ranges, HostMesh::blk_ptr)
    int32_t blk_steps;        // most steps of the blocked solve per launch (layers around the blocks), 0 = not blocked
    const int32_t* blk_ptr;   // [n_blocks + 1]
    const int32_t* blk_tri_ptr; // [n_blocks + 1] triangles at the nodes of each block
    const int32_t* blk_tri;
    int32_t max_blk_tri;
    const uint16_t* iell_loc; // [iell_w][Np] iell_tri as indices into the block's triangle list (padding: past its end)
    const int32_t* blk_cnt;   // [n_blocks][kBlockSteps + 1] nodes of a block and its first l layers
    const int32_t* blk_halo_ptr; // [n_blocks + 1]
    const int32_t* blk_halo;  // the layers' nodes, layer by layer
    const int32_t* blk_row;   // [n_blocks + 1] first row of each block in the two tables below
    const float* blk_val;     // per block [ell_w][rows] FP32 mass entries of the block and all layers but the last
    const uint32_t* blk_col;  // per block [ell_w / 2][rows] the columns after the first as pairs of 16-bit indices
                              // in the block's node list
    const float* ell_val;     // [ell_w][Np] FP32 mass entries (padding: own column, 0)
    const double* ell_lval;   // [ell_w][Np] patch-Laplacian coefficients of C (padding 0)
    int32_t iell_w;           // width of the ELL copy of node -> triangle incidence, 0 = none
    const int32_t* iell_tri;  // [iell_w][Np] incident triangle (padding: T, a zero residual row)
    const float* iell_bx32;   // [iell_w][Np] the node's shape gradient in that triangle
    const float* iell_by32;
    const float2* start32;    // [Np] tau_0 / m_i of the FP32 corrections (Start32)
    const float* inv_lumped32;// [Np]
    const double* lumped;     // [Np]
    const double* inv_vol;    // [Np] 1 / V_i
    const int32_t* inc_ptr;   // [N+1]
    const int32_t* inc_tri;   // [ninc]
    const double* inc_bx;     // [ninc]
    const double* inc_by;     // [ninc]
    const float* inc_bx32;    // [ninc]
    const float* inc_by32;    // [ninc]
    const int32_t* wall_a;    // [E]
    const int32_t* wall_b;
    const int32_t* wall_id;
    const double* wall_phi;   // [E] wetting potential phi_c of the edge's wall id
    const double* wall_len;
    const double* wall_nx;
    const double* wall_ny;
    const int32_t* winc_ptr;  // [N+1]
    const int32_t* winc_edge;
    const double* x;          // [Np]
    const double* y;
    const int32_t* perm;      // [N] new -> caller
    const int32_t* iperm;     // [N] caller -> new
};

struct Phys {
    double dt, tau_l, tau_v, rho_l, rho_v, kappa, beta, mobility;
    // element Laplacian of mu: 0 = face-averaged gradients (Sec. II.D),
    // 1 = vertex mean of the nodal patch Laplacian, lapmu_fac * sum l_ij (mu_j - mu_i)
    int lapmu_nodal;
    double lapmu_fac;
    double inv_tau_l, inv_tau_v;
    // FP32 copies, rounded once on the host
    float dt_f, dt3_f, dt2h_f, inv_tau_l_f, inv_tau_v_f, rho_v_f, drho_f, mobility_f;
};

struct Bufs {
    double* psi;     // [18][Np]
    double* C;       // [Np]
    double* p;
    double* ux;
    double* uy;
    double* mu;
    double* gmu;     // [2][Tp]; FELBM_LAPMU_NODAL: the first N hold the nodal Laplacian of mu
    double* lmu;     // alias of gmu (nodal mode)
    double* R;       // [T][18]
    double* rhs;     // [18][Np]
    double* x0;      // [18][Np] FP64 Chebyshev iterates; in the mixed solve
    double* x1;      // [18][Np] they hold x64 (solution) and rho64 (residual)
    double* x64;     // alias of x0
    double* rho64;   // alias of x1
    float* r32;      // [18 Np] FP32 residual of the current correction (layout: vec_at)
    float* e0;       // [18 Np] FP32 iterates
    float* e1;
    // FP32-deviation storage (precision FELBM_FP32_DEV); C above stays FP64
    float* dpsi;     // [18 Np] deviations from equilibrium (layout: vec_at)
    float* p32;      // [Np]
    float* ux32;
    float* uy32;
    float* mu32;
    float* gmu32;    // [2][Tp]; FELBM_LAPMU_NODAL: the first N hold the nodal Laplacian of mu
    float* lmu32;    // alias of gmu32 (nodal mode)
    float* R32;      // [T][18]
    double* stage;   // [18][Np] caller-order staging
    double* in0;     // [18][Np] two caller-order input buffers of felbm_set_state, used in
    double* in1;     //          turn so a copy can run while the previous input converts
    double* diag_part; // [kDiagBlocks][kDiagSlots]
    double* diag_out;  // [kDiagSlots]
    double* Cdiag;     // [Np]
    unsigned* diag_done;   // blocks of k_diag_fused32 finished (0 between launches)
};

// The FP32 vectors of the solve (r32, e0, e1): the moving populations as four
// planes of float4 [Np] (q = 1..4 and 5..8 of g, then of h), then the rest
// populations of g and h as one plane of float2 [Np].  A gathered neighbour is
// one 16-byte word per four right-hand sides.
constexpr int kPlanes = 5;
__device__ __forceinline__ size_t vec_at(int Np, int q18, int i) {
    const int part = q18 >= 9 ? 1 : 0, q = q18 - 9 * part, s = part * 8 + q - 1;
    return q == 0 ? (size_t)16 * Np + 2 * (size_t)i + part : ((size_t)(s >> 2) * Np + i) * 4 + (s & 3);
}
// q18 of component c of plane p
__host__ __device__ constexpr int vec_row(int p, int c) {
    return p == 4 ? 9 * c : 9 * (p >> 1) + 1 + 4 * (p & 1) + c;
}
// Plane p of node i as NV values (NV = 4 for p < 4, 2 for p = 4).
template <int NV>
__device__ __forceinline__ void load_vec(float (&v)[NV], const float* x, int Np, int p, int i) {
    if constexpr (NV == 4) {
        const float4 t = reinterpret_cast<const float4*>(x)[(size_t)p * Np + i];
        v[0] = t.x;
        v[1] = t.y;
        v[2] = t.z;
        v[3] = t.w;
    } else {
        const float2 t = reinterpret_cast<const float2*>(x + (size_t)16 * Np)[i];
        v[0] = t.x;
        v[1] = t.y;
    }
}
template <int NV>
__device__ __forceinline__ void store_vec(float* x, int Np, int p, int i, const float (&v)[NV]) {
    if constexpr (NV == 4)
        reinterpret_cast<float4*>(x)[(size_t)p * Np + i] = make_float4(v[0], v[1], v[2], v[3]);
    else
        reinterpret_cast<float2*>(x + (size_t)16 * Np)[i] = make_float2(v[0], v[1]);
}
template <int NV>
__device__ __forceinline__ void load_shared(float (&v)[NV], const float* x) {
    if constexpr (NV == 4) {
        const float4 t = *reinterpret_cast<const float4*>(x);
        v[0] = t.x;
        v[1] = t.y;
        v[2] = t.z;
        v[3] = t.w;
    } else {
        const float2 t = *reinterpret_cast<const float2*>(x);
        v[0] = t.x;
        v[1] = t.y;
    }
}
template <int NV>
__device__ __forceinline__ void store_shared(float* x, const float (&v)[NV]) {
    if constexpr (NV == 4)
        *reinterpret_cast<float4*>(x) = make_float4(v[0], v[1], v[2], v[3]);
    else
        *reinterpret_cast<float2*>(x) = make_float2(v[0], v[1]);
}

// All 18 values of node i, indexed by q18.
__device__ __forceinline__ void load_all(float (&d)[18], const float* x, int Np, int i) {
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        float v[4];
        load_vec(v, x, Np, p, i);
#pragma unroll
        for (int c = 0; c < 4; ++c) d[vec_row(p, c)] = v[c];
    }
    float v[2];
    load_vec(v, x, Np, 4, i);
    d[0] = v[0];
    d[9] = v[1];
}
__device__ __forceinline__ void store_all(float* x, int Np, int i, const float (&d)[18]) {
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        const float v[4] = {d[vec_row(p, 0)], d[vec_row(p, 1)], d[vec_row(p, 2)], d[vec_row(p, 3)]};
        store_vec(x, Np, p, i, v);
    }
    const float v[2] = {d[0], d[9]};
    store_vec(x, Np, 4, i, v);
}

// A float as a double through the integer pipe: the conversion instruction
// shares the FP64 pipe, whose rate is 1/64 of it.  Exact for every float
// (the rare denormals take the instruction).
__device__ __forceinline__ double widen(float x) {
    const uint32_t u = __float_as_uint(x), e = u & 0x7f800000u;
    if (e == 0u && (u << 1) != 0u) return (double)x;
    const uint32_t bias = e == 0u ? 0u : (e == 0x7f800000u ? 0x70000000u : 0x38000000u);
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + bias)), (int)(u << 29));
}

#include "felbm_start32.cuh"

constexpr int kBlock = 256;
constexpr int kWarpBlocksBelow = 512;   // items per multiprocessor (fp64_block)
constexpr int kDiagBlocks = 608;   // fixed grid (4 x 152 SMs): the reduction order never changes
constexpr int kDiagSlots = 16;
constexpr int kDiagSums = 13;        // slots of the final reduction (k_diag_final, or k_diag_fused32's last block)
constexpr int kDiagStepSlot = 15;    // felbm_diagnostics_enqueue: the step count
constexpr int kSolveResSlot = 13;    // slots 13, 14: sum r^2 and sum b^2 of the checked solve (felbm_solver_check)

// Programmatic dependent launch: a kernel launched with the attribute may
// start while its predecessor drains; it must wait before touching that
// kernel's outputs.  Both are no-ops in a kernel launched without it.  A
// pointer to such outputs is never const __restrict__: the compiler would load
// through the read-only path, ahead of the wait.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" :::); }

// ------------------------------------------------------ K1: collision -----
// Moments of the pre-collision state (C = sum h, p = sum g, rho u = sum e g /
// cs2) and BGK collision towards the equilibria of eqn::g_eq / eqn::f_eq,
// written in place: g_eq = w p + rho cs2 (Gamma - w), h_eq = Gamma C.
// Bound by the FP64 pipe, hence one division instead of six and each direction
// formed with its opposite: 155 us on 520,704 nodes against 207 us.  (With
// T = Gamma / w - 1 and the factors of omega folded it took 115 us, but the
// rounding of Gamma - w, which the 64-bit references share, then differs.)
__global__ void __launch_bounds__(kBlock) k_collide(DevMesh m, Phys c, Bufs b, int do_collide) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m.N) return;
    const int Np = m.Np;
    double g[9], h[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        g[q] = b.psi[q * Np + i];
        h[q] = b.psi[(9 + q) * Np + i];
    }
    double C = 0.0, p = 0.0;
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        C += h[q];
        p += g[q];
    }
    const double mx = (g[1] - g[3]) + (g[5] - g[6]) + (g[8] - g[7]);
    const double my = (g[2] - g[4]) + (g[5] + g[6]) - (g[7] + g[8]);
    const double rho = c.rho_v + C * (c.rho_l - c.rho_v);
    // omega = 1 / (tau + 1/2) = (1/tau) / (1 + 1/(2 tau)); one division for it and 1/rho
    const double inv_tau = fma(C, c.inv_tau_l - c.inv_tau_v, c.inv_tau_v);
    const double half = fma(0.5, inv_tau, 1.0), inv = 1.0 / (rho * half), inv_rho3 = 3.0 * half * inv;
    const double ux = mx * inv_rho3, uy = my * inv_rho3;
    b.C[i] = C;
    b.p[i] = p;
    b.ux[i] = ux;
    b.uy[i] = uy;
    if (!do_collide) return;
    const double omega = inv_tau * rho * inv;
    const double uu15 = 1.5 * (ux * ux + uy * uy), rcs2 = rho * (1.0 / 3.0);
    // a direction and its opposite share 4.5 (e.u)^2
#define FELBM_COLLIDE_Q(q, G0)                                                          \
    {                                                                                   \
        const double G = wq(q) * (G0);                                                  \
        const double geq = wq(q) * p + rcs2 * (G - wq(q));                              \
        b.psi[(q) * Np + i] = g[q] - omega * (g[q] - geq);                              \
        b.psi[(9 + (q)) * Np + i] = h[q] - omega * (h[q] - G * C);                      \
    }
#define FELBM_COLLIDE_PAIR(q)                                                           \
    {                                                                                   \
        const double eu = edot<q>(ux, uy), t = 4.5 * eu * eu;                           \
        FELBM_COLLIDE_Q(q, 1.0 + 3.0 * eu + t - uu15)                                   \
        FELBM_COLLIDE_Q(opp(q), 1.0 - 3.0 * eu + t - uu15)                              \
    }
    FELBM_COLLIDE_Q(0, 1.0 - uu15)
    FELBM_COLLIDE_PAIR(1) FELBM_COLLIDE_PAIR(2) FELBM_COLLIDE_PAIR(5) FELBM_COLLIDE_PAIR(6)
#undef FELBM_COLLIDE_PAIR
#undef FELBM_COLLIDE_Q
}

// --------------------------------------------- K2: chemical potential -----
// mu_i = 2 beta C (C-1)(2C-1) - kappa lap(C)_i with the patch Laplacian
// kappa lap(C)_i = kappa sum_j l_ij C_j + (1/V_i) sum_{wall e at i} -phi_c |e|
// [ (Ca+Cb)/2 - (Ca^2 + Ca Cb + Cb^2)/3 ]  (wall flux of eqn:bc2, C linear on e).
// kW > 0: the sum over the ELL copy of the row (zero padding), its columns and
// coefficients loaded up front so that the gathers of C are in flight
// together; kW = 0: CSR.
template <int kW>
__global__ void __launch_bounds__(kBlock) k_mu(DevMesh m, Phys c, Bufs b) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m.N) return;
    double lap = 0.0;
    int col[kW > 0 ? kW : 1];
    double l[kW > 0 ? kW : 1];
#pragma unroll
    for (int k = 0; k < kW; ++k) {
        col[k] = m.ell_col[k * m.Np + i];
        l[k] = m.ell_lval[k * m.Np + i];
    }
    const int w0 = m.winc_ptr[i], w1 = m.winc_ptr[i + 1];
    const double inv_vol = m.inv_vol[i];
    if constexpr (kW > 0) {
        double Cj[kW];
#pragma unroll
        for (int k = 0; k < kW; ++k) Cj[k] = b.C[col[k]];
#pragma unroll
        for (int k = 0; k < kW; ++k) lap = fma(l[k], Cj[k], lap);
    } else {
        for (int k = m.row_ptr[i]; k < m.row_ptr[i + 1]; ++k) lap += m.lval[k] * b.C[m.col[k]];
    }
    double wall = 0.0;
    for (int k = w0; k < w1; ++k) {
        int e = m.winc_edge[k];
        double Ca = b.C[m.wall_a[e]], Cb = b.C[m.wall_b[e]];
        double s = 0.5 * (Ca + Cb) - (Ca * Ca + Ca * Cb + Cb * Cb) * (1.0 / 3.0);
        wall -= m.wall_phi[e] * m.wall_len[e] * s;
    }
    double C = b.C[i];
    b.mu[i] = 2.0 * c.beta * C * (C - 1.0) * (2.0 * C - 1.0) - (c.kappa * lap + wall * inv_vol);
}

// ------------------------------------------------- K3: grad mu per T ------
__global__ void __launch_bounds__(kBlock) k_gradmu(DevMesh m, Bufs b) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= m.T) return;
    const int Tp = m.Tp;
    int v[3];
    double bx[3], by[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        v[k] = m.tri[k * Tp + t];
        bx[k] = m.grad[(2 * k) * Tp + t];
        by[k] = m.grad[(2 * k + 1) * Tp + t];
    }
    double gx = 0.0, gy = 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const double mu = b.mu[v[k]];
        gx += mu * bx[k];
        gy += mu * by[k];
    }
    b.gmu[t] = gx;
    b.gmu[Tp + t] = gy;
}

// K3' (FELBM_LAPMU_NODAL): nodal Laplacian of mu, the patch Laplacian of C
// applied to mu with zero wall flux (eqn:bc1), lumped P1 volume.
__global__ void __launch_bounds__(kBlock) k_lmu(DevMesh m, Phys c, Bufs b) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m.N) return;
    const double mi = b.mu[i];
    double lap = 0.0;
    for (int k = m.row_ptr[i]; k < m.row_ptr[i + 1]; ++k) lap += m.lval[k] * (b.mu[m.col[k]] - mi);
    b.lmu[i] = c.lapmu_fac * lap;
}

// ------------------------------- K4: forces and element residual ---------
// lap(mu)_T = (1/A) sum_{interior edges} 1/2 (grad mu_T + grad mu_T').nu_k with
// nu_k = -2 A b_k (outward normal x length of the edge opposite vertex k);
// wall edges give 0 (eqn:bc1).  Forces at the barycentre:
//   Phi_g = (e-u).[cs2 grad(rho) (Gamma - w) + mu grad(C) Gamma]
//   Phi_h = [(e-u).(grad C - C/(rho cs2) (grad p - mu grad C)) + M lap(mu)] Gamma
// Residual R_a = A (Phi_a - e_a . grad psi_hat_a), psi_hat P1 on the triangle.
// The FP64 pipe is 87 % busy, so the forces are factored to about 190 FP64
// instructions a triangle: 402 us on 1,040,384 triangles against 639 us for
// the terms as written above.
__global__ void __launch_bounds__(128) k_element(DevMesh m, Phys c, Bufs b) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= m.T) return;
    const int Tp = m.Tp, Np = m.Np;
    int v[3], nb[3];
    double bx[3], by[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        v[k] = m.tri[k * Tp + t];
        nb[k] = m.nbr[k * Tp + t];
        bx[k] = m.grad[(2 * k) * Tp + t];
        by[k] = m.grad[(2 * k + 1) * Tp + t];
    }
    const double A = m.area[t];
    const double third = 1.0 / 3.0;
    double Cv[3], pv[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        Cv[k] = b.C[v[k]];
        pv[k] = b.p[v[k]];
    }
    const double Cs = Cv[0] + Cv[1] + Cv[2];
    const double ux = third * (b.ux[v[0]] + b.ux[v[1]] + b.ux[v[2]]);
    const double uy = third * (b.uy[v[0]] + b.uy[v[1]] + b.uy[v[2]]);
    const double mub = third * (b.mu[v[0]] + b.mu[v[1]] + b.mu[v[2]]);
    const double gCx = fma(Cv[2], bx[2], fma(Cv[1], bx[1], Cv[0] * bx[0]));
    const double gCy = fma(Cv[2], by[2], fma(Cv[1], by[1], Cv[0] * by[0]));
    const double gpx = fma(pv[2], bx[2], fma(pv[1], bx[1], pv[0] * bx[0]));
    const double gpy = fma(pv[2], by[2], fma(pv[1], by[1], pv[0] * by[0]));
    double lapmu = 0.0;
    if (c.lapmu_nodal) {
        lapmu = (b.lmu[v[0]] + b.lmu[v[1]] + b.lmu[v[2]]) * third;
    } else {
        // -sum over interior edges of (grad mu_T + grad mu_T').b_k; the b_k sum
        // to zero, so grad mu_T enters only through the wall edges
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const double gx = nb[k] >= 0 ? -b.gmu[nb[k]] : b.gmu[t], gy = nb[k] >= 0 ? -b.gmu[Tp + nb[k]] : b.gmu[Tp + t];
            lapmu = fma(gx, bx[k], fma(gy, by[k], lapmu));
        }
    }
    const double drho = c.rho_l - c.rho_v, f = Cs / fma(Cs, third * drho, c.rho_v);   // C / (rho cs2)
    const double vhx = gCx - f * (gpx - mub * gCx), vhy = gCy - f * (gpy - mub * gCy);
    const double uu15 = 1.5 * (ux * ux + uy * uy);
    // With T = Gamma / w - 1, s = (e - u).grad C and cs2 grad rho = (drho / 3) grad C:
    //   A Phi_g = w s (P + Q T),  P = A mu,  Q = A (mu + drho / 3)
    //   A Phi_h = w A ((e - u).v + M lap mu) (1 + T)
    // formed for a direction and its opposite together (T = t2 +- 3 e.u); the
    // axis weight 1/9 is folded into the vectors, diagonals take a quarter,
    // rest four times.
    const double P = A * mub, Q = fma(A * third, drho, P), w1 = 1.0 / 9.0, Aw = A * w1;
    const double sx = w1 * gCx, sy = w1 * gCy, su = fma(ux, sx, uy * sy);
    const double vx = Aw * vhx, vy = Aw * vhy, vu = fma(ux, vx, uy * vy) - Aw * (c.mobility * lapmu);
    double abx[3], aby[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        abx[k] = A * bx[k];
        aby[k] = A * by[k];
    }
    double out[18];
    out[0] = -4.0 * su * fma(Q, -uu15, P);
    out[9] = -4.0 * fma(vu, -uu15, vu);
#define FELBM_ELEM_PAIR(q, f)                                                                     \
    {                                                                                             \
        const double eu = edot<q>(ux, uy), t2 = fma(4.5 * eu, eu, -uu15);                         \
        const double tp = fma(3.0, eu, t2), tm = fma(-3.0, eu, t2);                               \
        const double es = edot<q>((f) * sx, (f) * sy), ev = edot<q>((f) * vx, (f) * vy);          \
        const double vp = ev - (f) * vu, vm = -ev - (f) * vu;                                     \
        double gp = (es - (f) * su) * fma(Q, tp, P), gm = (-es - (f) * su) * fma(Q, tm, P);       \
        double hp = fma(vp, tp, vp), hm = fma(vm, tm, vm);                                        \
        for (int k = 0; k < 3; ++k) {                                                             \
            const double eb = edot<q>(abx[k], aby[k]);                                            \
            gp = fma(-b.psi[(q) * Np + v[k]], eb, gp);                                            \
            gm = fma(b.psi[opp(q) * Np + v[k]], eb, gm);                                          \
            hp = fma(-b.psi[(9 + (q)) * Np + v[k]], eb, hp);                                      \
            hm = fma(b.psi[(9 + opp(q)) * Np + v[k]], eb, hm);                                    \
        }                                                                                         \
        out[q] = gp;                                                                              \
        out[opp(q)] = gm;                                                                         \
        out[9 + (q)] = hp;                                                                        \
        out[9 + opp(q)] = hm;                                                                     \
    }
    FELBM_ELEM_PAIR(1, 1.0) FELBM_ELEM_PAIR(2, 1.0) FELBM_ELEM_PAIR(5, 0.25) FELBM_ELEM_PAIR(6, 0.25)
#undef FELBM_ELEM_PAIR
    double2* dst = reinterpret_cast<double2*>(b.R + (size_t)t * 18);
#pragma unroll
    for (int k = 0; k < 9; ++k) dst[k] = make_double2(out[2 * k], out[2 * k + 1]);
}

// The right-hand side of an FP32 correction and its first iterate.
__device__ __forceinline__ void store_start(const Bufs& b, int Np, int i, const double (&r)[18], const Start32& start) {
    float r32[18], e[18];
#pragma unroll
    for (int q = 0; q < 18; ++q) start(r[q], r32[q], e[q]);
    store_all(b.r32, Np, i, r32);
    store_all(b.e1, Np, i, e);
}

// ------------------------------------------- K5: streaming RHS gather -----
// RHS_{i,a} = sum_{T at i} R_{T,a} (dt/3 + dt^2/2 e_a.b_{i,T})
//           - dt sum_{wall e at i} (e_a.n) [L/3 (psi_opp - psi)_i + L/6 (psi_opp - psi)_o]
// (second sum only for incoming directions e_a.n < 0; o = other end of e).
// Also writes the first iterate of the solve x1 = first_scale * RHS / m_i
// (first_scale = 1/theta for the FP64 Chebyshev recurrence, tau_0 for the
// FP32 Richardson steps): in FP64 (FP64 Chebyshev) or, for the
// mixed-precision solve, in FP32 together with the FP32 copy of the
// right-hand side.
//
// Bound by the FP64 pipe (108 FMAs, 60 operations on the weights a node): 162 us on
// 520,704 nodes, 587 us on 2,082,816 (Start32 in FP64: 204 and 789); 256 us on
// 520,704 with the weights formed direction by direction as well.
// One thread per node, or (kSets = 2, consecutive blocks) one per node and set,
// which forms the weights twice but halves a thread's chain of loads and its
// straight-line code -- what a small mesh waits for (2,112 nodes: 15.5 us
// against 17.3).
template <bool kMixed, int kSets>
__global__ void __launch_bounds__(128) k_rhs(DevMesh m, Phys c, Bufs b, double first_scale) {
    constexpr int kN = kSets == 1 ? 18 : 9;
    const int nb = (int)blockIdx.x / kSets, set = (int)blockIdx.x - nb * kSets;
    const int i = nb * (int)blockDim.x + (int)threadIdx.x;
    if (i >= m.N) return;
    const int Np = m.Np;
    double acc[kN];
#pragma unroll
    for (int q = 0; q < kN; ++q) acc[q] = 0.0;
    const double c1 = c.dt * (1.0 / 3.0), c2 = 0.5 * c.dt * c.dt;
    // the next triangle's id and gradient are loaded while this one's residual is in flight
    const int k1 = m.inc_ptr[i + 1];
    int k = m.inc_ptr[i], t = k < k1 ? m.inc_tri[k] : 0;
    double bxi = k < k1 ? m.inc_bx[k] : 0.0, byi = k < k1 ? m.inc_by[k] : 0.0;
    const int w0 = m.winc_ptr[i], w1 = m.winc_ptr[i + 1];
    const float2 s32 = kMixed ? m.start32[i] : make_float2(0.0f, 0.0f);
    const double s = kMixed ? 0.0 : m.inv_lumped[i] * first_scale;
    const double* psi = b.psi + (size_t)9 * set * Np;
    while (k < k1) {
        const double* src = b.R + (size_t)t * 18 + 9 * set;
        double r[kN];
        if constexpr (kSets == 1) {
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                const double2 v2 = reinterpret_cast<const double2*>(src)[q];
                r[2 * q] = v2.x;
                r[2 * q + 1] = v2.y;
            }
        } else {
#pragma unroll
            for (int q = 0; q < 9; ++q) r[q] = src[q];
        }
        const double wx = c2 * bxi, wy = c2 * byi;
        if (++k < k1) {
            t = m.inc_tri[k];
            bxi = m.inc_bx[k];
            byi = m.inc_by[k];
        }
        const double xp = c1 + wx, xm = c1 - wx;      // c1 + c2 e.b for e = (+-1, 0); the diagonals add +-wy
        const double w[9] = {c1, xp, c1 + wy, xm, c1 - wy, xp + wy, xm + wy, xm - wy, xp - wy};
#pragma unroll
        for (int q = 0; q < kN; ++q) acc[q] = fma(r[q], w[q % 9], acc[q]);
    }
    for (int kw = w0; kw < w1; ++kw) {
        const int e = m.winc_edge[kw], a0 = m.wall_a[e], a1 = m.wall_b[e], o = a0 == i ? a1 : a0;
        const double L = m.wall_len[e], nx = m.wall_nx[e], ny = m.wall_ny[e];
        // all populations of both ends first, so that they are in flight together
        double pi[kN], po[kN];
#pragma unroll
        for (int q = 0; q < kN; ++q) {
            if (q % 9 == 0) continue;
            pi[q] = psi[q * Np + i];
            po[q] = psi[q * Np + o];
        }
        const double wi = L * (1.0 / 3.0), wo = L * (1.0 / 6.0);
#define FELBM_WALL_Q(q)                                                                      \
        {                                                                                    \
            const double en = edot<q>(nx, ny);                                               \
            if (en < 0.0) {                                                                  \
                const double f = -c.dt * en;                                                 \
                _Pragma("unroll") for (int h = 0; h < kN; h += 9)                            \
                    acc[h + q] += f * (wi * (pi[h + opp(q)] - pi[h + q]) + wo * (po[h + opp(q)] - po[h + q])); \
            }                                                                                \
        }
        FELBM_WALL_Q(1) FELBM_WALL_Q(2) FELBM_WALL_Q(3) FELBM_WALL_Q(4)
        FELBM_WALL_Q(5) FELBM_WALL_Q(6) FELBM_WALL_Q(7) FELBM_WALL_Q(8)
#undef FELBM_WALL_Q
    }
#pragma unroll
    for (int q = 0; q < kN; ++q) {
        b.rhs[(9 * set + q) * Np + i] = acc[q];
        if (!kMixed) b.x1[(9 * set + q) * Np + i] = acc[q] * s;
    }
    if constexpr (kMixed && kSets == 1) {
        store_start(b, Np, i, acc, Start32{s32, m.inv_lumped + i, first_scale});
    } else if constexpr (kMixed) {
        const Start32 start{s32, m.inv_lumped + i, first_scale};
        float r32[9], e[9];
#pragma unroll
        for (int q = 0; q < 9; ++q) start(acc[q], r32[q], e[q]);
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const float rp[4] = {r32[4 * p + 1], r32[4 * p + 2], r32[4 * p + 3], r32[4 * p + 4]};
            const float ep[4] = {e[4 * p + 1], e[4 * p + 2], e[4 * p + 3], e[4 * p + 4]};
            store_vec(b.r32, Np, 2 * set + p, i, rp);
            store_vec(b.e1, Np, 2 * set + p, i, ep);
        }
        b.r32[vec_at(Np, 9 * set, i)] = r32[0];
        b.e1[vec_at(Np, 9 * set, i)] = e[0];
    }
}

// Start of felbm_mass_solve: rows [0, k) from B ([k][N], caller order), the
// other rows of the planes in use (n4, see k_block32) zero; right-hand side and
// first iterate as k_cheb_start writes them.
template <bool kMixed>
__global__ void __launch_bounds__(kBlock) k_solve_in(DevMesh m, Bufs b, const double* __restrict__ B, int k, int n4,
                                                     double first_scale) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m.N) return;
    const int Np = m.Np, o = m.perm[i];
    const Start32 start{m.start32[i], m.inv_lumped + i, first_scale};
    const double s = m.inv_lumped[i] * first_scale;
    double v[18];
#pragma unroll
    for (int q = 0; q < 18; ++q) v[q] = q < k ? B[(size_t)q * m.N + o] : 0.0;
#pragma unroll
    for (int p = 0; p < kPlanes; ++p) {
        if (p >= n4 && p != 4) continue;
        double x[4] = {0.0, 0.0, 0.0, 0.0};
        float r[4], e[4];
#pragma unroll
        for (int c = 0; c < (p < 4 ? 4 : 2); ++c) {
            const int q = vec_row(p, c);
            b.rhs[q * Np + i] = v[q];
            if (!kMixed) b.x1[q * Np + i] = v[q] * s;
            x[c] = v[q];
        }
        if (kMixed)
#pragma unroll
            for (int c = 0; c < (p < 4 ? 4 : 2); ++c) start(x[c], r[c], e[c]);
        if (kMixed && p < 4) {
            store_vec(b.r32, Np, p, i, r);
            store_vec(b.e1, Np, p, i, e);
        } else if (kMixed) {
            const float r2[2] = {r[0], r[1]}, e2[2] = {e[0], e[1]};
            store_vec(b.r32, Np, 4, i, r2);
            store_vec(b.e1, Np, 4, i, e2);
        }
    }
}

// End of felbm_mass_solve: rows [0, k) of x64 plus (where given) the last
// correction e, to X ([k][N], caller order).
__global__ void __launch_bounds__(kBlock) k_solve_out(DevMesh m, const double* __restrict__ x64,
                                                      const float* __restrict__ e, double* X, int k, int have_x64) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m.N) return;
    const int o = m.perm[i];
#pragma unroll
    for (int q = 0; q < 18; ++q) {
        if (q >= k) continue;
        double x = have_x64 ? x64[(size_t)q * m.Np + i] : 0.0;
        if (e) {
            const double ed = widen(e[vec_at(m.Np, q, i)]);
            x = have_x64 ? x + ed : ed;
        }
        X[(size_t)q * m.N + o] = x;
    }
}

// Start of a standalone solve for the right-hand sides src ([18][Np], copied
// to rhs): x1 = first_scale * B / m_i (1/theta for the FP64 recurrence, tau_0
// for the FP32 steps).
template <bool kMixed>
__global__ void __launch_bounds__(kBlock) k_cheb_start(DevMesh m, Bufs b, const double* src, double first_scale) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m.N) return;
    const int Np = m.Np;
    double s = m.inv_lumped[i] * first_scale;
    double acc[18];
#pragma unroll
    for (int q = 0; q < 18; ++q) {
        acc[q] = src[q * Np + i];
    }
#pragma unroll
    for (int q = 0; q < 18; ++q) {
        if (src != b.rhs) b.rhs[q * Np + i] = acc[q];
        if (!kMixed) b.x1[q * Np + i] = acc[q] * s;
    }
    if constexpr (kMixed) store_start(b, Np, i, acc, Start32{m.start32[i], m.inv_lumped + i, first_scale});
}

// ---------------------------------------------- K6: Chebyshev sweep -------
// x_{k+1} = x_k + a (x_k - x_{k-1}) + c m^{-1} (b - M x_k), the three-term
// Chebyshev recurrence for the lumped-mass preconditioned consistent mass
// matrix, whose spectrum lies in [1/4, 1] on any P1 triangulation.
//   cur  = x_k (gathered), prev = x_{k-1} (own node only; ignored if first),
//   the new iterate overwrites prev, or is added to psi on the last sweep.
__global__ void __launch_bounds__(128) k_cheb(DevMesh m, Bufs b, const double* __restrict__ cur,
                                              double* prev, double a, double cc, int first,
                                              int add_to_psi) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m.N) return;
    const int Np = m.Np;
    double acc[18];
#pragma unroll
    for (int q = 0; q < 18; ++q) acc[q] = 0.0;
    for (int k = m.row_ptr[i]; k < m.row_ptr[i + 1]; ++k) {
        int j = m.col[k];
        double mv = m.mval[k];
#pragma unroll
        for (int q = 0; q < 18; ++q) acc[q] += mv * cur[q * Np + j];
    }
    double s = cc * m.inv_lumped[i];
#pragma unroll
    for (int q = 0; q < 18; ++q) {
        double xk = cur[q * Np + i];
        double xm = first ? 0.0 : prev[q * Np + i];
        double xn = xk + a * (xk - xm) + s * (b.rhs[q * Np + i] - acc[q]);
        if (add_to_psi)
            b.psi[q * Np + i] += xn;
        else
            prev[q * Np + i] = xn;
    }
}

// ------------------------------- K6': mixed-precision mass solve ---------
// Iterative refinement: x <- x + e, where each correction e solves
// M11 e = rho approximately with FP32 Chebyshev sweeps (same recurrence as
// k_cheb, FP32 matrix copy), and the residual rho is carried in FP64 by the
// recurrence rho <- rho - M11 e with M11 in FP64.  GB300 runs FP32 FMA at
// ~70x the FP64 rate, so only the refinement kernels pay FP64 matvecs.
enum Final { kStore = 0, kAddPsi = 1, kAddX64 = 2, kUpdateDev = 3 };

#include "felbm_dev32.cuh"
#include "felbm_adjoint.cuh"

#include "felbm_block32.cuh"

// One step of the FP32 correction solve (CSR rows): Richardson iteration
// x_{k+1} = x_k + tau_k m^{-1} (b - M x_k) with the Chebyshev step sizes
// tau_k = 1 / lambda_k, lambda_k the roots of the degree-K Chebyshev
// polynomial on the spectrum [1/4, 1] of m^{-1} M11 (taken smallest and
// largest alternately, which keeps every partial product below 1 and the
// round-off amplification below 3).  After K steps from x_0 = 0 the error
// polynomial is the same scaled Chebyshev polynomial as for the three-term
// recurrence, but each step reads only x_k (gathered) and b.
//   cur = x_k; the new iterate goes to nxt (or to the final destination).
template <int kFinal>
__global__ void __launch_bounds__(128) k_cheb32(DevMesh m, Phys c, Bufs b, const float* cur,
                                                float* nxt, float tau, int have_x64) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m.N) return;
    const int Np = m.Np;
    float acc[18];
#pragma unroll
    for (int q = 0; q < 18; ++q) acc[q] = 0.0f;
    for (int k = m.row_ptr[i]; k < m.row_ptr[i + 1]; ++k) {
        int j = m.col[k];
        float mv = m.mval32[k];
#pragma unroll
        for (int q = 0; q < 18; ++q) acc[q] = fmaf(mv, cur[vec_at(Np, q, j)], acc[q]);
    }
    float s = tau * m.inv_lumped32[i];
    float d[18];
#pragma unroll
    for (int q = 0; q < 18; ++q) {
        float xk = cur[vec_at(Np, q, i)];
        float xn = fmaf(s, b.r32[vec_at(Np, q, i)] - acc[q], xk);
        if (kFinal == kStore) {
            nxt[vec_at(Np, q, i)] = xn;
        } else if (kFinal == kUpdateDev) {
            d[q] = xn;
        } else {
            double x = have_x64 ? b.x64[q * Np + i] + (double)xn : (double)xn;
            if (kFinal == kAddPsi)
                b.psi[q * Np + i] += x;
            else
                b.x64[q * Np + i] = x;
        }
    }
    if (kFinal == kUpdateDev) dev32_update(m, c, b, i, d);
}

// Programmatic dependent launch: a sweep may be scheduled while its
// predecessor drains; it loads its (read-only) matrix row first and waits for
// the predecessor's results before touching them.  Both instructions are
// no-ops for a kernel launched without the attribute.

// Planes [vec_first(parts, part), vec_first(parts, part + 1)) of the iterate
// belong to one of the `parts` threads of a node (6 threads: five own a plane).
__host__ __device__ constexpr int vec_first(int parts, int part) {
    return parts == 6 ? (part < 5 ? part : 5) : kPlanes * part / parts;
}

// The planes [kP, kEnd) of one node's step; g: all gathered values are loaded
// before the first product (more loads in flight per thread).
template <int kP, int kEnd, int kFinal, int kW, bool kFromRhs>
__device__ __forceinline__ void sweep_planes(const DevMesh& m, const Bufs& b, const float* cur, float* nxt,
                                             int i, const int (&col)[kW], const float (&val)[kW],
                                             const float (&sc)[kFromRhs ? kW : 1], float s, int have_x64,
                                             float (&d)[18]) {
    if constexpr (kP < kEnd) {
        constexpr int NV = kP < 4 ? 4 : 2;
        const int Np = m.Np;
        float g[kW][NV], rr[NV];
        const float* src = kFromRhs ? b.r32 : cur;
#pragma unroll
        for (int k = 0; k < kW; ++k) load_vec(g[k], src, Np, kP, col[k]);
        if constexpr (kFromRhs) {
            // the row's first column is the node itself
#pragma unroll
            for (int c = 0; c < NV; ++c) rr[c] = g[0][c];
#pragma unroll
            for (int k = 0; k < kW; ++k)
#pragma unroll
                for (int c = 0; c < NV; ++c) g[k][c] *= sc[k];
        } else {
            load_vec(rr, b.r32, Np, kP, i);
        }
        float xn[NV];
#pragma unroll
        for (int c = 0; c < NV; ++c) {
            float acc = 0.0f;
#pragma unroll
            for (int k = 0; k < kW; ++k) acc = fmaf(val[k], g[k][c], acc);
            xn[c] = fmaf(s, rr[c] - acc, g[0][c]);
        }
        if constexpr (kFinal == kStore) {
            store_vec(nxt, Np, kP, i, xn);
        } else if constexpr (kFinal == kUpdateDev) {
#pragma unroll
            for (int c = 0; c < NV; ++c) d[vec_row(kP, c)] = xn[c];
        } else {
#pragma unroll
            for (int c = 0; c < NV; ++c) {
                const int r = vec_row(kP, c) * Np + i;
                const double x = have_x64 ? b.x64[r] + (double)xn[c] : (double)xn[c];
                if (kFinal == kAddPsi)
                    b.psi[r] += x;
                else
                    b.x64[r] = x;
            }
        }
        sweep_planes<kP + 1, kEnd, kFinal, kW, kFromRhs>(m, b, cur, nxt, i, col, val, sc, s, have_x64, d);
    }
}

template <int kPart, int kParts, int kFinal, int kW, bool kFromRhs>
__device__ __forceinline__ void sweep_part(int part, const DevMesh& m, const Bufs& b, const float* cur,
                                           float* nxt, int i, const int (&col)[kW], const float (&val)[kW],
                                           const float (&sc)[kFromRhs ? kW : 1], float s, int have_x64, float (&d)[18]) {
    if constexpr (kPart < kParts) {
        if (part == kPart)
            sweep_planes<vec_first(kParts, kPart), vec_first(kParts, kPart + 1), kFinal, kW, kFromRhs>(
                m, b, cur, nxt, i, col, val, sc, s, have_x64, d);
        else
            sweep_part<kPart + 1, kParts, kFinal, kW, kFromRhs>(part, m, b, cur, nxt, i, col, val, sc, s, have_x64, d);
    }
}

// The FP32 step of k_cheb32 on the ELL copy of the pattern (kW entries per
// row, the node's own first, padded with the own column and value 0).  Row
// indices and values are loaded up front (coalesced, column-major).
// kParts threads per node, each owning some of the iterate's planes; the
// field update needs all of them in one thread.  The parts of one node block
// are consecutive blocks (blockIdx.x = kParts * node block + part), so they
// run together and share the block's matrix rows through L2 instead of
// fetching them from DRAM once per part.
template <int kFinal, int kW, int kParts, bool kFromRhs = false>
__global__ void __launch_bounds__(128) k_sweep32(DevMesh m, Phys c, Bufs b, const float* cur,
                                                 float* nxt, float tau, int have_x64, float tau0) {
    pdl_release();
    static_assert(kFinal != kUpdateDev || kParts == 1, "the field update needs the whole node");
    const int nb = (int)blockIdx.x / kParts;
    const int i = nb * (int)blockDim.x + (int)threadIdx.x;
    const int part = (int)blockIdx.x - nb * kParts;
    const int Np = m.Np;
    int col[kW];
    float val[kW];
    // kFromRhs: the first step of the solve, whose iterate x_0 = tau_0 b / m
    // is formed here from the right-hand side (the RHS kernel stores b only)
    float sc[kFromRhs ? kW : 1];
    if (i < m.N) {
#pragma unroll
        for (int k = 0; k < kW; ++k) {
            col[k] = m.ell_col[k * Np + i];
            val[k] = m.ell_val[k * Np + i];
        }
        if constexpr (kFromRhs) {
#pragma unroll
            for (int k = 0; k < kW; ++k) sc[k] = m.inv_lumped32[col[k]] * tau0;
        }
    }
    const float s = tau * (i < m.N ? m.inv_lumped32[i] : 0.0f);
    pdl_wait();
    if (i >= m.N) return;
    float d[18];
    sweep_part<0, kParts, kFinal, kW, kFromRhs>(part, m, b, cur, nxt, i, col, val, sc, s, have_x64, d);
    if constexpr (kFinal == kUpdateDev) dev32_update(m, c, b, i, d);
}

// x <- x + e ; rho <- rho - M11 e (FP64) ; FP32 copy of rho and the first
// iterate of the next correction, tau_0 rho / m.  One thread per node and
// plane (consecutive blocks, which share the rows through L2): five times the
// warps and a fifth of the straight-line code, which is what a small mesh
// waits for (2,112 nodes: 8.3 us against 15.3 for all planes in a thread; on
// 520,704 nodes 212 against 197 us).  Bound by the FP64 pipe; with conversion
// instructions for the 126 gathered values it took 377 us.
template <int NV>
__device__ __forceinline__ void refine_plane(const DevMesh& m, const Bufs& b, const float* e,
                                             float* next_first, int first_round, double tau0, int p, int i) {
    const int Np = m.Np, k1 = m.row_ptr[i + 1];
    int k = m.row_ptr[i];
    const Start32 start{m.start32[i], m.inv_lumped + i, tau0};
    // every load of the node itself before the first store (the compiler keeps
    // their order, and one at a time they cost a latency each)
    const size_t at = (size_t)(NV == 2 ? 0 : 9 * (p >> 1) + 1 + 4 * (p & 1)) * Np + i, stride = (size_t)(NV == 2 ? 9 : 1) * Np;
    float ei[NV];
    double acc[NV], ro[NV], xo[NV];
    load_vec(ei, e, Np, p, i);
#pragma unroll
    for (int c = 0; c < NV; ++c) {
        acc[c] = 0.0;
        ro[c] = first_round ? b.rhs[at + c * stride] : b.rho64[at + c * stride];
        xo[c] = first_round ? 0.0 : b.x64[at + c * stride];
    }
#pragma unroll 4
    for (; k < k1; ++k) {
        const double mv = m.mval[k];
        float ej[NV];
        load_vec(ej, e, Np, p, m.col[k]);
#pragma unroll
        for (int c = 0; c < NV; ++c) acc[c] = fma(mv, widen(ej[c]), acc[c]);
    }
    double rn[NV];
    float r32[NV], first[NV];
#pragma unroll
    for (int c = 0; c < NV; ++c) {
        const double ed = widen(ei[c]);
        rn[c] = ro[c] - acc[c];
        b.x64[at + c * stride] = first_round ? ed : xo[c] + ed;
        b.rho64[at + c * stride] = rn[c];
        start(rn[c], r32[c], first[c]);
    }
    store_vec(b.r32, Np, p, i, r32);
    store_vec(next_first, Np, p, i, first);
}

__global__ void __launch_bounds__(128) k_refine(DevMesh m, Bufs b, const float* e,
                                                float* next_first, int first_round, double tau0, int n4) {
    const int nb = (int)blockIdx.x / (n4 + 1), l = (int)blockIdx.x - (n4 + 1) * nb, p = l < n4 ? l : 4;
    const int i = nb * (int)blockDim.x + (int)threadIdx.x;
    if (i >= m.N) return;
    if (p < 4)
        refine_plane<4>(m, b, e, next_first, first_round, tau0, p, i);
    else
        refine_plane<2>(m, b, e, next_first, first_round, tau0, p, i);
}

// The last correction's iterate e added up (FP64): psi += x64 + e (the time
// step), or x64 += e.  A kernel of its own: inside k_block32 the 108 extra
// loads and stores a node spill its registers (136 us against 66 + 48 us on
// 520,704 nodes).
template <bool kPsi>
__global__ void __launch_bounds__(128) k_add64(DevMesh m, Bufs b, const float* e, int have_x64) {
    pdl_wait();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m.N) return;
    const int Np = m.Np;
    float ei[18];
    double xo[18], po[18];
    load_all(ei, e, Np, i);
#pragma unroll
    for (int q = 0; q < 18; ++q) {
        xo[q] = have_x64 ? b.x64[q * Np + i] : 0.0;
        if (kPsi) po[q] = b.psi[q * Np + i];
    }
#pragma unroll
    for (int q = 0; q < 18; ++q) {
        const double x = have_x64 ? xo[q] + widen(ei[q]) : widen(ei[q]);
        if (kPsi)
            b.psi[q * Np + i] = po[q] + x;
        else
            b.x64[q * Np + i] = x;
    }
}

// -------------------------------------- solve residual (opt-in check) ----
// Before the last step of the solve: sum over nodes and right-hand sides of
// r^2, r = b_k - M x (FP32 rows, as the steps form them; b_k the current
// correction's right-hand side), and of the solve's original right-hand
// side squared (FP64 rhs for the mixed solve, the FP32 copy for FP32
// storage).  Fixed grid, per-block partials, one ordered final sum: the
// result does not depend on scheduling.
template <bool kRhs64>
__global__ void __launch_bounds__(kBlock) k_solve_resid(DevMesh m, Bufs b, const float* __restrict__ x,
                                                        double* part) {
    const int Np = m.Np;
    double rr = 0.0, bb = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m.N; i += gridDim.x * blockDim.x) {
        const int k0 = m.row_ptr[i], k1 = m.row_ptr[i + 1];
        for (int q = 0; q < 18; ++q) {
            float acc = 0.0f;
            for (int k = k0; k < k1; ++k) acc = fmaf(m.mval32[k], x[vec_at(Np, q, m.col[k])], acc);
            const float r = b.r32[vec_at(Np, q, i)] - acc;
            rr += (double)r * (double)r;
            const double bq = kRhs64 ? b.rhs[q * Np + i] : (double)b.r32[vec_at(Np, q, i)];
            bb += bq * bq;
        }
    }
    __shared__ double sh[2][kBlock / 32];
    for (int o = 16; o > 0; o >>= 1) {
        rr += __shfl_down_sync(0xffffffffu, rr, o);
        bb += __shfl_down_sync(0xffffffffu, bb, o);
    }
    if ((threadIdx.x & 31) == 0) {
        sh[0][threadIdx.x >> 5] = rr;
        sh[1][threadIdx.x >> 5] = bb;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, c = 0.0;
        for (int w = 0; w < kBlock / 32; ++w) {
            a += sh[0][w];
            c += sh[1][w];
        }
        part[2 * blockIdx.x] = a;
        part[2 * blockIdx.x + 1] = c;
    }
}
__global__ void k_solve_resid_final(const double* __restrict__ part, int n, double* out) {
    double a = 0.0, c = 0.0;
    for (int k = 0; k < n; ++k) {
        a += part[2 * k];
        c += part[2 * k + 1];
    }
    out[0] = a;
    out[1] = c;
}

// ----------------------------------------------- permutation kernels ------
__global__ void k_scatter_in(DevMesh m, const double* __restrict__ stage, double* dst, int rows) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m.N) return;
    int o = m.perm[i];
    for (int q = 0; q < rows; ++q) dst[q * m.Np + i] = stage[(size_t)q * m.N + o];
}
__global__ void k_gather_out(DevMesh m, const double* __restrict__ src, double* stage, int rows) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m.N) return;
    int o = m.perm[i];
    for (int q = 0; q < rows; ++q) stage[(size_t)q * m.N + o] = src[q * m.Np + i];
}
// Initial state at equilibrium with the fields C0, p0, u0 (caller order in
// stage: C0 [N], then p0 [N] if has_p, then u0 [2N] as x, y if has_u; the
// missing ones are zero): g = w p + rho cs2 (Gamma(u) - w), h = Gamma(u) C
// (eqn::g_eq, eqn::f_eq), rho = C rho_l + (1 - C) rho_v.
__global__ void k_init_state(DevMesh m, Phys c, const double* __restrict__ stage, double* psi, int has_p,
                             int has_u) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m.N) return;
    const int o = m.perm[i], N = m.N;
    const double C = stage[o];
    const double p = has_p ? stage[N + o] : 0.0;
    const double* u = stage + (has_p ? 2 : 1) * (size_t)N;
    const double ux = has_u ? u[o] : 0.0, uy = has_u ? u[N + o] : 0.0;
    const double rcs2 = (c.rho_v + C * (c.rho_l - c.rho_v)) * (1.0 / 3.0);
    const double uu15 = 1.5 * (ux * ux + uy * uy);
#define FELBM_INIT_Q(q)                                                      \
    {                                                                        \
        const double eu = edot<q>(ux, uy);                                   \
        const double G = wq(q) * (1.0 + 3.0 * eu + 4.5 * eu * eu - uu15);    \
        psi[q * m.Np + i] = wq(q) * p + rcs2 * (G - wq(q));                  \
        psi[(9 + q) * m.Np + i] = G * C;                                     \
    }
    FELBM_INIT_Q(0) FELBM_INIT_Q(1) FELBM_INIT_Q(2) FELBM_INIT_Q(3) FELBM_INIT_Q(4)
    FELBM_INIT_Q(5) FELBM_INIT_Q(6) FELBM_INIT_Q(7) FELBM_INIT_Q(8)
#undef FELBM_INIT_Q
}

// ------------------------------------------------------ diagnostics -------
// Slots: 0 mass, 1 sum rho|u|^2, 2 band weight, 3 band sum m rho|u|^2,
// 4 liquid weight, 5 liquid sum m p, 6 vapour weight, 7 vapour sum m p,
// 8 unused, 9 non-finite count, 10 max |u|^2 (node pass);
// 11 wetted length, 12 max contour height (edge pass).
struct DiagReq {
    double cx, cy, R, band;
    double period_x, period_y;
    int substrate;
    int use_band;
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
    return v;
}

__device__ __forceinline__ double min_image(double d, double L) {
    return L > 0.0 ? d - L * rint(d / L) : d;
}

// Block reduction of NS sums and NM maxima to out[0 .. NS+NM), in a fixed
// order.  FP64 adds run at 1/64 of the FP32 rate on this part, so every
// value is added once: the threads' partials go to shared memory, NV x NW
// threads each combine one interleaved segment of 32, and NV threads combine
// the NW segments (a warp-shuffle tree in every lane would add each value
// five times over).
template <int NS, int NM>
__device__ void block_reduce_store(double (&s)[NS], double (&mx)[NM], double* out) {
    constexpr int NV = NS + NM, NW = kBlock / 32, L = kBlock + 2;
    __shared__ double sh[NV][L];
    __shared__ double part[NV][NW];
#pragma unroll
    for (int k = 0; k < NV; ++k) sh[k][threadIdx.x] = k < NS ? s[k] : mx[k - NS];
    __syncthreads();
    if (threadIdx.x < NV * NW) {
        const int k = threadIdx.x / NW, seg = threadIdx.x - k * NW;
        double r = sh[k][seg];
        for (int j = 1; j < 32; ++j) r = k < NS ? r + sh[k][seg + NW * j] : fmax(r, sh[k][seg + NW * j]);
        part[k][seg] = r;
    }
    __syncthreads();
    if (threadIdx.x < NV) {
        const int k = threadIdx.x;
        double r = part[k][0];
        for (int w = 1; w < NW; ++w) r = k < NS ? r + part[k][w] : fmax(r, part[k][w]);
        out[k] = r;
    }
}

// Comparisons of a double with a positive threshold on the bit patterns (the
// integer pipe; FP64 compares share the 1/64-rate FP64 pipe).  For x >= 0 the
// patterns order like the values, and every x with the sign bit set is a
// negative integer, below the pattern of t.  NaNs compare by their pattern;
// non-finite states are reported through their own slot.
__device__ __forceinline__ bool ge_pos(double x, double t) { return __double_as_longlong(x) >= __double_as_longlong(t); }
__device__ __forceinline__ bool le_pos(double x, double t) { return __double_as_longlong(x) <= __double_as_longlong(t); }
__device__ __forceinline__ bool finite_bits(double x) {
    return (__double_as_longlong(x) & 0x7ff0000000000000LL) != 0x7ff0000000000000LL;
}

// Per-node contributions (slots 0..9 sums, one max); writes the node's C.
template <bool kDev32>
__device__ __forceinline__ void diag_node(const DevMesh& m, const Phys& c, const Bufs& b, const DiagReq& rq,
                                          int i, double (&s)[10], double (&mx)[1]) {
    const int Np = m.Np;
    double C = 0, p = 0, uu, ruu;
    bool finite;
    if (kDev32) {
        // FP32 fields: |u|^2 and rho |u|^2 in FP32 (FP64 runs at 1/64 rate), summed in FP64
        C = b.C[i];
        p = b.p32[i];
        const float uxf = b.ux32[i], uyf = b.uy32[i];
        const float rhof = c.rho_v_f + (float)C * c.drho_f;
        const float uuf = uxf * uxf + uyf * uyf;
        uu = uuf;
        ruu = rhof * uuf;
        float dsum = 0.0f, dev[18];
        load_all(dev, b.dpsi, Np, i);
#pragma unroll
        for (int q = 0; q < 18; ++q) dsum += dev[q];
        // non-finite deviations are reported too
        finite = finite_bits(C) && isfinite(b.p32[i]) && isfinite(uuf) && isfinite(dsum);
    } else {
        double g[9];
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            g[q] = b.psi[q * Np + i];
            p += g[q];
            C += b.psi[(9 + q) * Np + i];
        }
        double mxm = (g[1] - g[3]) + (g[5] - g[6]) + (g[8] - g[7]);
        double mym = (g[2] - g[4]) + (g[5] + g[6]) - (g[7] + g[8]);
        const double rho = c.rho_v + C * (c.rho_l - c.rho_v);
        const double ux = 3.0 * mxm / rho, uy = 3.0 * mym / rho;
        uu = ux * ux + uy * uy;
        ruu = rho * uu;
        finite = isfinite(C) && isfinite(p) && isfinite(uu);
    }
    double w = m.lumped[i];
    b.Cdiag[i] = C;
    if (!finite) s[9] += 1.0;
    s[0] += w * C;
    s[1] += ruu;
    if (rq.use_band) {
        double dx = min_image(m.x[i] - rq.cx, rq.period_x), dy = min_image(m.y[i] - rq.cy, rq.period_y);
        double r = sqrt(dx * dx + dy * dy);
        if (fabs(r - rq.R) <= rq.band) {
            s[2] += w;
            s[3] += w * ruu;
        }
    }
    if (ge_pos(C, 0.95)) {
        s[4] += w;
        s[5] += w * p;
    }
    if (le_pos(C, 0.05)) {
        s[6] += w;
        s[7] += w * p;
    }
    mx[0] = fmax(mx[0], uu);
}

// Wetted length of a substrate wall edge (C linear along it).
__device__ __forceinline__ void diag_wall(const DevMesh& m, const double* Cn, const DiagReq& rq, int e, double& wet) {
    if (m.wall_id[e] != rq.substrate) return;
    double Ca = Cn[m.wall_a[e]], Cb = Cn[m.wall_b[e]], L = m.wall_len[e];
    const bool a = ge_pos(Ca, 0.5), bb = ge_pos(Cb, 0.5);
    if (a && bb)
        wet += L;
    else if (a || bb) {
        double hi = fmax(Ca, Cb), lo = fmin(Ca, Cb);
        wet += L * (hi - 0.5) / (hi - lo);
    }
}

// Highest crossing of the C = 1/2 contour on the edges of a triangle.
__device__ __forceinline__ void diag_tri(const DevMesh& m, const double* Cn, const DiagReq& rq, int t, double& ymax) {
    const int Tp = m.Tp;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        int ia = m.tri[((k + 1) % 3) * Tp + t], ic = m.tri[((k + 2) % 3) * Tp + t];
        double Ca = Cn[ia], Cc = Cn[ic];
        if (ge_pos(Ca, 0.5) != ge_pos(Cc, 0.5)) {
            double tt = (0.5 - Ca) / (Cc - Ca);
            double dy = min_image(m.y[ic] - m.y[ia], rq.period_y);
            ymax = fmax(ymax, m.y[ia] + tt * dy);
        }
    }
}

template <bool kDev32>
__global__ void __launch_bounds__(kBlock) k_diag_nodes(DevMesh m, Phys c, Bufs b, DiagReq rq) {
    double s[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    double mx[1] = {0.0};
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m.N; i += gridDim.x * blockDim.x)
        diag_node<kDev32>(m, c, b, rq, i, s, mx);
    block_reduce_store<10, 1>(s, mx, b.diag_part + (size_t)blockIdx.x * kDiagSlots);
}

// wetted length on substrate wall edges; highest crossing of the C = 1/2
// contour on triangle edges (both from the nodal C written by k_diag_nodes)
__global__ void __launch_bounds__(kBlock) k_diag_edges(DevMesh m, Bufs b, DiagReq rq) {
    double s[1] = {0.0};
    double mx[1] = {-1e300};
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < m.E; e += gridDim.x * blockDim.x)
        diag_wall(m, b.Cdiag, rq, e, s[0]);
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < m.T; t += gridDim.x * blockDim.x)
        diag_tri(m, b.Cdiag, rq, t, mx[0]);
    block_reduce_store<1, 1>(s, mx, b.diag_part + (size_t)blockIdx.x * kDiagSlots + 11);
}

// Tables of the connected components (groups) of the mesh.
struct GroupTables {
    const int32_t* node_begin;   // [G] internal node range of each group
    const int32_t* node_end;
    const int32_t* tri_begin;    // [G] triangle range
    const int32_t* tri_end;
    const int32_t* wall_ptr;     // [G+1] wall edges of each group (CSR)
    const int32_t* wall_edge;
    DiagReq* reqs;               // [G] per-group request (written by the host per call)
    double* out;                 // [G][kDiagSlots]
    int32_t* cta_groups;         // [G] groups run by k_step_cta32
};

// One block per group: the same slots as k_diag_nodes/k_diag_edges, reduced
// over the group's own nodes, wall edges and triangles in a fixed order.
template <bool kDev32>
__global__ void __launch_bounds__(kBlock) k_diag_groups(DevMesh m, Phys c, Bufs b, GroupTables gt) {
    const int g = blockIdx.x;
    const DiagReq rq = gt.reqs[g];
    double s[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    double mx[1] = {0.0};
    for (int i = gt.node_begin[g] + threadIdx.x; i < gt.node_end[g]; i += blockDim.x)
        diag_node<kDev32>(m, c, b, rq, i, s, mx);
    __syncthreads();   // the group's C (Cdiag) is complete; it is read below
    double we[1] = {0.0};
    double ym[1] = {-1e300};
    for (int k = gt.wall_ptr[g] + threadIdx.x; k < gt.wall_ptr[g + 1]; k += blockDim.x)
        diag_wall(m, b.Cdiag, rq, gt.wall_edge[k], we[0]);
    for (int t = gt.tri_begin[g] + threadIdx.x; t < gt.tri_end[g]; t += blockDim.x) diag_tri(m, b.Cdiag, rq, t, ym[0]);
    block_reduce_store<10, 1>(s, mx, gt.out + (size_t)g * kDiagSlots);
    block_reduce_store<1, 1>(we, ym, gt.out + (size_t)g * kDiagSlots + 11);
}

// One warp per slot: lane l reduces blocks l, l+32, ... in order, then a
// fixed shuffle tree -- the same order on every call.
__global__ void k_diag_final(Bufs b) {
    int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (k >= kDiagSums) return;
    bool is_max = (k == 10 || k == 12);
    double r = is_max ? -1e300 : 0.0;
    // every lane's partials loaded before they are combined (in block order)
    constexpr int kPer = (kDiagBlocks + 31) / 32;
    double v[kPer];
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int blk = lane + 32 * j;
        v[j] = blk < kDiagBlocks ? b.diag_part[(size_t)blk * kDiagSlots + k] : (is_max ? -1e300 : 0.0);
    }
#pragma unroll
    for (int j = 0; j < kPer; ++j) r = is_max ? fmax(r, v[j]) : r + v[j];
    r = is_max ? warp_max(r) : warp_sum(r);
    if (lane == 0) b.diag_out[k] = r;
}

// FP32-deviation states keep C in FP64, so the edge pass needs no node pass
// before it: one kernel accumulates every slot, and the last block to finish
// (a device-scope counter after a fence; no block waits for another) combines
// the blocks' partials in block order exactly as k_diag_final does.
__global__ void __launch_bounds__(kBlock) k_diag_fused32(DevMesh m, Phys c, Bufs b, DiagReq rq) {
    double s[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    double mx[1] = {0.0};
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m.N; i += gridDim.x * blockDim.x)
        diag_node<true>(m, c, b, rq, i, s, mx);
    double we[1] = {0.0};
    double ym[1] = {-1e300};
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < m.E; e += gridDim.x * blockDim.x)
        diag_wall(m, b.C, rq, e, we[0]);
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < m.T; t += gridDim.x * blockDim.x)
        diag_tri(m, b.C, rq, t, ym[0]);
    block_reduce_store<10, 1>(s, mx, b.diag_part + (size_t)blockIdx.x * kDiagSlots);
    block_reduce_store<1, 1>(we, ym, b.diag_part + (size_t)blockIdx.x * kDiagSlots + 11);
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(b.diag_done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int lane = threadIdx.x & 31;
    for (int k = threadIdx.x >> 5; k < kDiagSums; k += kBlock / 32) {
        const bool is_max = (k == 10 || k == 12);
        constexpr int kPer = (kDiagBlocks + 31) / 32;
        double v[kPer];
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const int blk = lane + 32 * j;
            v[j] = blk < kDiagBlocks ? __ldcg(b.diag_part + (size_t)blk * kDiagSlots + k) : (is_max ? -1e300 : 0.0);
        }
        double r = is_max ? -1e300 : 0.0;
#pragma unroll
        for (int j = 0; j < kPer; ++j) r = is_max ? fmax(r, v[j]) : r + v[j];
        r = is_max ? warp_max(r) : warp_sum(r);
        if (lane == 0) b.diag_out[k] = r;
    }
    if (threadIdx.x == 0) *b.diag_done = 0u;
}

// ------------------------------------------- one CTA per batch member ------
// The whole FP32-deviation step of one small batch member in one thread
// block: the member is a contiguous range of nodes and triangles (its
// group), every phase is a block-stride loop over that range, and
// __syncthreads() orders the phases -- no kernel boundary and no grid-wide
// synchronisation inside the step.  Data written in one phase is read in
// the next through plain (coherent) loads.
constexpr int kCtaThreads = 512;
constexpr int kMaxSweeps = 64;
struct ChebCoef {
    float tau[kMaxSweeps];   // Richardson step sizes of the FP32 solve (see k_cheb32)
};

// One FP32 step of a node for the per-member schedule, the 18 values of a
// neighbour as five vector loads (one value at a time, a warp's load strides 16
// bytes: 675 against 361 us a step on 64 members of 1,012 to 3,960 nodes).
__device__ __forceinline__ void sweep32_node(const DevMesh& m, const Phys& c, const Bufs& b, int i,
                                             const float* cur, float* nxt, float tau, bool update) {
    const int Np = m.Np;
    float acc[18];
#pragma unroll
    for (int q = 0; q < 18; ++q) acc[q] = 0.0f;
    const auto add = [&](int j, float v) {
        float x[18];
        load_all(x, cur, Np, j);
#pragma unroll
        for (int q = 0; q < 18; ++q) acc[q] = fmaf(v, x[q], acc[q]);
    };
    if (m.ell_w > 0)
        for (int k = 0; k < m.ell_w; ++k) add(m.ell_col[k * Np + i], m.ell_val[k * Np + i]);
    else
        for (int k = m.row_ptr[i]; k < m.row_ptr[i + 1]; ++k) add(m.col[k], m.mval32[k]);
    const float s = tau * m.inv_lumped32[i];
    float d[18], r[18];
    load_all(d, cur, Np, i);
    load_all(r, b.r32, Np, i);
#pragma unroll
    for (int q = 0; q < 18; ++q) d[q] = fmaf(s, r[q] - acc[q], d[q]);
    if (update)
        dev32_update(m, c, b, i, d);
    else
        store_all(nxt, Np, i, d);
}

__global__ void __launch_bounds__(kCtaThreads, 1) k_step_cta32(DevMesh m, Phys c, Bufs b, GroupTables gt,
                                                               const int32_t* __restrict__ groups, ChebCoef cf,
                                                               int sweeps, float tau0) {
    const int g = groups[blockIdx.x];
    const int n0 = gt.node_begin[g], n1 = gt.node_end[g], t0 = gt.tri_begin[g], t1 = gt.tri_end[g];
    const int tid = threadIdx.x, nt = blockDim.x;
    for (int i = n0 + tid; i < n1; i += nt) mu32_node(m, c, b, i);
    __syncthreads();
    if (c.lapmu_nodal)
        for (int i = n0 + tid; i < n1; i += nt) lmu32_node(m, c, b, i);
    else
        for (int t = t0 + tid; t < t1; t += nt) gradmu32_tri(m, b, t);
    __syncthreads();
    for (int t = t0 + tid; t < t1; t += nt) element32_tri(m, c, b, t);
    __syncthreads();
    for (int i = n0 + tid; i < n1; i += nt) rhs32_node(m, c, b, i, tau0);
    __syncthreads();
    float* cur = b.e1;
    float* prv = b.e0;
    for (int k = 1; k < sweeps; ++k) {
        const bool last = k == sweeps - 1;
        for (int i = n0 + tid; i < n1; i += nt) sweep32_node(m, c, b, i, cur, prv, cf.tau[k], last);
        __syncthreads();
        float* tmp = cur;
        cur = prv;
        prv = tmp;
    }
}

// ------------------------------------------- FP64 FMA rate (instrument) --
// Eight independent FP64 FMA chains per thread: the issue rate of the FP64
// pipe, the roof of the FP64 kernels.  The result is stored only when it is
// a value the chains cannot reach, so the work is kept but nothing is written.
__device__ double g_fma_sink;
__global__ void __launch_bounds__(256) k_fp64_fma_rate(int iters, double a) {
    double x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = (double)(threadIdx.x + k) * 1e-3;
    for (int it = 0; it < iters; ++it)
#pragma unroll
        for (int k = 0; k < 8; ++k) x[k] = fma(x[k], a, 1e-9);
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) s += x[k];
    if (s == -1.0) g_fma_sink = s;
}

// --------------------------------------------------------- host side ------
static int cuda_fail(cudaError_t e, const char* what) {
    char buf[256];
    snprintf(buf, sizeof buf, "%s: %s", what, cudaGetErrorString(e));
    set_error(buf);
    return FELBM_ERR_CUDA;
}
#define FELBM_CUDA(call)                                   \
    do {                                                   \
        cudaError_t e_ = (call);                           \
        if (e_ != cudaSuccess) return cuda_fail(e_, #call); \
    } while (0)

// Bump allocator over the caller's workspace (256-byte aligned pieces).
struct Carver {
    char* base;
    size_t off = 0;
    explicit Carver(void* b) : base(static_cast<char*>(b)) {}
    template <class T>
    T* take(size_t n) {
        off = (off + 255) & ~size_t(255);
        T* p = base ? reinterpret_cast<T*>(base + off) : nullptr;
        off += n * sizeof(T);
        return p;
    }
};

static size_t pad64(size_t n) { return (n + 63) & ~size_t(63); }

}  // namespace felbm

struct felbm_state {
    felbm::HostMesh hm;
    felbm_params prm;
    felbm::DevMesh dm{};
    felbm::Phys phys{};
    felbm::Bufs buf{};
    cudaStream_t stream = nullptr;
    cudaStream_t cap_stream = nullptr;
    cudaGraphExec_t graph_exec = nullptr;
    cudaGraph_t graph = nullptr;
    int mode = FELBM_SOLVER_MIXED;
    int sweeps = 14;   // per correction (mixed) or in total (FP64)
    int rounds = 3;    // corrections of the mixed solve
    std::vector<double> cheb_a, cheb_c;   // three-term recurrence of the FP64 solve
    double inv_theta = 1.0;               // its first iterate x_1 = m^{-1} b / theta
    std::vector<double> tau;              // Richardson step sizes of the FP32 solves; tau[0] gives x_1
    int64_t step = 0;
    double mass0 = 0.0;
    int device = 0;
    bool timing = false;
    bool timed_step_ran = false;
    cudaEvent_t ev[7] = {};
    bool dev32 = false;   // FELBM_FP32_DEV storage
    bool use_pdl = true;  // programmatic dependent launch between solve sweeps
    int sweep_parts = 2;  // threads per node of the FP32 store sweeps (1, 2, 3, 6)
    int sweep_tiled = -1;      // several steps of a node block per launch (k_block32): 1, never: 0, where faster: -1
    bool check = false;        // felbm_solver_check: residual of every solve before its last step
    double check_tol = 0.0;
    int n_sm = 1;              // multiprocessors of the device
    felbm::GroupTables gt{};
    felbm::AdjBufs adj{};         // adjoint buffers (FP64 states)
    std::vector<double> gmass0;   // per-group mass at felbm_init
    // batch schedule (FP32_DEV): groups of at most cta_max_nodes nodes run one
    // CTA each (k_step_cta32); the rest, a prefix of the node and triangle
    // ranges, run the tiled kernels.  cta_max_nodes = 0: tiled only.
    int32_t cta_max_nodes = 0;
    int32_t n_cta = 0, tiled_N = 0, tiled_T = 0, tiled_blocks = 0;
    int32_t* d_cta_groups = nullptr;   // [G] in the workspace
    cudaStream_t side_stream = nullptr;
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    cudaEvent_t ev_copied = nullptr;   // set_state: the host arrays have been read
    cudaStream_t copy_stream = nullptr;     // set_state's host-to-device copies
    cudaEvent_t ev_in_free[2] = {};         // the conversion that last read buf.in0 / in1 has run
    int in_next = 0;                        // input buffer of the next set_state
};

namespace felbm {

// ELL width used by the FP32 sweeps: the longest row rounded up to one of
// the compiled widths; 0 (CSR sweeps) beyond 16.
static int ell_width(const HostMesh& h) {
    int w = h.max_degree;
    for (int c : {7, 9, 12, 16})
        if (w <= c) return c;
    return 0;
}

// Width of the incidence ELL used by the FP32 RHS gather: the most triangles
// at one node rounded up to a compiled width; 0 (CSR) beyond 12.
static int inc_width(const HostMesh& h) {
    int w = 0;
    for (int32_t i = 0; i < h.N; ++i) w = std::max(w, h.inc_ptr[i + 1] - h.inc_ptr[i]);
    for (int c : {6, 8, 12})
        if (w <= c) return c;
    return 0;
}

// Meshes felbm_sweep_tiled takes: an ELL width with a compiled blocked solve (a
// thread keeps its nodes' rows in registers; 16 entries do not fit) and tiles
// whose first layer is small.  The blocked solve itself needs no more than
// n_layers > 0; the tiles' limit stays so that the calls that were refused are.
static bool tiled_ok(const HostMesh& h, int ell_w) {
    return (ell_w == 7 || ell_w == 9 || ell_w == 12) && h.max_halo <= kHaloMax;
}

// Rows of the blocked solve's tables: per block its own nodes and all layers
// but the last, rounded up to 32.  first (blocks + 1 entries): where each
// block's rows start.
static int64_t block_rows(const HostMesh& h, int32_t* first) {
    const int32_t nb = (int32_t)h.blk_ptr.size() - 1;
    int64_t rows = 0;
    for (int32_t t = 0; t < nb; ++t) {
        if (first) first[t] = (int32_t)rows;
        rows += (h.layer_cnt[(size_t)t * (kBlockSteps + 1) + h.n_layers - 1] + 31) & ~31;
    }
    if (first) first[nb] = (int32_t)rows;
    return rows;
}

// Layout of the workspace; with base == nullptr only the size is computed.
static size_t carve(const HostMesh& h, bool dev32, void* base, DevMesh* dm, Bufs* b,
                    GroupTables* gtab = nullptr, AdjBufs* adj = nullptr) {
    Carver cv(base);
    size_t Np = pad64(h.N), Tp = pad64(h.T);
    size_t nnz = h.row_ptr[h.N], ninc = h.inc_ptr[h.N], nwinc = h.winc_ptr[h.N];
    size_t E = std::max<int32_t>(h.E, 1);
    DevMesh d{};
    d.tri = cv.take<int32_t>(3 * Tp);
    d.area = cv.take<double>(Tp);
    d.grad = cv.take<double>(6 * Tp);
    d.area32 = cv.take<float>(Tp);
    d.grad32 = cv.take<float>(6 * Tp);
    d.nbr = cv.take<int32_t>(3 * Tp);
    d.nbr_slot = cv.take<int32_t>(3 * Tp);
    d.row_ptr = cv.take<int32_t>(h.N + 1);
    d.col = cv.take<int32_t>(nnz);
    d.mval = cv.take<double>(nnz);
    d.lval = cv.take<double>(nnz);
    d.inv_lumped = cv.take<double>(Np);
    d.mval32 = cv.take<float>(nnz);
    const int ellw = ell_width(h);
    d.ell_w = ellw;
    d.ell_col = cv.take<int32_t>((size_t)std::max(ellw, 1) * Np);
    d.ell_val = cv.take<float>((size_t)std::max(ellw, 1) * Np);
    d.n_blocks = (int32_t)h.blk_ptr.size() - 1;
    d.blk_steps = tiled_ok(h, ellw) ? h.n_layers : 0;
    const size_t brows = d.blk_steps > 0 ? (size_t)block_rows(h, nullptr) : 1;
    d.blk_ptr = cv.take<int32_t>(h.blk_ptr.size());
    d.blk_cnt = cv.take<int32_t>(h.layer_cnt.size());
    d.blk_halo_ptr = cv.take<int32_t>(h.halo_ptr.size());
    d.blk_halo = cv.take<int32_t>(std::max<size_t>(h.halo.size(), 1));
    d.blk_row = cv.take<int32_t>(h.blk_ptr.size());
    d.blk_val = cv.take<float>(brows * std::max(ellw, 1));
    d.blk_col = cv.take<uint32_t>(brows * std::max(ellw / 2, 1));
    d.ell_lval = cv.take<double>((size_t)std::max(ellw, 1) * Np);
    const int iw = inc_width(h);
    d.iell_w = iw;
    d.iell_tri = cv.take<int32_t>((size_t)std::max(iw, 1) * Np);
    d.iell_bx32 = cv.take<float>((size_t)std::max(iw, 1) * Np);
    d.iell_by32 = cv.take<float>((size_t)std::max(iw, 1) * Np);
    d.max_blk_tri = dev32 && iw > 0 && h.max_blk_tri <= kForceTris ? h.max_blk_tri : 0;   // 0: k_force32 unused
    d.blk_tri_ptr = cv.take<int32_t>(h.blk_tri_ptr.size());
    d.blk_tri = cv.take<int32_t>(d.max_blk_tri > 0 ? h.blk_tri.size() : 1);
    d.iell_loc = cv.take<uint16_t>(d.max_blk_tri > 0 ? (size_t)iw * Np : 1);
    d.inv_lumped32 = cv.take<float>(Np);
    d.start32 = cv.take<float2>(Np);
    d.lumped = cv.take<double>(Np);
    d.inv_vol = cv.take<double>(Np);
    d.inc_ptr = cv.take<int32_t>(h.N + 1);
    d.inc_tri = cv.take<int32_t>(ninc);
    d.inc_bx = cv.take<double>(ninc);
    d.inc_by = cv.take<double>(ninc);
    d.inc_bx32 = cv.take<float>(ninc);
    d.inc_by32 = cv.take<float>(ninc);
    d.wall_a = cv.take<int32_t>(E);
    d.wall_b = cv.take<int32_t>(E);
    d.wall_id = cv.take<int32_t>(E);
    d.wall_phi = cv.take<double>(E);
    d.wall_len = cv.take<double>(E);
    d.wall_nx = cv.take<double>(E);
    d.wall_ny = cv.take<double>(E);
    d.winc_ptr = cv.take<int32_t>(h.N + 1);
    d.winc_edge = cv.take<int32_t>(std::max<size_t>(nwinc, 1));
    d.x = cv.take<double>(Np);
    d.y = cv.take<double>(Np);
    d.perm = cv.take<int32_t>(h.N);
    d.iperm = cv.take<int32_t>(h.N);
    Bufs bb{};
    bb.C = cv.take<double>(Np);
    if (!dev32) {
        bb.psi = cv.take<double>(18 * Np);
        bb.p = cv.take<double>(Np);
        bb.ux = cv.take<double>(Np);
        bb.uy = cv.take<double>(Np);
        bb.mu = cv.take<double>(Np);
        bb.gmu = cv.take<double>(2 * Tp);
        bb.lmu = bb.gmu;
        bb.R = cv.take<double>(18 * (size_t)h.T);
    } else {
        bb.dpsi = cv.take<float>(18 * Np);
        bb.p32 = cv.take<float>(Np);
        bb.ux32 = cv.take<float>(Np);
        bb.uy32 = cv.take<float>(Np);
        bb.mu32 = cv.take<float>(Np);
        bb.gmu32 = cv.take<float>(2 * Tp);
        bb.lmu32 = bb.gmu32;
        bb.R32 = cv.take<float>(18 * ((size_t)h.T + 1));   // row T: zeros (incidence padding)
    }
    bb.rhs = cv.take<double>(18 * Np);
    bb.x0 = cv.take<double>(18 * Np);
    bb.x1 = cv.take<double>(18 * Np);
    bb.x64 = bb.x0;
    bb.rho64 = bb.x1;
    bb.r32 = cv.take<float>(18 * Np);
    bb.e0 = cv.take<float>(18 * Np);
    bb.e1 = cv.take<float>(18 * Np);
    bb.stage = cv.take<double>(18 * Np);
    bb.in0 = cv.take<double>(18 * Np);
    bb.in1 = cv.take<double>(18 * Np);
    bb.diag_part = cv.take<double>((size_t)kDiagBlocks * kDiagSlots);
    bb.diag_out = cv.take<double>(kDiagSlots);
    bb.Cdiag = cv.take<double>(Np);
    bb.diag_done = cv.take<unsigned>(1);
    GroupTables g{};
    const size_t G = std::max<int32_t>(h.G, 1);
    g.node_begin = cv.take<int32_t>(G);
    g.node_end = cv.take<int32_t>(G);
    g.tri_begin = cv.take<int32_t>(G);
    g.tri_end = cv.take<int32_t>(G);
    g.wall_ptr = cv.take<int32_t>(G + 1);
    g.wall_edge = cv.take<int32_t>(E);
    g.reqs = cv.take<DiagReq>(G);
    g.out = cv.take<double>(G * kDiagSlots);
    g.cta_groups = cv.take<int32_t>(G);
    if (gtab) *gtab = g;
    AdjBufs ad{};
    if (!dev32) {
        ad.lam = cv.take<double>(18 * Np);
        ad.lamhat = cv.take<double>(18 * Np);
        ad.lamR = cv.take<double>(18 * (size_t)h.T);
        ad.lamE = cv.take<double>(9 * (size_t)h.T);
        ad.lamG = cv.take<double>(2 * Tp);
        ad.lamMu = cv.take<double>(Np);
        ad.lamC = cv.take<double>(Np);
        ad.lamP = cv.take<double>(Np);
        ad.lamUx = cv.take<double>(Np);
        ad.lamUy = cv.take<double>(Np);
        ad.dphi = cv.take<double>(E);
        ad.kval = cv.take<double>(nnz);
    }
    if (adj) *adj = ad;
    if (dm) {
        d.N = h.N;
        d.T = h.T;
        d.E = h.E;
        d.Np = (int32_t)Np;
        d.Tp = (int32_t)Tp;
        d.period_y = h.period[1];
        *dm = d;
    }
    if (b) *b = bb;
    return cv.off + 256;
}

static int check_params(const felbm_params* p) {
    if (!p || !(p->dt > 0.0) || !(p->tau_l > 0.0) || !(p->tau_v > 0.0) || !(p->rho_l > 0.0) ||
        !(p->rho_v > 0.0) || !(p->kappa >= 0.0) || !(p->beta >= 0.0) || !(p->mobility >= 0.0) ||
        p->lap_mode < 0 || p->lap_mode > 1 || p->solver_iters < 0 || p->solver_iters == 1 ||
        p->solver_iters > 1000 || p->solver_rounds < 0 || p->solver_rounds > 20 ||
        p->solver_mode < 0 || p->solver_mode > 1 ||
        p->n_wall_ids < 0 || p->n_wall_ids > FELBM_MAX_WALL_IDS ||
        (p->lapmu_mode != FELBM_LAPMU_FACE && p->lapmu_mode != FELBM_LAPMU_NODAL)) {
        set_error("felbm: invalid params (dt, tau, rho > 0; kappa, beta, mobility >= 0; lap_mode 0/1; "
                  "solver_mode 0/1; solver_iters 0 or 2..1000; solver_rounds 0..20; lapmu_mode 0/1)");
        return FELBM_ERR_INVALID_ARG;
    }
    if (p->precision != FELBM_FP64 && p->precision != FELBM_FP32_DEV) {
        set_error("felbm: unknown precision");
        return FELBM_ERR_UNSUPPORTED;
    }
    if (p->precision == FELBM_FP32_DEV && (p->solver_mode != FELBM_SOLVER_MIXED || p->solver_rounds > 1)) {
        set_error("felbm: FELBM_FP32_DEV solves in FP32 (solver_mode MIXED, solver_rounds 0 or 1)");
        return FELBM_ERR_UNSUPPORTED;
    }
    return FELBM_OK;
}

template <class T>
static cudaError_t up(const T* dst, const std::vector<T>& src, cudaStream_t s) {
    if (src.empty()) return cudaSuccess;
    return cudaMemcpyAsync(const_cast<T*>(dst), src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice, s);
}

static unsigned grid_for(int n, int block) { return (unsigned)((n + block - 1) / block); }

// Threads per block of the FP64 kernels: `most`, or a warp where that spreads
// n items over the multiprocessors more evenly (the FP64 pipe of each is what
// the kernels wait for): a step on 2,112 nodes took 101 us against 125, on
// 18,432 nodes 162 against 186 (with the other FP64 changes); on 520,704 nodes
// the two are the same.
static int fp64_block(const felbm_state* st, int n, int most) { return n < kWarpBlocksBelow * st->n_sm ? 32 : most; }

// Launch with or without programmatic dependent launch (PDL).
template <typename... KArgs, typename... Args>
static void launch_k(bool pdl, void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                     Args&&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}

// One blocked launch: K steps from cur (or from b) to nxt.  All planes of a
// block in one thread block; one plane or pair of right-hand sides each where
// that would leave multiprocessors idle.
template <bool kFromRhs>
static void launch_block(const felbm_state* st, const DevMesh& m, const Bufs& b, cudaStream_t s, const float* cur,
                         float* nxt, const BlockTau& bt, int K, float tau0, int n4, bool update, bool pdl) {
    const bool full = m.n_blocks >= kSplitPlanesBelow * st->n_sm, pairs = split_pairs(m.n_blocks, st->n_sm);
    const dim3 grid((unsigned)m.n_blocks, full ? 1 : (pairs ? 2 * n4 + 1 : n4 + 1));
    const auto go = [&](auto kern, auto pair_kern, auto update_kern) {
        // dependent launch places the blocks of a small grid on whatever
        // multiprocessors the previous kernel has left, two on one while
        // others idle: 82 against 74 us a step on 2,112 nodes (FP64)
        launch_k(pdl && full && st->use_pdl, update ? update_kern : (pairs ? pair_kern : kern), grid, dim3(kBlockThreads),
                 update ? sizeof(BlockUpdateSmem) : sizeof(BlockSmem), s, m, st->phys, b, cur, nxt, bt, K, tau0, n4);
    };
    switch (m.ell_w) {
        case 7: go(k_block32<7, kFromRhs, false>, k_block32<7, kFromRhs, true>, k_block32<7, false, false, true>); break;
        case 9: go(k_block32<9, kFromRhs, false>, k_block32<9, kFromRhs, true>, k_block32<9, false, false, true>); break;
        default: go(k_block32<12, kFromRhs, false>, k_block32<12, kFromRhs, true>, k_block32<12, false, false, true>);
    }
}

// Shared memory beyond the default 48 KB for the blocked kernels.
template <int kW>
static cudaError_t allow_block_smem() {
    cudaError_t e = cudaSuccess;
    const auto set = [&](auto kern) {
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(BlockUpdateSmem));
    };
    set(k_block32<kW, false, false>);
    set(k_block32<kW, true, false>);
    set(k_block32<kW, false, true>);
    set(k_block32<kW, true, true>);
    set(k_block32<kW, false, false, true>);
    return e;
}

// One FP32 Chebyshev sweep: the ELL kernel of the mesh's width, else CSR.
// pdl: the previous launch on the stream is a sweep (a kernel that waits).
// parts: threads per node for the store sweeps (1, 2, 3 or 6; autotuned).
template <int kFinal, int kW>
static void launch_sweep_w(felbm_state* st, const DevMesh& m, const Bufs& b, cudaStream_t s, const float* cur,
                           float* nxt, float tau, int have_x64, bool pdl) {
    const dim3 block(128);
    const int parts = kFinal == kUpdateDev ? 1 : st->sweep_parts;
    const dim3 grid(grid_for(m.N, 128) * parts);
    switch (parts) {
        case 1:
            launch_k(pdl, k_sweep32<kFinal, kW, 1>, grid, block, 0, s, m, st->phys, b, cur, nxt, tau, have_x64, 0.0f);
            break;
        case 3:
            if constexpr (kFinal != kUpdateDev)
                launch_k(pdl, k_sweep32<kFinal, kW, 3>, grid, block, 0, s, m, st->phys, b, cur, nxt, tau, have_x64, 0.0f);
            break;
        case 6:
            if constexpr (kFinal != kUpdateDev)
                launch_k(pdl, k_sweep32<kFinal, kW, 6>, grid, block, 0, s, m, st->phys, b, cur, nxt, tau, have_x64, 0.0f);
            break;
        default:
            if constexpr (kFinal != kUpdateDev)
                launch_k(pdl, k_sweep32<kFinal, kW, 2>, grid, block, 0, s, m, st->phys, b, cur, nxt, tau, have_x64, 0.0f);
    }
}

template <int kFinal>
static void launch_sweep(felbm_state* st, const DevMesh& m, const Bufs& b, cudaStream_t s, const float* cur,
                         float* nxt, float tau, int have_x64, bool pdl) {
    pdl = pdl && st->use_pdl;
    switch (m.ell_w) {
        case 7:
            launch_sweep_w<kFinal, 7>(st, m, b, s, cur, nxt, tau, have_x64, pdl);
            break;
        case 9:
            launch_sweep_w<kFinal, 9>(st, m, b, s, cur, nxt, tau, have_x64, pdl);
            break;
        case 12:
            launch_sweep_w<kFinal, 12>(st, m, b, s, cur, nxt, tau, have_x64, pdl);
            break;
        case 16:
            launch_sweep_w<kFinal, 16>(st, m, b, s, cur, nxt, tau, have_x64, pdl);
            break;
        default:
            k_cheb32<kFinal><<<grid_for(m.N, 128), 128, 0, s>>>(m, st->phys, b, cur, nxt, tau, have_x64);
    }
}

// ELL widths with compiled gathered solve steps
static bool gathered_width(int ell_w) { return ell_w == 7 || ell_w == 9 || ell_w == 12 || ell_w == 16; }

// The first step of the FP32 time-step solve with x_0 formed from b (gathered
// ELL widths and the untiled steps only).
template <int kW>
static void launch_first_w(felbm_state* st, const DevMesh& m, const Bufs& b, cudaStream_t s, float* nxt,
                           float tau, float tau0, bool pdl) {
    const dim3 block(128);
    const int parts = st->sweep_parts;
    const dim3 grid(grid_for(m.N, 128) * parts);
    switch (parts) {
        case 1: launch_k(pdl, k_sweep32<kStore, kW, 1, true>, grid, block, 0, s, m, st->phys, b, nullptr, nxt, tau, 0, tau0); break;
        case 3: launch_k(pdl, k_sweep32<kStore, kW, 3, true>, grid, block, 0, s, m, st->phys, b, nullptr, nxt, tau, 0, tau0); break;
        case 6: launch_k(pdl, k_sweep32<kStore, kW, 6, true>, grid, block, 0, s, m, st->phys, b, nullptr, nxt, tau, 0, tau0); break;
        default: launch_k(pdl, k_sweep32<kStore, kW, 2, true>, grid, block, 0, s, m, st->phys, b, nullptr, nxt, tau, 0, tau0);
    }
}

// Only called when gathered_width(m.ell_w) (first_from_rhs checks it).
static void launch_first(felbm_state* st, const DevMesh& m, const Bufs& b, cudaStream_t s, float* nxt, float tau,
                         float tau0, bool pdl) {
    pdl = pdl && st->use_pdl;
    switch (m.ell_w) {
        case 7: launch_first_w<7>(st, m, b, s, nxt, tau, tau0, pdl); break;
        case 9: launch_first_w<9>(st, m, b, s, nxt, tau, tau0, pdl); break;
        case 12: launch_first_w<12>(st, m, b, s, nxt, tau, tau0, pdl); break;
        default: launch_first_w<16>(st, m, b, s, nxt, tau, tau0, pdl);
    }
}

// Thread blocks, two to a multiprocessor, in waves that are at least four fifths
// full altogether.
static bool full_waves(int n_blocks, int n_sm) {
    const int slots = 2 * n_sm, waves = (n_blocks + slots - 1) / slots;
    return 5LL * n_blocks >= 4LL * waves * slots;
}

// Where the blocked solve of all rows is the faster form (GB300, solve phase of
// an FP32 step of 10 steps, blocked against one launch per step; rows of 7
// unless stated).
//  * Up to kL2Nodes nodes the three vectors of a step (216 bytes a node) stay in
//    L2 and a step per launch costs 48 ps a node, beyond it 56 to 70.  There the
//    blocked form wins: 168 against 205 us on 405,900 nodes, 670 against 1,004
//    on 2,082,816, and with two steps a launch 889 against 1,018.
//  * With all planes in a thread block and the vectors in L2 it wins in one full
//    wave (80,400 nodes in 256 blocks: 44 against 45; 128,000: 42 against 55) and
//    wins or ties where blocks are nearly full too (rows of 9, step: 576 blocks of
//    512, 230 against 254; 261,726 nodes, 512 of 511: 101 against 103).  Smaller
//    blocks compute too many rows of their layers and a partial wave leaves
//    multiprocessors idle: 131,584 nodes in 512 blocks of 257: 74 against 61; a
//    batch of 145,852 nodes in 392 blocks: 77 against 63; rows of 9, 320 blocks
//    of 512, step: 176 against 152.
//  * With a plane per thread block it wins or ties: 19 against 31 on 20,200
//    nodes, 35 against 34 on 65,341.  Rows of more than 9 entries leave one
//    thread block to a multiprocessor: 33 against 35 on 26,180 nodes (64
//    blocks), 52 against 37 on 43,380 (128 blocks), 175 against 150 on 235,620.
//  * It needs steps to share a load: one step a solve takes 60 against 30 us on
//    525,312 nodes, nine launches of one step (one layer) 48 against 35 on 36,120.
constexpr int kL2Nodes = 340000;
static bool blocked_is_faster(const felbm_state* st, const DevMesh& m) {
    const bool in_l2 = m.N <= kL2Nodes;
    if (st->sweeps < 3 || m.blk_steps < (in_l2 ? 3 : 2)) return false;
    if (!in_l2) return true;
    if (m.n_blocks < kSplitPlanesBelow * st->n_sm) return m.ell_w <= 9 || kPlanes * m.n_blocks <= 3 * st->n_sm;
    return m.ell_w <= 9 && full_waves(m.n_blocks, st->n_sm) && (m.n_blocks <= 2 * st->n_sm || m.N >= 480 * m.n_blocks);
}

// Whether the solve of all rows on m runs blocked.
static bool blocked(const felbm_state* st, const DevMesh& m) {
    if (m.blk_steps == 0 || st->mode == FELBM_SOLVER_FP64) return false;
    return st->sweep_tiled < 0 ? blocked_is_faster(st, m) : st->sweep_tiled != 0;
}

static bool first_from_rhs(const felbm_state* st, const DevMesh& m);

// Whether the last launch of an FP32-deviation state's solve, whose first step
// is `first`, updates fields and deviations: all planes in one thread block, and
// not the launch that forms x_0.
static bool fused_update(const felbm_state* st, const DevMesh& m, int first) {
    return st->dev32 && m.n_blocks >= kSplitPlanesBelow * st->n_sm &&
           (first > 1 || st->sweeps - 1 > m.blk_steps || !first_from_rhs(st, m));
}

// The steps [k, end) of one correction in as few blocked launches as the
// layers allow, of about equal length.  At most 2, 3, 4, 5 and 8 steps a launch
// took, us a step: 2,112 nodes (blocks of 264) FP32 30.9, 26.8, 26.9, 24.9, 24.8,
// FP64 103, 90, 84, 78, 74; 525,312 nodes (257) FP32 458, 413, 412, 408, 407, FP64
// 2,628, 2,486, 2,440, 2,431, 2,513; 2,099,200 nodes (342, four layers) FP32 1,503,
// 1,378 from 3 on; 352,800 nodes, rows of 9 (345) FP32 330, 318, 319, 328, 327: as
// many as fit is within 4 % of the best.  update: the last launch also updates
// fields and deviations (fused_update).  Returns the buffer with the last iterate.
static float* enqueue_blocked(felbm_state* st, const DevMesh& m, const Bufs& b, cudaStream_t s, float* cur, float* prv,
                              int k, int end, bool from_rhs, int n4, bool update, bool pdl) {
    int left = (end - k + m.blk_steps - 1) / m.blk_steps;
    for (; left > 0; --left) {
        const int K = (end - k + left - 1) / left;
        BlockTau bt{};
        for (int j = 0; j < K; ++j) bt.tau[j] = (float)st->tau[k + j];
        const float tau0 = (float)st->tau[0];
        if (from_rhs)
            launch_block<true>(st, m, b, s, nullptr, prv, bt, K, tau0, n4, false, pdl);
        else
            launch_block<false>(st, m, b, s, cur, prv, bt, K, tau0, n4, update && left == 1, pdl);
        from_rhs = false;
        pdl = true;
        k += K;
        std::swap(cur, prv);
    }
    return cur;
}

// The checked solve's residual of the iterate cur (felbm_solver_check).
static void enqueue_resid(felbm_state* st, const DevMesh& m, const Bufs& b, cudaStream_t s, const float* cur) {
    if (st->dev32)
        k_solve_resid<false><<<kDiagBlocks, kBlock, 0, s>>>(m, b, cur, b.diag_part);
    else
        k_solve_resid<true><<<kDiagBlocks, kBlock, 0, s>>>(m, b, cur, b.diag_part);
    k_solve_resid_final<<<1, 1, 0, s>>>(b.diag_part, kDiagBlocks, b.diag_out + kSolveResSlot);
}

// Whether the FP32 time step forms x_0 inside its first solve step (then the
// RHS kernel stores b only): one correction round, gathered steps, at least
// two steps after the first, no residual check, an ELL width with kernels.
static bool first_from_rhs(const felbm_state* st, const DevMesh& m) {
    return st->dev32 && st->rounds == 1 && st->sweeps > 2 && !st->check && (blocked(st, m) || gathered_width(m.ell_w));
}

static void launch_mu(const DevMesh& m, const Phys& c, const Bufs& b, unsigned grid, int block, cudaStream_t s) {
    switch (m.ell_w) {
        case 7: k_mu<7><<<grid, block, 0, s>>>(m, c, b); break;
        case 9: k_mu<9><<<grid, block, 0, s>>>(m, c, b); break;
        case 12: k_mu<12><<<grid, block, 0, s>>>(m, c, b); break;
        case 16: k_mu<16><<<grid, block, 0, s>>>(m, c, b); break;
        default: k_mu<0><<<grid, block, 0, s>>>(m, c, b);
    }
}

// Enqueue the mass solve for the right-hand side in b.rhs (first iterate
// already written, unless from_rhs).  into_psi: add the increment to psi (time step); else
// leave the solution in x1/x0 (FP64 mode, returned) or x64 (mixed mode).
// b: the buffers the solve reads and writes (the state's own, or another set of
// scratch buffers with the same layout).  tiled: blocked.  n4: planes in use (k_block32; blocked
// solves only).  last: where given (blocked, not into_psi), the last correction
// is not added to x64 but returned through it.
static const double* enqueue_solve(felbm_state* st, const DevMesh& m, const Bufs& b, cudaStream_t s,
                                   bool into_psi, bool tiled, bool after_release = false, bool from_rhs = false,
                                   int n4 = 4, const float** last = nullptr) {
    const int nb = fp64_block(st, m.N, 128);
    const unsigned grid = grid_for(m.N, nb);
    if (st->mode == FELBM_SOLVER_FP64) {
        const double* result = b.x1;
        for (int k = 1; k < st->sweeps; ++k) {
            const double* cur = (k & 1) ? b.x1 : b.x0;
            double* prev = (k & 1) ? b.x0 : b.x1;
            k_cheb<<<grid, nb, 0, s>>>(m, b, cur, prev, st->cheb_a[k], st->cheb_c[k], k == 1,
                                        into_psi && k == st->sweeps - 1);
            result = prev;
        }
        return result;
    }
    float* A = b.e1;
    float* B = b.e0;
    const int have_x64 = st->rounds > 1;
    for (int r = 0; r < st->rounds; ++r) {
        float* cur = A;
        float* prv = B;
        const bool last_round = r == st->rounds - 1;
        if (tiled) {
            bool pdl = r == 0 && after_release;
            int k = 1;
            if (last_round && st->check) {
                float* const x = enqueue_blocked(st, m, b, s, cur, prv, 1, st->sweeps - 1, false, n4, false, pdl);
                prv = x == cur ? prv : cur;
                cur = x;
                enqueue_resid(st, m, b, s, cur);
                k = st->sweeps - 1;
                pdl = false;
            }
            const bool update = last_round && into_psi && fused_update(st, m, k);
            float* const x = enqueue_blocked(st, m, b, s, cur, prv, k, st->sweeps, from_rhs && r == 0, n4, update, pdl);
            prv = x == cur ? prv : cur;
            cur = x;
            if (last_round && into_psi && st->dev32 && !update)
                launch_k(st->use_pdl, k_update32, dim3(grid_for(m.N, 128)), dim3(128), 0, s, m, st->phys, b,
                         (const float*)cur);
            else if (last_round && into_psi && st->dev32)
                ;   // updated in the last launch
            else if (last_round && last)
                *last = cur;
            else if (last_round)
                launch_k(st->use_pdl, into_psi ? k_add64<true> : k_add64<false>, dim3(grid), dim3(nb), 0, s, m, b,
                         (const float*)cur, have_x64);
        }
        for (int k = 1; k < st->sweeps && !tiled; ++k) {
            const float tau = (float)st->tau[k];
            const bool last = last_round && k == st->sweeps - 1;
            // the previous launch is a sweep of this round, or a kernel that released its dependents
            bool pdl = k > 1 || (k == 1 && r == 0 && after_release);
            if (last && st->check) {
                enqueue_resid(st, m, b, s, cur);
                pdl = false;
            }
            if (from_rhs && r == 0 && k == 1)
                launch_first(st, m, b, s, prv, tau, (float)st->tau[0], pdl);
            else if (!last)
                launch_sweep<kStore>(st, m, b, s, cur, prv, tau, have_x64, pdl);
            else if (!into_psi)
                launch_sweep<kAddX64>(st, m, b, s, cur, prv, tau, have_x64, pdl);
            else if (st->dev32)
                launch_sweep<kUpdateDev>(st, m, b, s, cur, prv, tau, have_x64, pdl);
            else
                launch_sweep<kAddPsi>(st, m, b, s, cur, prv, tau, have_x64, pdl);
            std::swap(cur, prv);
        }
        if (!last_round) {
            k_refine<<<grid * (n4 + 1), nb, 0, s>>>(m, b, cur, prv, r == 0, st->tau[0], n4);
            A = prv;
            B = cur;
        }
    }
    return b.x64;
}

// X = M11^{-1} B for rows [0, k) (device, caller order), with scratch b.  A
// blocked solve takes only the planes that hold those rows (5 of 18 rows on
// 80,000 nodes take 168 us instead of 378), so it is the default for them.
static void enqueue_mass_solve(felbm_state* st, const Bufs& b, const double* B, double* X, int k, cudaStream_t s) {
    const DevMesh& m = st->dm;
    const unsigned grid = grid_for(m.N, kBlock);
    const int planes = st->check ? 4 : k <= 1 ? 0 : k <= 5 ? 1 : k <= 10 ? 2 : k <= 14 ? 3 : 4;   // the checked residual covers all rows
    const bool some = planes < 4 && st->sweep_tiled < 0 && m.blk_steps > 0 && st->mode != FELBM_SOLVER_FP64;
    const bool tiled = some || blocked(st, m), part = tiled && !st->check;
    const int n4 = part ? planes : 4;
    if (st->mode == FELBM_SOLVER_FP64)
        k_solve_in<false><<<grid, kBlock, 0, s>>>(m, b, B, k, n4, st->inv_theta);
    else
        k_solve_in<true><<<grid, kBlock, 0, s>>>(m, b, B, k, n4, st->tau[0]);
    const float* last = nullptr;
    const double* x = enqueue_solve(st, m, b, s, false, tiled, false, false, n4, part ? &last : nullptr);
    k_solve_out<<<grid, kBlock, 0, s>>>(m, x, last, X, k, !last || st->rounds > 1);
}

// The part of the mesh that the launches of a step cover: the members that have
// no CTA of their own, a prefix of nodes, triangles and blocks (set_schedule).
static DevMesh launched_part(const felbm_state* st) {
    DevMesh m = st->dm;
    m.N = st->tiled_N;
    m.T = st->tiled_T;
    m.n_blocks = st->tiled_blocks;
    return m;
}

static int solve_launches(const felbm_state* st, const DevMesh& m) {
    if (m.N == 0) return 0;
    if (st->mode == FELBM_SOLVER_FP64) return st->sweeps - 1;
    const int refines = st->rounds - 1;
    if (!blocked(st, m)) return st->rounds * (st->sweeps - 1) + refines;
    const int most = m.blk_steps;
    const auto groups = [&](int steps) { return (steps + most - 1) / most; };
    const int last = st->check ? groups(st->sweeps - 2) + 1 : groups(st->sweeps - 1);
    const bool update = fused_update(st, m, st->check ? st->sweeps - 1 : 1);
    return refines * (groups(st->sweeps - 1) + 1) + last + (update ? 0 : 1);
}

// FP32 states: residuals and their gather in one kernel (k_force32) or in two.
// One kernel needs the device full, with two thread blocks of 384 threads on a
// multiprocessor, and few walls: the bounce-back of a wall node is a chain of
// loads that two thread blocks hide worse than the separate gather's eight.
// Step of one solve step, us, one kernel against two (GB300):
//   no walls (rows of 9)  128 blocks 26.8 / 24.7, 160 35.1 / 33.2, 176 34.9 / 35.0, 256 49.5 / 57.5,
//                         320 72.4 / 69.4, 448 92.4 / 90.8, 512 55.1 / 59.5, 688 140 / 135
//   walls                 256 blocks, 8,000 x 15 cells (12 % of the nodes) 58.4 / 59.3; batches of 176 to
//                         1,376 blocks (3 to 8 %) 41.4 / 35.7 to 193 / 181; 450,000 nodes with 0.7, 2 and
//                         4 %: 165 / 163, 174 / 166, 189 / 173
//   2,082,816 nodes (0.2 %) 627 / 652
//   405,900 nodes (0.4 %) in blocks of 396, which fill two of three rounds of threads: 156 / 148
// Hence: any walls in one full wave, below 1 % of the nodes in more full waves or
// in one wave of at least 1.15 blocks to a multiprocessor.
static bool fused_forces(const felbm_state* st, const DevMesh& m) {
    if (!st->dev32 || m.max_blk_tri == 0) return false;
    const int nb = m.n_blocks;
    const bool one = nb <= 2 * st->n_sm, full = full_waves(nb, st->n_sm);
    if (100LL * st->hm.E > st->hm.N) return one && full;
    return full || (one && 20 * nb >= 23 * st->n_sm);
}

static int step_launches(const felbm_state* st, const DevMesh& m) {
    const int ctas = st->n_cta > 0 ? 1 : 0;
    if (m.N == 0) return ctas;
    return ctas + (st->dev32 ? (fused_forces(st, m) ? 3 : 4) : 5) + solve_launches(st, m);
}

int set_schedule(felbm_state* st, int32_t max_nodes);

// Enqueue the kernels of one time step on stream s (optionally with the
// phase events, recorded as external event nodes of the captured graph).
static void enqueue_step(felbm_state* st, cudaStream_t s) {
    const DevMesh& m = st->dm;
    const Bufs& b = st->buf;
    auto mark = [&](int k) {
        if (st->timing) cudaEventRecordWithFlags(st->ev[k], s, cudaEventRecordExternal);
    };
    mark(0);
    if (st->dev32) {
        // small batch members: one CTA each, on a side branch of the graph
        if (st->n_cta > 0) {
            ChebCoef cf{};
            for (int k = 1; k < st->sweeps && k < kMaxSweeps; ++k) cf.tau[k] = (float)st->tau[k];
            cudaEventRecord(st->ev_fork, s);
            cudaStreamWaitEvent(st->side_stream, st->ev_fork, 0);
            k_step_cta32<<<st->n_cta, kCtaThreads, 0, st->side_stream>>>(m, st->phys, b, st->gt, st->gt.cta_groups,
                                                                         cf, st->sweeps, (float)st->tau[0]);
            cudaEventRecord(st->ev_join, st->side_stream);
        }
        // the rest (a prefix of nodes and triangles): tiled kernels
        const DevMesh mt = launched_part(st);
        // collision is folded into the element, RHS and update kernels
        mark(1);
        if (mt.N > 0) {
            // programmatic dependent launch along the chain when no phase
            // events sit between the kernels
            const bool chain = st->use_pdl && !st->timing;
            switch (mt.ell_w) {
                case 7: k_mu32<7><<<grid_for(mt.N, kBlock), kBlock, 0, s>>>(mt, st->phys, b); break;
                case 9: k_mu32<9><<<grid_for(mt.N, kBlock), kBlock, 0, s>>>(mt, st->phys, b); break;
                case 12: k_mu32<12><<<grid_for(mt.N, kBlock), kBlock, 0, s>>>(mt, st->phys, b); break;
                case 16: k_mu32<16><<<grid_for(mt.N, kBlock), kBlock, 0, s>>>(mt, st->phys, b); break;
                default: k_mu32<0><<<grid_for(mt.N, kBlock), kBlock, 0, s>>>(mt, st->phys, b);
            }
            mark(2);
            if (st->phys.lapmu_nodal)
                launch_k(chain, k_lmu32, dim3(grid_for(mt.N, kBlock)), dim3(kBlock), 0, s, mt, st->phys, b);
            else
                launch_k(chain, k_gradmu32, dim3(grid_for(mt.T, kBlock)), dim3(kBlock), 0, s, mt, b);
            mark(3);
            const bool from_rhs = first_from_rhs(st, mt);
            const float tau0 = (float)st->tau[0];
            // residuals and their gather in one kernel where the blocks fill the device
            const bool fused = fused_forces(st, mt);
            if (fused) {
                const size_t smem = force_smem_bytes(mt.max_blk_tri);
                const auto go = [&](auto kern) {
                    launch_k(chain, kern, dim3(mt.n_blocks), dim3(kForceThreads), smem, s, mt, st->phys, b, tau0,
                             from_rhs ? 0 : 1);
                };
                mt.iell_w == 6 ? go(k_force32<6>) : mt.iell_w == 8 ? go(k_force32<8>) : go(k_force32<12>);
            } else {
                launch_k(chain, k_element32, dim3(grid_for(mt.T, 128)), dim3(128), 0, s, mt, st->phys, b);
            }
            mark(4);
            const dim3 gn(grid_for(mt.N, 128)), bn(128);
            if (!fused) switch (mt.iell_w * 2 + (from_rhs ? 1 : 0)) {
                case 12: launch_k(chain, k_rhs32<6, true>, gn, bn, 0, s, mt, st->phys, b, tau0); break;
                case 13: launch_k(chain, k_rhs32<6, false>, gn, bn, 0, s, mt, st->phys, b, tau0); break;
                case 16: launch_k(chain, k_rhs32<8, true>, gn, bn, 0, s, mt, st->phys, b, tau0); break;
                case 17: launch_k(chain, k_rhs32<8, false>, gn, bn, 0, s, mt, st->phys, b, tau0); break;
                case 24: launch_k(chain, k_rhs32<12, true>, gn, bn, 0, s, mt, st->phys, b, tau0); break;
                case 25: launch_k(chain, k_rhs32<12, false>, gn, bn, 0, s, mt, st->phys, b, tau0); break;
                default:
                    if (from_rhs)
                        launch_k(chain, k_rhs32<0, false>, gn, bn, 0, s, mt, st->phys, b, tau0);
                    else
                        launch_k(chain, k_rhs32<0, true>, gn, bn, 0, s, mt, st->phys, b, tau0);
            }
            mark(5);
            enqueue_solve(st, mt, st->buf, s, true, blocked(st, mt), chain, from_rhs);
        } else {
            mark(2);
            mark(3);
            mark(4);
            mark(5);
        }
        if (st->n_cta > 0) cudaStreamWaitEvent(s, st->ev_join, 0);
        mark(6);
        return;
    }
    const int nb = fp64_block(st, m.N, 128), tb = fp64_block(st, m.T, 128);
    const unsigned ng = grid_for(m.N, nb), tg = grid_for(m.T, tb);
    k_collide<<<ng, nb, 0, s>>>(m, st->phys, b, 1);
    mark(1);
    launch_mu(m, st->phys, b, ng, nb, s);
    mark(2);
    if (st->phys.lapmu_nodal)
        k_lmu<<<ng, nb, 0, s>>>(m, st->phys, b);
    else
        k_gradmu<<<tg, tb, 0, s>>>(m, b);
    mark(3);
    k_element<<<tg, tb, 0, s>>>(m, st->phys, b);
    mark(4);
    // a small mesh takes a thread per node and set
    const auto rhs = [&](auto kern, int sets, double scale) { kern<<<sets * ng, nb, 0, s>>>(m, st->phys, b, scale); };
    if (st->mode == FELBM_SOLVER_FP64)
        nb == 32 ? rhs(k_rhs<false, 2>, 2, st->inv_theta) : rhs(k_rhs<false, 1>, 1, st->inv_theta);
    else
        nb == 32 ? rhs(k_rhs<true, 2>, 2, st->tau[0]) : rhs(k_rhs<true, 1>, 1, st->tau[0]);
    mark(5);
    enqueue_solve(st, m, st->buf, s, true, blocked(st, m));
    mark(6);
}

}  // namespace felbm

using namespace felbm;

extern "C" {

int felbm_workspace_bytes(const felbm_mesh* mesh, const felbm_params* params, size_t* bytes) {
    if (!mesh || !bytes) {
        set_error("felbm_workspace_bytes: invalid argument");
        return FELBM_ERR_INVALID_ARG;
    }
    int rc = check_params(params);
    if (rc) return rc;
    *bytes = carve(mesh->h, params->precision == FELBM_FP32_DEV, nullptr, nullptr, nullptr);
    return FELBM_OK;
}

// The tables and the first state of a new felbm_state; what it returns or throws
// leaves st to the caller.  No allocation stands between the first upload and
// the wait for the stream.
static int set_up(felbm_state* st, const HostMesh& h, const felbm_params* params, const double* C0, const double* p0,
                  const double* u0, void* d_workspace, void* stream) {
    const bool dev32 = params->precision == FELBM_FP32_DEV;
    st->hm = h;
    st->prm = *params;
    st->stream = static_cast<cudaStream_t>(stream);
    st->dev32 = dev32;
    carve(h, dev32, d_workspace, &st->dm, &st->buf, &st->gt, &st->adj);
    Phys& ph = st->phys;
    ph.dt = params->dt;
    ph.tau_l = params->tau_l;
    ph.tau_v = params->tau_v;
    ph.rho_l = params->rho_l;
    ph.rho_v = params->rho_v;
    ph.kappa = params->kappa;
    ph.beta = params->beta;
    ph.mobility = params->mobility;
    ph.lapmu_nodal = params->lapmu_mode == FELBM_LAPMU_NODAL;
    // lval = -2 K_ij / (s |patch_i|); the lumped P1 Laplacian is -K_ij / (|patch_i| / 3)
    ph.lapmu_fac = (params->lap_mode == FELBM_LAP_PAPER ? 1.0 : 2.0 / 3.0) * 1.5;
    ph.inv_tau_l = 1.0 / params->tau_l;
    ph.inv_tau_v = 1.0 / params->tau_v;
    ph.dt_f = (float)params->dt;
    ph.dt3_f = (float)(params->dt / 3.0);
    ph.dt2h_f = (float)(0.5 * params->dt * params->dt);
    ph.inv_tau_l_f = (float)(1.0 / params->tau_l);
    ph.inv_tau_v_f = (float)(1.0 / params->tau_v);
    ph.rho_v_f = (float)params->rho_v;
    ph.drho_f = (float)(params->rho_l - params->rho_v);
    ph.mobility_f = (float)params->mobility;

    // Chebyshev coefficients for the spectrum [1/4, 1] of m^{-1} M11
    st->mode = params->solver_mode;
    // FP32-deviation states take 10 steps per solve (bound 2*3^-10 on the
    // increment): against the FP64 path that leaves contact angles within
    // 2e-4 degree, mass drift below 1e-8 and C within 1e-7 of the oracle
    // after 20 steps, the FP32 level of the other terms
    st->sweeps = params->solver_iters ? params->solver_iters
                                      : (st->mode == FELBM_SOLVER_FP64 ? 32 : (dev32 ? 10 : 14));
    st->rounds = st->mode == FELBM_SOLVER_FP64 ? 1 : (params->solver_rounds ? params->solver_rounds : (dev32 ? 1 : 3));
    const double lmin = 0.25, lmax = 1.0;
    const double theta = 0.5 * (lmax + lmin), delta = 0.5 * (lmax - lmin), sigma1 = theta / delta;
    st->inv_theta = 1.0 / theta;
    st->cheb_a.assign(st->sweeps, 0.0);
    st->cheb_c.assign(st->sweeps, 0.0);
    double rho_prev = 1.0 / sigma1;
    for (int k = 1; k < st->sweeps; ++k) {
        double rho = 1.0 / (2.0 * sigma1 - rho_prev);
        st->cheb_a[k] = rho * rho_prev;
        st->cheb_c[k] = 2.0 * rho / delta;
        rho_prev = rho;
    }
    // FP32 solves: Richardson steps 1/lambda_j at the Chebyshev roots
    // lambda_j = theta + delta cos((2j+1) pi / 2K), j = 0..K-1, in the order
    // j = 0, K-1, 1, K-2, ... (largest and smallest root alternately)
    st->tau.assign(st->sweeps, 1.0);
    {
        const int K = st->sweeps;
        for (int k = 0; k < K; ++k) {
            const int j = (k & 1) ? K - 1 - k / 2 : k / 2;
            st->tau[k] = 1.0 / (theta + delta * std::cos((2.0 * j + 1.0) * 3.14159265358979323846 / (2.0 * K)));
        }
    }

    // host-side derived tables
    const double scale = params->lap_mode == FELBM_LAP_PAPER ? 1.0 : 2.0 / 3.0;
    std::vector<double> inv_vol(h.N), inv_lumped(h.N), lval(h.row_ptr[h.N]);
    std::vector<float2> start32(h.N);
    std::vector<float> inv_lumped32(h.N), mval32(h.mass.begin(), h.mass.end());
    std::vector<double> wall_phi(h.E);
    for (int32_t e = 0; e < h.E; ++e) wall_phi[e] = params->phi_c[h.wall_id[e]];
    const int ellw = st->dm.ell_w;
    std::vector<int32_t> ell_col((size_t)std::max(ellw, 1) * st->dm.Np, 0);
    std::vector<float> ell_val((size_t)std::max(ellw, 1) * st->dm.Np, 0.0f);
    std::vector<double> ell_lval((size_t)std::max(ellw, 1) * st->dm.Np, 0.0);
    if (const char* env = std::getenv("FELBM_PDL")) st->use_pdl = std::atoi(env) != 0;
    for (int32_t i = 0; i < h.N; ++i) {
        inv_vol[i] = 1.0 / (scale * h.patch[i]);
        inv_lumped[i] = 1.0 / h.lumped[i];
        inv_lumped32[i] = (float)inv_lumped[i];
        start32[i] = split_scale(inv_lumped[i] * st->tau[0]);
        for (int32_t k = h.row_ptr[i]; k < h.row_ptr[i + 1]; ++k) lval[k] = -2.0 * h.stiff[k] * inv_vol[i];
    }
    for (int32_t i = 0; i < h.N && ellw > 0; ++i) {
        // the diagonal first (the solve steps hold the node's own value already),
        // then the other columns in order
        const int32_t r0 = h.row_ptr[i], len = h.row_ptr[i + 1] - r0;
        int at_k = 1;
        for (int k = 0; k < len; ++k) {
            const int32_t c = h.col[r0 + k];
            const size_t at = (size_t)(c == i ? 0 : at_k++) * st->dm.Np + i;
            ell_col[at] = c;
            ell_val[at] = (float)h.mass[r0 + k];
            ell_lval[at] = lval[r0 + k];
        }
        for (int k = len; k < ellw; ++k) ell_col[(size_t)k * st->dm.Np + i] = i;
    }
    // the blocked solve's rows: a block's node list is its own run, then its
    // layers; every node but the last layer's gets its ELL row with columns as
    // indices into that list (padding: the node itself with entry 0)
    const int32_t nblk = st->dm.n_blocks;
    std::vector<int32_t> blk_row(nblk + 1, 0);
    std::vector<float> blk_val;
    std::vector<uint32_t> blk_col;
    if (st->dm.blk_steps > 0) {
        const int wc = ellw / 2;
        const int64_t rows = block_rows(h, blk_row.data());
        blk_val.assign((size_t)rows * ellw, 0.0f);
        blk_col.assign((size_t)rows * wc, 0);
        std::atomic<int> stray{0};
        const int32_t Np = st->dm.Np;
        parallel_for(nblk, 4, []() { return NodePlaces(); }, [&](int32_t t, NodePlaces& around) {
            const int32_t s0 = h.blk_ptr[t], ni = h.blk_ptr[t + 1] - s0;
            const int32_t* cnt = h.layer_cnt.data() + (size_t)t * (kBlockSteps + 1);
            const int32_t* halo = h.halo.data() + h.halo_ptr[t];
            const int32_t nr = cnt[h.n_layers - 1], stride = blk_row[t + 1] - blk_row[t];
            float* val = blk_val.data() + (size_t)ellw * blk_row[t];
            uint32_t* col = blk_col.data() + (size_t)wc * blk_row[t];
            around.clear();
            for (int32_t r = ni; r < cnt[h.n_layers]; ++r) around.add(halo[r - ni], r);
            for (int32_t r = 0; r < nr; ++r) {
                const int32_t i = r < ni ? s0 + r : halo[r - ni];
                for (int k = 0; k < ellw; ++k) {
                    val[(size_t)k * stride + r] = ell_val[(size_t)k * Np + i];
                    if (k == 0) continue;
                    const int32_t c = ell_col[(size_t)k * Np + i];
                    uint32_t at = (uint32_t)(c - s0);
                    if (c < s0 || c >= s0 + ni) {
                        const size_t slot = around.slot(c);
                        if (around.node[slot] != c) stray = 1;
                        at = around.node[slot] == c ? (uint32_t)around.place[slot] : (uint32_t)r;
                    }
                    uint32_t& pair = col[(size_t)((k - 1) / 2) * stride + r];
                    pair = (k & 1) ? at | (uint32_t)r << 16 : (pair & 0xffffu) | at << 16;
                }
            }
        });
        if (stray) {
            set_error("felbm_init: internal error, a row entry outside its block's layers");
            return FELBM_ERR_BAD_MESH;
        }
    }
    auto pad_tri = [&](const std::vector<int32_t>& src, int rows) {
        std::vector<int32_t> outv((size_t)rows * st->dm.Tp, 0);
        for (int r = 0; r < rows; ++r)
            std::copy(src.begin() + (size_t)r * h.T, src.begin() + (size_t)(r + 1) * h.T,
                      outv.begin() + (size_t)r * st->dm.Tp);
        return outv;
    };
    auto pad_trid = [&](const std::vector<double>& src, int rows) {
        std::vector<double> outv((size_t)rows * st->dm.Tp, 0.0);
        for (int r = 0; r < rows; ++r)
            std::copy(src.begin() + (size_t)r * h.T, src.begin() + (size_t)(r + 1) * h.T,
                      outv.begin() + (size_t)r * st->dm.Tp);
        return outv;
    };
    std::vector<int32_t> tri_p = pad_tri(h.tri, 3), nbr_p = pad_tri(h.nbr, 3), slot_p = pad_tri(h.nbr_slot, 3);
    std::vector<double> grad_p = pad_trid(h.grad, 6), area_p = pad_trid(h.area, 1);
    std::vector<float> grad32_p(grad_p.begin(), grad_p.end()), area32_p(area_p.begin(), area_p.end());
    std::vector<float> inc_bx32(h.inc_bx.begin(), h.inc_bx.end()), inc_by32(h.inc_by.begin(), h.inc_by.end());
    // node -> triangle incidence (padding: the zero residual row T), and as indices
    // into the block's triangle list (padding: past its end)
    const int iw = st->dm.iell_w;
    std::vector<int32_t> itri((size_t)std::max(iw, 1) * st->dm.Np, h.T);
    std::vector<float> ibx(itri.size(), 0.0f), iby(itri.size(), 0.0f);
    for (int32_t i = 0; i < h.N && iw > 0; ++i)
        for (int32_t k = h.inc_ptr[i]; k < h.inc_ptr[i + 1]; ++k) {
            const size_t at = (size_t)(k - h.inc_ptr[i]) * st->dm.Np + i;
            itri[at] = h.inc_tri[k];
            ibx[at] = inc_bx32[k];
            iby[at] = inc_by32[k];
        }
    std::vector<uint16_t> iloc;
    if (st->dm.max_blk_tri > 0) {
        iloc.resize((size_t)iw * st->dm.Np);
        parallel_for(nblk, 4, []() { return 0; }, [&](int32_t t, int&) {
            const int32_t* l0 = h.blk_tri.data() + h.blk_tri_ptr[t];
            const int32_t* l1 = h.blk_tri.data() + h.blk_tri_ptr[t + 1];
            for (int32_t i = h.blk_ptr[t]; i < h.blk_ptr[t + 1]; ++i)
                for (int k = 0; k < iw; ++k) {
                    const size_t at = (size_t)k * st->dm.Np + i;
                    iloc[at] = (uint16_t)(itri[at] < h.T ? std::lower_bound(l0, l1, itri[at]) - l0 : l1 - l0);
                }
        });
    }
    // The tables above are all made before the first copy and outlive the last: a
    // copy from pageable memory may still read them when the call returns, so the
    // stream is waited for on every way out.
    cudaStream_t s = st->stream;
    const DevMesh& d = st->dm;
    auto fail = [&](cudaError_t e, const char* what) {
        cudaStreamSynchronize(s);
        return cuda_fail(e, what);
    };
    cudaError_t e = cudaSuccess;
#define UP(dst, src) \
    if (e == cudaSuccess) e = up(dst, src, s)
    UP(d.tri, tri_p);
    UP(d.area, area_p);
    UP(d.grad, grad_p);
    UP(d.grad32, grad32_p);
    UP(d.area32, area32_p);
    UP(d.nbr, nbr_p);
    UP(d.nbr_slot, slot_p);
    UP(d.row_ptr, h.row_ptr);
    UP(d.col, h.col);
    UP(d.mval, h.mass);
    UP(d.lval, lval);
    UP(d.inv_lumped, inv_lumped);
    UP(d.mval32, mval32);
    UP(d.ell_col, ell_col);
    UP(d.ell_val, ell_val);
    UP(d.blk_ptr, h.blk_ptr);
    UP(d.blk_cnt, h.layer_cnt);
    UP(d.blk_halo_ptr, h.halo_ptr);
    UP(d.blk_halo, h.halo);
    UP(d.blk_row, blk_row);
    UP(d.blk_val, blk_val);
    UP(d.blk_col, blk_col);
    int cur_dev = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&cur_dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&st->n_sm, cudaDevAttrMultiProcessorCount, cur_dev);
    if (e == cudaSuccess && st->dm.blk_steps > 0) {
        switch (ellw) {
            case 7: e = allow_block_smem<7>(); break;
            case 9: e = allow_block_smem<9>(); break;
            default: e = allow_block_smem<12>();
        }
    }
    UP(d.ell_lval, ell_lval);
    UP(d.inv_lumped32, inv_lumped32);
    UP(d.start32, start32);
    UP(d.lumped, h.lumped);
    UP(d.inv_vol, inv_vol);
    UP(d.inc_ptr, h.inc_ptr);
    UP(d.inc_tri, h.inc_tri);
    UP(d.inc_bx, h.inc_bx);
    UP(d.inc_by, h.inc_by);
    UP(d.inc_bx32, inc_bx32);
    UP(d.inc_by32, inc_by32);
    UP(d.iell_tri, itri);
    UP(d.iell_bx32, ibx);
    UP(d.iell_by32, iby);
    if (st->dm.max_blk_tri > 0) {
        UP(d.blk_tri_ptr, h.blk_tri_ptr);
        UP(d.blk_tri, h.blk_tri);
        UP(d.iell_loc, iloc);
        // (the limit holds for every state of the process: the largest any may ask for)
        const int bytes = (int)force_smem_bytes(kForceTris);
        const auto allow = [&](auto kern) {
            if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        };
        allow(k_force32<6>);
        allow(k_force32<8>);
        allow(k_force32<12>);
    }
    if (dev32 && e == cudaSuccess) e = cudaMemsetAsync(st->buf.R32 + (size_t)18 * h.T, 0, 18 * sizeof(float), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(st->buf.diag_done, 0, sizeof(unsigned), s);
    UP(d.wall_a, h.wall_a);
    UP(d.wall_b, h.wall_b);
    UP(d.wall_id, h.wall_id);
    UP(d.wall_phi, wall_phi);
    UP(d.wall_len, h.wall_len);
    UP(d.wall_nx, h.wall_nx);
    UP(d.wall_ny, h.wall_ny);
    UP(d.winc_ptr, h.winc_ptr);
    UP(d.winc_edge, h.winc_edge);
    UP(d.x, h.x);
    UP(d.y, h.y);
    UP(d.perm, h.perm);
    UP(d.iperm, h.iperm);
    UP(st->gt.node_begin, h.grp_node_begin);
    UP(st->gt.node_end, h.grp_node_end);
    UP(st->gt.tri_begin, h.grp_tri_begin);
    UP(st->gt.tri_end, h.grp_tri_end);
    UP(st->gt.wall_ptr, h.grp_wall_ptr);
    UP(st->gt.wall_edge, h.grp_wall_edge);
    if (!dev32) UP(st->adj.kval, h.stiff);
#undef UP
    if (e != cudaSuccess) return fail(e, "felbm_init: upload");
    {
        double* dst = st->buf.stage;
        e = cudaMemcpyAsync(dst, C0, sizeof(double) * h.N, cudaMemcpyHostToDevice, s);
        dst += h.N;
        if (e == cudaSuccess && p0) {
            e = cudaMemcpyAsync(dst, p0, sizeof(double) * h.N, cudaMemcpyHostToDevice, s);
            dst += h.N;
        }
        if (e == cudaSuccess && u0) e = cudaMemcpyAsync(dst, u0, sizeof(double) * 2 * h.N, cudaMemcpyHostToDevice, s);
    }
    if (e != cudaSuccess) return fail(e, "felbm_init: upload C0, p0, u0");
    if (dev32)
        k_init_dev32<<<grid_for(h.N, kBlock), kBlock, 0, s>>>(st->dm, st->buf, st->buf.stage, p0 != nullptr,
                                                               u0 != nullptr);
    else
        k_init_state<<<grid_for(h.N, kBlock), kBlock, 0, s>>>(st->dm, st->phys, st->buf.stage, st->buf.psi,
                                                               p0 != nullptr, u0 != nullptr);
    e = cudaGetLastError();
    if (e != cudaSuccess) return fail(e, "felbm_init: launch");
    e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return fail(e, "felbm_init: synchronize");
    e = cudaGetDevice(&st->device);
    if (e != cudaSuccess) return fail(e, "felbm_init: cudaGetDevice");
    // mass at t = 0 (for the drift)
    felbm_diag dg;
    int rc = felbm_diagnostics(st, nullptr, &dg);
    if (rc != FELBM_OK && rc != FELBM_ERR_NONFINITE) return rc;
    st->mass0 = dg.mass;
    st->gmass0.assign(h.G, dg.mass);
    if (h.G > 1) {   // one member: its mass is the mass
        std::vector<felbm_diag> gd(h.G);
        rc = felbm_diagnostics_groups(st, nullptr, h.G, gd.data());
        if (rc != FELBM_OK && rc != FELBM_ERR_NONFINITE) return rc;
        for (int32_t g = 0; g < h.G; ++g) st->gmass0[g] = gd[g].mass;
    }
    return set_schedule(st, 0);
}

int felbm_init(const felbm_mesh* mesh, const felbm_params* params, const double* C0, const double* p0,
               const double* u0, void* d_workspace, size_t workspace_bytes, void* stream, felbm_state** out) {
    if (!mesh || !C0 || !out) {
        set_error("felbm_init: invalid argument");
        return FELBM_ERR_INVALID_ARG;
    }
    *out = nullptr;
    int rc = check_params(params);
    if (rc) return rc;
    const HostMesh& h = mesh->h;
    for (int32_t e = 0; e < h.E; ++e)
        if (h.wall_id[e] >= params->n_wall_ids) {
            set_error("felbm_init: a wall id has no phi_c (n_wall_ids too small)");
            return FELBM_ERR_INVALID_ARG;
        }
    const bool dev32 = params->precision == FELBM_FP32_DEV;
    size_t need = carve(h, dev32, nullptr, nullptr, nullptr);
    if (!d_workspace || workspace_bytes < need || (reinterpret_cast<uintptr_t>(d_workspace) & 255)) {
        set_error("felbm_init: workspace missing, not 256-byte aligned or smaller than felbm_workspace_bytes");
        return FELBM_ERR_WORKSPACE;
    }
    felbm_state* st = new (std::nothrow) felbm_state;
    if (!st) {
        set_error("felbm_init: out of host memory");
        return FELBM_ERR_INVALID_ARG;
    }
    try {
        rc = set_up(st, h, params, C0, p0, u0, d_workspace, stream);
    } catch (const std::exception& ex) {
        set_error(std::string("felbm_init: ") + ex.what());
        rc = FELBM_ERR_INVALID_ARG;
    }
    if (rc != FELBM_OK) {
        delete st;
        return rc;
    }
    *out = st;
    return FELBM_OK;
}

}  // extern "C"

namespace felbm {

// Split the groups: those of at most max_nodes nodes run one CTA each.  The
// groups are laid out largest first, so the others form a prefix.
int set_schedule(felbm_state* st, int32_t max_nodes) {
    const HostMesh& h = st->hm;
    std::vector<int32_t> cta;
    int32_t tiled_N = 0, tiled_T = 0;
    for (int32_t g = 0; g < h.G; ++g) {
        if (st->dev32 && max_nodes > 0 && h.grp_size[g] <= max_nodes) {
            cta.push_back(g);
        } else {
            tiled_N = std::max(tiled_N, h.grp_node_end[g]);
            tiled_T = std::max(tiled_T, h.grp_tri_end[g]);
        }
    }
    for (int32_t g : cta)
        if (h.grp_node_begin[g] < tiled_N || h.grp_tri_begin[g] < tiled_T) {
            set_error("felbm: batch schedule needs the small members after the large ones");
            return FELBM_ERR_INVALID_ARG;
        }
    if (st->sweeps >= kMaxSweeps && !cta.empty()) {
        set_error("felbm: too many solver sweeps for the per-member CTA schedule");
        return FELBM_ERR_UNSUPPORTED;
    }
    if (!cta.empty()) {
        if (!st->side_stream) FELBM_CUDA(cudaStreamCreateWithFlags(&st->side_stream, cudaStreamNonBlocking));
        if (!st->ev_fork) FELBM_CUDA(cudaEventCreateWithFlags(&st->ev_fork, cudaEventDisableTiming));
        if (!st->ev_join) FELBM_CUDA(cudaEventCreateWithFlags(&st->ev_join, cudaEventDisableTiming));
        FELBM_CUDA(cudaMemcpyAsync(st->gt.cta_groups, cta.data(), sizeof(int32_t) * cta.size(),
                                   cudaMemcpyHostToDevice, st->stream));
        FELBM_CUDA(cudaStreamSynchronize(st->stream));
    }
    st->cta_max_nodes = cta.empty() ? 0 : max_nodes;
    st->n_cta = (int32_t)cta.size();
    st->tiled_N = tiled_N;
    st->tiled_T = tiled_T;
    st->tiled_blocks = (int32_t)(std::upper_bound(h.blk_ptr.begin(), h.blk_ptr.end(), tiled_N) - h.blk_ptr.begin()) - 1;
    return FELBM_OK;
}

}  // namespace felbm

extern "C" {

static int build_graph(felbm_state* st) {
    if (!st->cap_stream) FELBM_CUDA(cudaStreamCreateWithFlags(&st->cap_stream, cudaStreamNonBlocking));
    FELBM_CUDA(cudaStreamBeginCapture(st->cap_stream, cudaStreamCaptureModeThreadLocal));
    enqueue_step(st, st->cap_stream);
    cudaError_t e = cudaStreamEndCapture(st->cap_stream, &st->graph);
    if (e != cudaSuccess) return cuda_fail(e, "felbm_step: capture");
    FELBM_CUDA(cudaGraphInstantiate(&st->graph_exec, st->graph, 0));
    return FELBM_OK;
}

int felbm_step(felbm_state* st, int32_t n_steps) {
    if (!st || n_steps < 0) {
        set_error("felbm_step: invalid argument");
        return FELBM_ERR_INVALID_ARG;
    }
    if (!st->graph_exec) {
        int rc = build_graph(st);
        if (rc) return rc;
    }
    for (int32_t k = 0; k < n_steps; ++k) FELBM_CUDA(cudaGraphLaunch(st->graph_exec, st->stream));
    st->step += n_steps;
    if (n_steps > 0 && st->timing) st->timed_step_ran = true;
    return FELBM_OK;
}

static void drop_graph(felbm_state* st) {
    if (st->graph_exec) cudaGraphExecDestroy(st->graph_exec);
    if (st->graph) cudaGraphDestroy(st->graph);
    st->graph_exec = nullptr;
    st->graph = nullptr;
}

int felbm_timing_enable(felbm_state* st, int32_t enable) {
    if (!st) {
        set_error("felbm_timing_enable: invalid argument");
        return FELBM_ERR_INVALID_ARG;
    }
    if (enable && !st->ev[0])
        for (auto& e : st->ev) FELBM_CUDA(cudaEventCreate(&e));
    FELBM_CUDA(cudaStreamSynchronize(st->stream));
    drop_graph(st);
    st->timing = enable != 0;
    st->timed_step_ran = false;
    return FELBM_OK;
}

int felbm_fp64_fma_rate(void* stream, double* tflops) {
    if (!tflops) {
        set_error("felbm_fp64_fma_rate: invalid argument");
        return FELBM_ERR_INVALID_ARG;
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int dev = 0, n_sm = 0;
    FELBM_CUDA(cudaGetDevice(&dev));
    FELBM_CUDA(cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev));
    const int blocks = n_sm * 8, iters = 4096;
    cudaEvent_t e0, e1;
    FELBM_CUDA(cudaEventCreate(&e0));
    FELBM_CUDA(cudaEventCreate(&e1));
    float best = 1e30f;
    for (int rep = 0; rep < 4; ++rep) {   // the first launch is a warm-up
        cudaEventRecord(e0, s);
        k_fp64_fma_rate<<<blocks, 256, 0, s>>>(iters, 0.999999);
        cudaEventRecord(e1, s);
        cudaError_t e = cudaEventSynchronize(e1);
        float ms = 0.0f;
        if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
        if (e != cudaSuccess) {
            cudaEventDestroy(e0);
            cudaEventDestroy(e1);
            return cuda_fail(e, "felbm_fp64_fma_rate");
        }
        if (rep > 0) best = std::min(best, ms);
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    *tflops = 2.0 * 8.0 * iters * (double)blocks * 256.0 / (best * 1e-3) / 1e12;
    return FELBM_OK;
}

int felbm_timing_get(felbm_state* st, felbm_step_timing* out) {
    if (!st || !out || !st->timing || !st->timed_step_ran) {
        set_error("felbm_timing_get: timing is off or no timed step ran");
        return FELBM_ERR_INVALID_ARG;
    }
    FELBM_CUDA(cudaStreamSynchronize(st->stream));
    float t[6];
    for (int k = 0; k < 6; ++k) FELBM_CUDA(cudaEventElapsedTime(&t[k], st->ev[k], st->ev[k + 1]));
    out->collide_ms = t[0];
    out->mu_ms = t[1];
    out->gradmu_ms = t[2];
    out->element_ms = t[3];
    out->rhs_ms = t[4];
    out->solve_ms = t[5];
    out->total_ms = t[0] + t[1] + t[2] + t[3] + t[4] + t[5];
    const DevMesh m = launched_part(st);
    out->solve_launches = solve_launches(st, m);
    out->launches = step_launches(st, m);
    return FELBM_OK;
}

}  // extern "C"

namespace felbm {

static DiagReq make_req(const felbm_state* st, const felbm_diag_request* req) {
    DiagReq rq{};
    rq.period_x = st->hm.period[0];
    rq.period_y = st->hm.period[1];
    rq.substrate = req ? req->substrate_wall_id : 0;
    rq.use_band = req && req->band > 0.0;
    if (req) {
        rq.cx = req->centre[0];
        rq.cy = req->centre[1];
        rq.R = req->radius;
        rq.band = req->band;
    }
    return rq;
}

// felbm_diag from the reduced slots; the contact angle uses the mean height
// of the substrate wall nodes among the given wall edges.
// The diagnostics reductions of the whole mesh into buf.diag_out.
static void enqueue_diag(felbm_state* st, const DiagReq& rq, cudaStream_t s) {
    if (st->dev32) {
        k_diag_fused32<<<kDiagBlocks, kBlock, 0, s>>>(st->dm, st->phys, st->buf, rq);
        return;
    }
    k_diag_nodes<false><<<kDiagBlocks, kBlock, 0, s>>>(st->dm, st->phys, st->buf, rq);
    k_diag_edges<<<kDiagBlocks, kBlock, 0, s>>>(st->dm, st->buf, rq);
    k_diag_final<<<1, kDiagSums * 32, 0, s>>>(st->buf);
}

// res: the two sums of the solve check (sum r^2, sum b^2), read when it is on.
static felbm_diag fill_diag(const felbm_state* st, const double* v, double mass0, int64_t nodes, int substrate,
                            const int32_t* edges, int32_t n_edges, int64_t step, const double* res) {
    const HostMesh& h = st->hm;
    felbm_diag d{};
    d.step = step;
    d.mass = v[0];
    d.mass0 = mass0;
    d.mass_drift_rel = mass0 != 0.0 ? (v[0] - mass0) / mass0 : 0.0;
    d.kinetic_energy = 0.5 * v[1] / (double)std::max<int64_t>(nodes, 1);
    d.max_u = std::sqrt(v[10]);
    d.interface_rho_uu = v[2] > 0.0 ? v[3] / v[2] : 0.0;
    d.p_in = v[5] / std::max(v[4], 1e-300);
    d.p_out = v[7] / std::max(v[6], 1e-300);
    d.delta_p = d.p_in - d.p_out;
    d.wetted_length = v[11];
    double ysum = 0.0;
    int ny = 0;
    std::vector<int32_t> nodes_seen;
    for (int32_t k = 0; k < n_edges; ++k) {
        int32_t e = edges ? edges[k] : k;
        if (h.wall_id[e] != substrate) continue;
        nodes_seen.push_back(h.wall_a[e]);
        nodes_seen.push_back(h.wall_b[e]);
    }
    std::sort(nodes_seen.begin(), nodes_seen.end());
    nodes_seen.erase(std::unique(nodes_seen.begin(), nodes_seen.end()), nodes_seen.end());
    for (int32_t n : nodes_seen) {
        ysum += h.y[n];
        ++ny;
    }
    d.height = ny ? v[12] - ysum / ny : std::nan("");
    double b = d.wetted_length, hh = d.height;
    if (ny && hh > 0.0 && b > 0.0) {
        double r = (4.0 * hh * hh + b * b) / (8.0 * hh);
        d.theta_deg = std::atan2(b, 2.0 * (r - hh)) * 180.0 / M_PI;
    } else {
        d.theta_deg = std::nan("");
    }
    d.status = v[9] > 0.0 ? FELBM_ERR_NONFINITE : FELBM_OK;
    d.solver_sweeps = st->mode == FELBM_SOLVER_FP64 ? st->sweeps : st->sweeps * st->rounds;
    d.solver_residual = std::nan("");
    if (st->check && res) {
        d.solver_residual = std::sqrt(res[0] / std::max(res[1], 1e-300));
        if (d.status == FELBM_OK && !(d.solver_residual <= st->check_tol)) d.status = FELBM_ERR_NOT_CONVERGED;
    }
    return d;
}

}  // namespace felbm

extern "C" {

int felbm_diagnostics(felbm_state* st, const felbm_diag_request* req, felbm_diag* out) {
    if (!st || !out) {
        set_error("felbm_diagnostics: invalid argument");
        return FELBM_ERR_INVALID_ARG;
    }
    DiagReq rq = make_req(st, req);
    cudaStream_t s = st->stream;
    enqueue_diag(st, rq, s);
    FELBM_CUDA(cudaGetLastError());
    double v[kDiagSlots];
    FELBM_CUDA(cudaMemcpyAsync(v, st->buf.diag_out, sizeof v, cudaMemcpyDeviceToHost, s));
    FELBM_CUDA(cudaStreamSynchronize(s));
    *out = fill_diag(st, v, st->mass0, st->hm.N, rq.substrate, nullptr, st->hm.E, st->step, v + kSolveResSlot);
    if (out->status == FELBM_ERR_NOT_CONVERGED) {
        set_error("felbm_diagnostics: the last solve's residual is above the tolerance of felbm_solver_check");
        return FELBM_ERR_NOT_CONVERGED;
    }
    if (out->status != FELBM_OK) {
        set_error("felbm_diagnostics: non-finite values in the state");
        return FELBM_ERR_NONFINITE;
    }
    return FELBM_OK;
}

int felbm_diagnostics_enqueue(felbm_state* st, const felbm_diag_request* req, double* slots) {
    if (!st || !slots) {
        set_error("felbm_diagnostics_enqueue: invalid argument");
        return FELBM_ERR_INVALID_ARG;
    }
    static_assert(kDiagSlots == FELBM_DIAG_SLOTS, "raw diagnostic sums");
    DiagReq rq = make_req(st, req);
    cudaStream_t s = st->stream;
    enqueue_diag(st, rq, s);
    FELBM_CUDA(cudaGetLastError());
    // the reduced sums arrive asynchronously; the step count is the host's now
    FELBM_CUDA(cudaMemcpyAsync(slots, st->buf.diag_out, sizeof(double) * (kSolveResSlot + 2), cudaMemcpyDeviceToHost,
                               s));
    slots[kDiagStepSlot] = (double)st->step;
    return FELBM_OK;
}

int felbm_diag_finish(felbm_state* st, const felbm_diag_request* req, const double* slots, felbm_diag* out) {
    if (!st || !slots || !out) {
        set_error("felbm_diag_finish: invalid argument");
        return FELBM_ERR_INVALID_ARG;
    }
    const DiagReq rq = make_req(st, req);
    *out = fill_diag(st, slots, st->mass0, st->hm.N, rq.substrate, nullptr, st->hm.E,
                     (int64_t)slots[kDiagStepSlot], slots + kSolveResSlot);
    if (out->status == FELBM_ERR_NOT_CONVERGED) {
        set_error("felbm_diag_finish: the last solve's residual is above the tolerance of felbm_solver_check");
        return FELBM_ERR_NOT_CONVERGED;
    }
    if (out->status != FELBM_OK) {
        set_error("felbm_diag_finish: non-finite values in the state");
        return FELBM_ERR_NONFINITE;
    }
    return FELBM_OK;
}

int felbm_diagnostics_groups(felbm_state* st, const felbm_diag_request* reqs, int32_t n_groups, felbm_diag* out) {
    if (!st || !out || n_groups != st->hm.G || n_groups < 1) {
        set_error("felbm_diagnostics_groups: invalid argument (n_groups must equal the mesh's group count)");
        return FELBM_ERR_INVALID_ARG;
    }
    const HostMesh& h = st->hm;
    std::vector<DiagReq> rq(n_groups);
    for (int32_t g = 0; g < n_groups; ++g) {
        rq[g] = make_req(st, reqs ? reqs + g : nullptr);
        rq[g].period_x = h.grp_period_x[g];
        rq[g].period_y = h.grp_period_y[g];
    }
    cudaStream_t s = st->stream;
    FELBM_CUDA(cudaMemcpyAsync(st->gt.reqs, rq.data(), sizeof(DiagReq) * n_groups, cudaMemcpyHostToDevice, s));
    if (st->dev32)
        k_diag_groups<true><<<n_groups, kBlock, 0, s>>>(st->dm, st->phys, st->buf, st->gt);
    else
        k_diag_groups<false><<<n_groups, kBlock, 0, s>>>(st->dm, st->phys, st->buf, st->gt);
    FELBM_CUDA(cudaGetLastError());
    std::vector<double> v((size_t)n_groups * kDiagSlots);
    double res[2] = {0.0, 0.0};
    FELBM_CUDA(cudaMemcpyAsync(v.data(), st->gt.out, sizeof(double) * v.size(), cudaMemcpyDeviceToHost, s));
    FELBM_CUDA(cudaMemcpyAsync(res, st->buf.diag_out + kSolveResSlot, sizeof res, cudaMemcpyDeviceToHost, s));
    FELBM_CUDA(cudaStreamSynchronize(s));
    bool bad = false, unconverged = false;
    for (int32_t g = 0; g < n_groups; ++g) {
        const double* vg = v.data() + (size_t)g * kDiagSlots;
        double m0 = g < (int32_t)st->gmass0.size() ? st->gmass0[g] : vg[0];
        out[g] = fill_diag(st, vg, m0, h.grp_size[g], rq[g].substrate, h.grp_wall_edge.data() + h.grp_wall_ptr[g],
                           h.grp_wall_ptr[g + 1] - h.grp_wall_ptr[g], st->step, res);
        bad = bad || out[g].status == FELBM_ERR_NONFINITE;
        unconverged = unconverged || out[g].status == FELBM_ERR_NOT_CONVERGED;
    }
    if (bad) {
        set_error("felbm_diagnostics_groups: non-finite values in the state");
        return FELBM_ERR_NONFINITE;
    }
    if (unconverged) {
        set_error("felbm_diagnostics_groups: the last solve's residual is above the tolerance of felbm_solver_check");
        return FELBM_ERR_NOT_CONVERGED;
    }
    return FELBM_OK;
}

int felbm_get_state(felbm_state* st, double* g, double* h) {
    if (!st || !g || !h) {
        set_error("felbm_get_state: invalid argument");
        return FELBM_ERR_INVALID_ARG;
    }
    cudaStream_t s = st->stream;
    const int N = st->dm.N;
    if (st->dev32)
        k_dev32_to_full<<<grid_for(N, kBlock), kBlock, 0, s>>>(st->dm, st->phys, st->buf, st->buf.stage);
    else
        k_gather_out<<<grid_for(N, kBlock), kBlock, 0, s>>>(st->dm, st->buf.psi, st->buf.stage, 18);
    FELBM_CUDA(cudaGetLastError());
    FELBM_CUDA(cudaMemcpyAsync(g, st->buf.stage, sizeof(double) * 9 * N, cudaMemcpyDeviceToHost, s));
    FELBM_CUDA(cudaMemcpyAsync(h, st->buf.stage + (size_t)9 * N, sizeof(double) * 9 * N, cudaMemcpyDeviceToHost, s));
    FELBM_CUDA(cudaStreamSynchronize(s));
    return FELBM_OK;
}

int felbm_set_state(felbm_state* st, const double* g, const double* h) {
    if (!st || !g || !h) {
        set_error("felbm_set_state: invalid argument");
        return FELBM_ERR_INVALID_ARG;
    }
    cudaStream_t s = st->stream;
    const int N = st->dm.N;
    if (!st->copy_stream) FELBM_CUDA(cudaStreamCreateWithFlags(&st->copy_stream, cudaStreamNonBlocking));
    if (!st->ev_copied) FELBM_CUDA(cudaEventCreateWithFlags(&st->ev_copied, cudaEventDisableTiming));
    for (auto& ev : st->ev_in_free)
        if (!ev) FELBM_CUDA(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
    // The copy runs on its own stream into the input buffer not used by the
    // previous call, so it overlaps whatever the state's stream is running
    // (the previous step); it waits only for the conversion that last read
    // this buffer.  The conversion waits for the copy on the state's stream.
    const int k = st->in_next;
    st->in_next ^= 1;
    double* in = k ? st->buf.in1 : st->buf.in0;
    FELBM_CUDA(cudaStreamWaitEvent(st->copy_stream, st->ev_in_free[k], 0));
    FELBM_CUDA(cudaMemcpyAsync(in, g, sizeof(double) * 9 * N, cudaMemcpyHostToDevice, st->copy_stream));
    FELBM_CUDA(cudaMemcpyAsync(in + (size_t)9 * N, h, sizeof(double) * 9 * N, cudaMemcpyHostToDevice, st->copy_stream));
    FELBM_CUDA(cudaEventRecord(st->ev_copied, st->copy_stream));
    FELBM_CUDA(cudaStreamWaitEvent(s, st->ev_copied, 0));
    if (st->dev32)
        k_full_to_dev32<<<grid_for(N, kBlock), kBlock, 0, s>>>(st->dm, st->phys, st->buf, in);
    else
        k_scatter_in<<<grid_for(N, kBlock), kBlock, 0, s>>>(st->dm, in, st->buf.psi, 18);
    FELBM_CUDA(cudaGetLastError());
    FELBM_CUDA(cudaEventRecord(st->ev_in_free[k], s));
    // return once the host arrays have been read; the conversion stays queued
    FELBM_CUDA(cudaEventSynchronize(st->ev_copied));
    return FELBM_OK;
}

int felbm_get_fields(felbm_state* st, double* C, double* p, double* ux, double* uy, double* mu) {
    if (!st) {
        set_error("felbm_get_fields: invalid argument");
        return FELBM_ERR_INVALID_ARG;
    }
    cudaStream_t s = st->stream;
    const DevMesh& m = st->dm;
    double* outs[5] = {C, p, ux, uy, mu};
    if (st->dev32) {
        k_mu32<0><<<grid_for(m.N, kBlock), kBlock, 0, s>>>(m, st->phys, st->buf);
        FELBM_CUDA(cudaGetLastError());
        const float* srcs[5] = {nullptr, st->buf.p32, st->buf.ux32, st->buf.uy32, st->buf.mu32};
        for (int k = 0; k < 5; ++k) {
            if (!outs[k]) continue;
            if (k == 0)
                k_gather_out<<<grid_for(m.N, kBlock), kBlock, 0, s>>>(m, st->buf.C, st->buf.stage, 1);
            else
                k_gather_out_f<<<grid_for(m.N, kBlock), kBlock, 0, s>>>(m, srcs[k], st->buf.stage);
            FELBM_CUDA(cudaGetLastError());
            FELBM_CUDA(cudaMemcpyAsync(outs[k], st->buf.stage, sizeof(double) * m.N, cudaMemcpyDeviceToHost, s));
            FELBM_CUDA(cudaStreamSynchronize(s));
        }
        return FELBM_OK;
    }
    k_collide<<<grid_for(m.N, kBlock), kBlock, 0, s>>>(m, st->phys, st->buf, 0);
    launch_mu(m, st->phys, st->buf, grid_for(m.N, kBlock), kBlock, s);
    FELBM_CUDA(cudaGetLastError());
    double* srcs[5] = {st->buf.C, st->buf.p, st->buf.ux, st->buf.uy, st->buf.mu};
    for (int k = 0; k < 5; ++k) {
        if (!outs[k]) continue;
        k_gather_out<<<grid_for(m.N, kBlock), kBlock, 0, s>>>(m, srcs[k], st->buf.stage, 1);
        FELBM_CUDA(cudaGetLastError());
        FELBM_CUDA(cudaMemcpyAsync(outs[k], st->buf.stage, sizeof(double) * m.N, cudaMemcpyDeviceToHost, s));
        FELBM_CUDA(cudaStreamSynchronize(s));
    }
    return FELBM_OK;
}

int felbm_mass_solve(felbm_state* st, const double* B, double* X, int32_t k) {
    if (!st || !B || !X || k < 1 || k > 18) {
        set_error("felbm_mass_solve: invalid argument (1 <= k <= 18)");
        return FELBM_ERR_INVALID_ARG;
    }
    cudaStream_t s = st->stream;
    const DevMesh& m = st->dm;
    const Bufs& b = st->buf;
    FELBM_CUDA(cudaMemcpyAsync(b.stage, B, sizeof(double) * k * m.N, cudaMemcpyHostToDevice, s));
    enqueue_mass_solve(st, b, b.stage, b.stage, k, s);
    FELBM_CUDA(cudaGetLastError());
    FELBM_CUDA(cudaMemcpyAsync(X, b.stage, sizeof(double) * k * m.N, cudaMemcpyDeviceToHost, s));
    FELBM_CUDA(cudaStreamSynchronize(s));
    return FELBM_OK;
}

}  // extern "C"

// ---------------------------------------- no-allocation mass solve -------
// The iterates of felbm_mass_solve_static live here, not in any allocation.
static __device__ __align__(256) unsigned char g_static_scratch[FELBM_STATIC_SCRATCH_BYTES];

namespace felbm {

static std::mutex g_static_mu;
static void* g_static_addr[64] = {};   // device address of g_static_scratch per device ordinal

// Device address of the scratch array on `device`, looked up once per device
// with that device current (the host-side symbol is not a device address).
static int static_scratch(int device, void** out) {
    if (device < 0 || device >= 64) {
        set_error("felbm_mass_solve_static: device ordinal out of range");
        return FELBM_ERR_INVALID_ARG;
    }
    std::lock_guard<std::mutex> lock(g_static_mu);
    if (!g_static_addr[device]) {
        int current = 0;
        FELBM_CUDA(cudaGetDevice(&current));
        if (current != device) FELBM_CUDA(cudaSetDevice(device));
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
        if (current != device) cudaSetDevice(current);
        if (e != cudaSuccess) return cuda_fail(e, "felbm_mass_solve_static: cudaGetSymbolAddress");
        g_static_addr[device] = p;
    }
    *out = g_static_addr[device];
    return FELBM_OK;
}

}  // namespace felbm

extern "C" {

int felbm_mass_solve_static(felbm_state* st, const double* d_B, double* d_X, int32_t k) {
    if (!st || !d_B || !d_X || k < 1 || k > 18 || d_B == d_X) {
        set_error("felbm_mass_solve_static: invalid argument (device B, X distinct; 1 <= k <= 18)");
        return FELBM_ERR_INVALID_ARG;
    }
    const DevMesh& m = st->dm;
    // the solve's buffers: 18 rows of stride Np, 256-byte aligned pieces
    Carver cv(nullptr);
    const size_t rows = 18 * (size_t)m.Np;
    cv.take<double>(rows);
    cv.take<double>(rows);
    cv.take<double>(rows);
    cv.take<float>(rows);
    cv.take<float>(rows);
    cv.take<float>(rows);
    if (cv.off > FELBM_STATIC_SCRATCH_BYTES) {
        char buf[256];
        snprintf(buf, sizeof buf,
                 "felbm_mass_solve_static: %d nodes need %zu bytes of scratch, the static array holds %u",
                 m.N, cv.off, (unsigned)FELBM_STATIC_SCRATCH_BYTES);
        set_error(buf);
        return FELBM_ERR_WORKSPACE;
    }
    void* base = nullptr;
    int rc = static_scratch(st->device, &base);
    if (rc) return rc;
    Carver sc(base);
    Bufs sb = st->buf;
    sb.rhs = sc.take<double>(rows);
    sb.x0 = sc.take<double>(rows);
    sb.x1 = sc.take<double>(rows);
    sb.x64 = sb.x0;
    sb.rho64 = sb.x1;
    sb.r32 = sc.take<float>(rows);
    sb.e0 = sc.take<float>(rows);
    sb.e1 = sc.take<float>(rows);
    cudaStream_t s = st->stream;
    enqueue_mass_solve(st, sb, d_B, d_X, k, s);
    FELBM_CUDA(cudaGetLastError());
    return FELBM_OK;
}

int felbm_batch_schedule(felbm_state* st, int32_t cta_max_nodes) {
    if (!st || cta_max_nodes < 0) {
        set_error("felbm_batch_schedule: invalid argument");
        return FELBM_ERR_INVALID_ARG;
    }
    FELBM_CUDA(cudaStreamSynchronize(st->stream));
    int rc = set_schedule(st, cta_max_nodes);
    if (rc) return rc;
    drop_graph(st);
    return FELBM_OK;
}

int felbm_solver_check(felbm_state* st, int32_t enable, double tol) {
    if (!st || (enable != 0 && enable != 1) || (enable && !(tol > 0.0))) {
        set_error("felbm_solver_check: invalid argument (enable 0 or 1, tol > 0)");
        return FELBM_ERR_INVALID_ARG;
    }
    if (enable && st->mode == FELBM_SOLVER_FP64) {
        set_error("felbm_solver_check: needs the FP32 steps of the mixed or FP32-deviation solve");
        return FELBM_ERR_UNSUPPORTED;
    }
    FELBM_CUDA(cudaStreamSynchronize(st->stream));
    FELBM_CUDA(cudaMemsetAsync(st->buf.diag_out + kSolveResSlot, 0, 2 * sizeof(double), st->stream));
    FELBM_CUDA(cudaStreamSynchronize(st->stream));
    st->check = enable != 0;
    st->check_tol = tol;
    drop_graph(st);
    return FELBM_OK;
}

int felbm_sweep_tiled(felbm_state* st, int32_t on) {
    if (!st || (on != 0 && on != 1)) {
        set_error("felbm_sweep_tiled: invalid argument (0 or 1)");
        return FELBM_ERR_INVALID_ARG;
    }
    if (on && !tiled_ok(st->hm, st->dm.ell_w)) {
        set_error("felbm_sweep_tiled: this mesh has no ELL copy, rows of more than 12 entries, or a tile "
                  "with more than 504 nodes in its first layer");
        return FELBM_ERR_UNSUPPORTED;
    }
    FELBM_CUDA(cudaStreamSynchronize(st->stream));
    st->sweep_tiled = on != 0;
    drop_graph(st);
    return FELBM_OK;
}

int felbm_sweep_parts(felbm_state* st, int32_t parts) {
    if (!st || !(parts == 1 || parts == 2 || parts == 3 || parts == 6)) {
        set_error("felbm_sweep_parts: invalid argument (1, 2, 3 or 6)");
        return FELBM_ERR_INVALID_ARG;
    }
    FELBM_CUDA(cudaStreamSynchronize(st->stream));
    st->sweep_parts = parts;
    drop_graph(st);
    return FELBM_OK;
}

}  // extern "C"



extern "C" {

static int checkpoint_copy(felbm_state* st, void* dst_v, const void* src_v, bool save);

// Mean device time of one step over `trials` steps after one warm-up step.
static int time_steps(felbm_state* st, int32_t trials, cudaEvent_t e0, cudaEvent_t e1, float* ms) {
    int rc = felbm_step(st, 1);
    if (rc) return rc;
    FELBM_CUDA(cudaEventRecord(e0, st->stream));
    if ((rc = felbm_step(st, trials)) != FELBM_OK) return rc;
    FELBM_CUDA(cudaEventRecord(e1, st->stream));
    FELBM_CUDA(cudaEventSynchronize(e1));
    FELBM_CUDA(cudaEventElapsedTime(ms, e0, e1));
    *ms /= trials;
    return FELBM_OK;
}

int felbm_autotune(felbm_state* st, int32_t trials, felbm_tune_result* out) {
    if (!st || !out || trials < 1) {
        set_error("felbm_autotune: invalid argument");
        return FELBM_ERR_INVALID_ARG;
    }
    *out = felbm_tune_result{};
    const HostMesh& h = st->hm;
    FELBM_CUDA(cudaStreamSynchronize(st->stream));
    void* save = st->buf.stage;   // the state fits the staging buffer in both precisions
    int rc = checkpoint_copy(st, save, nullptr, true);
    if (rc) return rc;
    const int64_t step0 = st->step;
    const bool timing0 = st->timing;
    st->timing = false;
    cudaEvent_t e0, e1;
    FELBM_CUDA(cudaEventCreate(&e0));
    FELBM_CUDA(cudaEventCreate(&e1));
    // 1. threads per node of the FP32 sweeps (tiled schedule)
    //    and where the iterate comes from (gathered, or staged per node tile)
    const int parts_c[4] = {1, 2, 3, 6};
    int best_parts = st->sweep_parts;
    int best_tiled = st->sweep_tiled;
    float best = 1e30f;
    if (st->mode != FELBM_SOLVER_FP64 && st->dm.ell_w > 0) {
        rc = set_schedule(st, 0);
        for (int tiled = 0; tiled < 2 && rc == FELBM_OK; ++tiled) {
            if (tiled && st->dm.blk_steps == 0) break;
            for (int k = 0; k < 4 && rc == FELBM_OK; ++k) {
                st->sweep_parts = parts_c[k];
                st->sweep_tiled = tiled;
                if (tiled && parts_c[k] != 3) continue;   // the blocked solve has one form
                drop_graph(st);
                float ms = 0.0f;
                if ((rc = time_steps(st, trials, e0, e1, &ms)) != FELBM_OK) break;
                (tiled ? out->tiled_ms : out->parts_ms)[k] = ms;
                if (ms < best) {
                    best = ms;
                    best_parts = parts_c[k];
                    best_tiled = tiled;
                }
                rc = checkpoint_copy(st, nullptr, save, false);
            }
        }
    }
    st->sweep_parts = best_parts;
    st->sweep_tiled = best_tiled;
    drop_graph(st);
    out->sweep_parts = best_parts;
    out->sweep_tiled = blocked(st, st->dm) ? 1 : 0;
    // 2. batch schedule: CTA per member up to a node threshold (FP32_DEV batches)
    int32_t best_t = 0;
    if (rc == FELBM_OK && st->dev32 && h.G > 1) {
        std::vector<int32_t> cand = {0, 1 << 11, 1 << 12, 1 << 13, 1 << 14, 1 << 15, 1 << 16, 1 << 17};
        int last_n_cta = -1;
        best = 1e30f;
        for (int32_t t : cand) {
            int32_t n_cta = 0;
            for (int32_t g = 0; g < h.G; ++g) n_cta += (t > 0 && h.grp_size[g] <= t);
            if (n_cta == last_n_cta) continue;   // same split as the previous candidate
            last_n_cta = n_cta;
            if ((rc = set_schedule(st, t)) != FELBM_OK) break;
            drop_graph(st);
            float ms = 0.0f;
            if ((rc = time_steps(st, trials, e0, e1, &ms)) != FELBM_OK) break;
            if (out->n_candidates < 16) {
                out->candidates[out->n_candidates] = t;
                out->step_ms[out->n_candidates] = ms;
                out->n_candidates++;
            }
            if (ms < best) {
                best = ms;
                best_t = t;
            }
            if ((rc = checkpoint_copy(st, nullptr, save, false)) != FELBM_OK) break;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    int rc2 = checkpoint_copy(st, nullptr, save, false);
    FELBM_CUDA(cudaStreamSynchronize(st->stream));
    st->step = step0;
    st->timing = timing0;
    if (rc) return rc;
    if (rc2) return rc2;
    out->cta_max_nodes = best_t;
    return felbm_batch_schedule(st, best_t);
}

// ------------------------------------------------------------- adjoint ----
int felbm_set_wetting(felbm_state* st, const double* phi_c, int32_t n_wall_ids) {
    if (!st || !phi_c || n_wall_ids < 1 || n_wall_ids > FELBM_MAX_WALL_IDS) {
        set_error("felbm_set_wetting: invalid argument");
        return FELBM_ERR_INVALID_ARG;
    }
    const HostMesh& h = st->hm;
    std::vector<double> wall_phi(std::max<int32_t>(h.E, 1), 0.0);
    for (int32_t e = 0; e < h.E; ++e) {
        if (h.wall_id[e] >= n_wall_ids) {
            set_error("felbm_set_wetting: a wall id has no phi_c");
            return FELBM_ERR_INVALID_ARG;
        }
        wall_phi[e] = phi_c[h.wall_id[e]];
    }
    for (int32_t k = 0; k < n_wall_ids; ++k) st->prm.phi_c[k] = phi_c[k];
    if (h.E > 0)
        FELBM_CUDA(cudaMemcpyAsync(const_cast<double*>(st->dm.wall_phi), wall_phi.data(), sizeof(double) * h.E,
                                   cudaMemcpyHostToDevice, st->stream));
    FELBM_CUDA(cudaStreamSynchronize(st->stream));
    return FELBM_OK;
}

int felbm_checkpoint_bytes(const felbm_state* st, size_t* bytes) {
    if (!st || !bytes) {
        set_error("felbm_checkpoint_bytes: invalid argument");
        return FELBM_ERR_INVALID_ARG;
    }
    *bytes = st->dev32 ? (size_t)st->dm.Np * (18 * sizeof(float) + sizeof(double) + 3 * sizeof(float))
                       : (size_t)st->dm.Np * 18 * sizeof(double);
    return FELBM_OK;
}

static int checkpoint_copy(felbm_state* st, void* dst_v, const void* src_v, bool save) {
    const DevMesh& m = st->dm;
    const Bufs& b = st->buf;
    char* ck = reinterpret_cast<char*>(save ? dst_v : const_cast<void*>(src_v));
    std::vector<std::pair<void*, size_t>> parts;
    if (st->dev32) {
        parts = {{b.dpsi, 18 * (size_t)m.Np * sizeof(float)}, {b.C, (size_t)m.Np * sizeof(double)},
                 {b.p32, (size_t)m.Np * sizeof(float)}, {b.ux32, (size_t)m.Np * sizeof(float)},
                 {b.uy32, (size_t)m.Np * sizeof(float)}};
    } else {
        parts = {{b.psi, 18 * (size_t)m.Np * sizeof(double)}};
    }
    size_t off = 0;
    for (auto& pr : parts) {
        void* d = save ? (void*)(ck + off) : pr.first;
        const void* sr = save ? (const void*)pr.first : (const void*)(ck + off);
        FELBM_CUDA(cudaMemcpyAsync(d, sr, pr.second, cudaMemcpyDeviceToDevice, st->stream));
        off += pr.second;
    }
    return FELBM_OK;
}

int felbm_checkpoint_save(felbm_state* st, void* d_dst) {
    if (!st || !d_dst) {
        set_error("felbm_checkpoint_save: invalid argument");
        return FELBM_ERR_INVALID_ARG;
    }
    return checkpoint_copy(st, d_dst, nullptr, true);
}

int felbm_checkpoint_load(felbm_state* st, const void* d_src) {
    if (!st || !d_src) {
        set_error("felbm_checkpoint_load: invalid argument");
        return FELBM_ERR_INVALID_ARG;
    }
    return checkpoint_copy(st, nullptr, d_src, false);
}

int felbm_adjoint_seed(felbm_state* st, const double* dL_dg, const double* dL_dh) {
    if (!st || !dL_dg || !dL_dh) {
        set_error("felbm_adjoint_seed: invalid argument");
        return FELBM_ERR_INVALID_ARG;
    }
    if (st->phys.lapmu_nodal) {
        set_error("felbm_adjoint_seed: the adjoint covers FELBM_LAPMU_FACE only");
        return FELBM_ERR_UNSUPPORTED;
    }
    if (st->dev32) {
        set_error("felbm_adjoint_seed: the adjoint is available for FELBM_FP64 states");
        return FELBM_ERR_UNSUPPORTED;
    }
    cudaStream_t s = st->stream;
    const int N = st->dm.N;
    FELBM_CUDA(cudaMemcpyAsync(st->buf.stage, dL_dg, sizeof(double) * 9 * N, cudaMemcpyHostToDevice, s));
    FELBM_CUDA(cudaMemcpyAsync(st->buf.stage + (size_t)9 * N, dL_dh, sizeof(double) * 9 * N, cudaMemcpyHostToDevice, s));
    k_scatter_in<<<grid_for(N, kBlock), kBlock, 0, s>>>(st->dm, st->buf.stage, st->adj.lam, 18);
    FELBM_CUDA(cudaGetLastError());
    if (st->hm.E > 0) FELBM_CUDA(cudaMemsetAsync(st->adj.dphi, 0, sizeof(double) * st->hm.E, s));
    FELBM_CUDA(cudaStreamSynchronize(s));
    return FELBM_OK;
}

int felbm_adjoint_step(felbm_state* st) {
    if (!st) {
        set_error("felbm_adjoint_step: invalid argument");
        return FELBM_ERR_INVALID_ARG;
    }
    if (st->phys.lapmu_nodal) {
        set_error("felbm_adjoint_step: the adjoint covers FELBM_LAPMU_FACE only");
        return FELBM_ERR_UNSUPPORTED;
    }
    if (st->dev32) {
        set_error("felbm_adjoint_step: the adjoint is available for FELBM_FP64 states");
        return FELBM_ERR_UNSUPPORTED;
    }
    cudaStream_t s = st->stream;
    const DevMesh& m = st->dm;
    Bufs& b = st->buf;
    AdjBufs& a = st->adj;
    const int nb = fp64_block(st, m.N, 128), tb = fp64_block(st, m.T, 128);
    const unsigned ng = grid_for(m.N, nb), tg = grid_for(m.T, tb);
    // fields of the state psi^n (the input of the step being reversed)
    k_collide<<<ng, nb, 0, s>>>(m, st->phys, b, 0);
    launch_mu(m, st->phys, b, ng, nb, s);
    k_gradmu<<<tg, tb, 0, s>>>(m, b);
    // lambda_RHS = M11^{-1} lambda with the step's solver
    if (st->mode == FELBM_SOLVER_FP64)
        k_cheb_start<false><<<ng, nb, 0, s>>>(m, b, a.lam, st->inv_theta);
    else
        k_cheb_start<true><<<ng, nb, 0, s>>>(m, b, a.lam, st->tau[0]);
    a.lamRHS = enqueue_solve(st, m, b, s, false, blocked(st, m));
    k_adj_elem_a<<<tg, tb, 0, s>>>(m, st->phys, b, a);
    k_adj_elem_b<<<tg, tb, 0, s>>>(m, a);
    k_adj_node_d<<<ng, nb, 0, s>>>(m, st->phys, a);
    k_adj_node_e<<<ng, nb, 0, s>>>(m, st->phys, b, a);
    FELBM_CUDA(cudaGetLastError());
    return FELBM_OK;
}

int felbm_adjoint_get(felbm_state* st, double* dL_dg, double* dL_dh, double* dL_dphi_c) {
    if (!st || (!dL_dg != !dL_dh)) {
        set_error("felbm_adjoint_get: invalid argument");
        return FELBM_ERR_INVALID_ARG;
    }
    if (st->phys.lapmu_nodal) {
        set_error("felbm_adjoint_get: the adjoint covers FELBM_LAPMU_FACE only");
        return FELBM_ERR_UNSUPPORTED;
    }
    if (st->dev32) {
        set_error("felbm_adjoint_get: the adjoint is available for FELBM_FP64 states");
        return FELBM_ERR_UNSUPPORTED;
    }
    cudaStream_t s = st->stream;
    const int N = st->dm.N;
    if (dL_dg) {
        k_gather_out<<<grid_for(N, kBlock), kBlock, 0, s>>>(st->dm, st->adj.lam, st->buf.stage, 18);
        FELBM_CUDA(cudaGetLastError());
        FELBM_CUDA(cudaMemcpyAsync(dL_dg, st->buf.stage, sizeof(double) * 9 * N, cudaMemcpyDeviceToHost, s));
        FELBM_CUDA(cudaMemcpyAsync(dL_dh, st->buf.stage + (size_t)9 * N, sizeof(double) * 9 * N,
                                   cudaMemcpyDeviceToHost, s));
    }
    std::vector<double> de(std::max<int32_t>(st->hm.E, 1));
    if (st->hm.E > 0)
        FELBM_CUDA(cudaMemcpyAsync(de.data(), st->adj.dphi, sizeof(double) * st->hm.E, cudaMemcpyDeviceToHost, s));
    FELBM_CUDA(cudaStreamSynchronize(s));
    if (dL_dphi_c) {
        for (int k = 0; k < st->prm.n_wall_ids; ++k) dL_dphi_c[k] = 0.0;
        for (int32_t e = 0; e < st->hm.E; ++e) dL_dphi_c[st->hm.wall_id[e]] += de[e];   // edge order: fixed
    }
    return FELBM_OK;
}

void felbm_state_destroy(felbm_state* st) {
    if (!st) return;
    drop_graph(st);
    if (st->cap_stream) cudaStreamDestroy(st->cap_stream);
    if (st->side_stream) cudaStreamDestroy(st->side_stream);
    if (st->ev_fork) cudaEventDestroy(st->ev_fork);
    if (st->ev_copied) cudaEventDestroy(st->ev_copied);
    if (st->ev_join) cudaEventDestroy(st->ev_join);
    if (st->copy_stream) cudaStreamDestroy(st->copy_stream);
    for (auto& e : st->ev_in_free)
        if (e) cudaEventDestroy(e);
    for (auto& e : st->ev)
        if (e) cudaEventDestroy(e);
    delete st;
}

}  // extern "C"
