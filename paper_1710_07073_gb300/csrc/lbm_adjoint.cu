// Reverse mode of the coupled step (hand-written adjoint), with checkpointed
// recomputation.
//
// Objective: L = (ubar - target)^2, ubar the mean over bubbles and over the
// last `window` steps of the bubble rise velocity u_b,z.  Gradients: with
// respect to the drag scale s_D (Table 1 drag times s_D), each bubble's
// diameter d_b (through its volume, mass, buoyancy, drag closure and mapping
// window n = width_factor d_b), and the initial liquid velocity field u0 (with
// the initial populations f = f^eq(rho, u0), Algorithm 1 initialisation).
//
// One forward step n maps (f^n, bubble state) to (f^{n+1}, bubble state'):
//   bubble update   u_l = sum_j W_j(x^n) u(f^n)_j (Eq. 20), sub-stepped
//                   Newton update (Eq. 4, Table 1), psi = -mean F_D;
//   spreading       F(y) = sum_b W_y(x^{n+1}_b) psi_b (Eq. 21);
//   liquid          f^{n+1} = Stream(Collide(f^n, F)) (Eq. 12-16).
// The reverse step (step n, newest first):
//   k_adj_liquid    Lambda^n = C_f^T S^T Lambda^{n+1} per node (transposed
//                   streaming with bounce-back, linearised forced BGK) at
//                   every node outside the bubbles' interpolation windows;
//   k_adj_bubbles   (a CTA per bubble, on a second stream alongside
//                   k_adj_liquid: both read only Lambda^{n+1} and f^n)
//                   spreading adjoint, reverse of the sub-steps and the
//                   interpolation's adjoint with respect to the bubble;
//   k_adj_window    (after k_adj_bubbles, same stream) Lambda^n at the
//                   windows' nodes: as k_adj_liquid plus the interpolation's
//                   adjoint with respect to the liquid.
//   In all:         per bubble: spreading adjoint (Lambda_psi, Lambda_x^{n+1},
//                   Lambda_n from the force adjoint at the window nodes),
//                   reverse of the sub-steps, interpolation adjoint (adds to
//                   Lambda^n at the window nodes, Lambda_x^n, Lambda_n).
// Liquid adjoints are FP32 (like the forward sweep); the bubble adjoint and
// the accumulated parameter gradients are FP64.
#include <cmath>
#include <vector>

#include "lbm_ctx.hpp"
#include "lbm_device.cuh"

using namespace lbm;

namespace {

constexpr int ADJ_MAX_BUBBLES = 256;
constexpr int ADJ_THREADS = 256;   // worker threads of k_adj_bubbles
constexpr int ADJ_MAX_SUB = 64;

// Bubble state snapshot: before a step (x, u, q = u_l history, h, active) and
// after it (ul = u_l of the step, psi, x', u', rec = spreading record).
struct BubbleSnap {
    double x[3], u[3], q[3], ul[3], psi[3];
    float xh[3], xl[3];   // the centre as stored (x = xh + xl), for an exact restore
    int h, active;
    int lo[3], cnt[3];    // before a step: the interpolation window's cells
    BubbleRec rec;
};

// Per-bubble adjoint state carried between reverse steps.
struct BubbleAdj {
    double lx[3], lu[3], lq[3];
};

// Closure constants in FP64 together with their d-derivatives (Table 1, Eq. 3).
struct AdjConst {
    double nu, dt_b, dt_l, sn_coeff, sn_exp, width_factor, drag_scale;
    double rho_l, rho_b, g, sigma, c_am;
    int substeps, two_way;
};

__global__ void k_restore(BubbleDev B, const BubbleSnap* in) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B.nb) return;
    const BubbleSnap& s = in[b];
    for (int a = 0; a < 3; ++a) {
        B.xh[3 * b + a] = s.xh[a];
        B.xl[3 * b + a] = s.xl[a];
        B.u[3 * b + a] = (float)s.u[a];
        B.ulprev[3 * b + a] = (float)s.q[a];
    }
    B.has_prev[b] = s.h;
    B.active[b] = s.active;
}

__global__ void k_record_uz(BubbleDev B, double* uz) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < B.nb) uz[b] = B.u[3 * b + 2];
}

// ubar over the last `window` steps; out = {ubar, loss}.
__global__ void k_adj_loss(const double* uz, int nsteps, int nb, int window, double target,
                           double* out) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    double s = 0.0;
    for (int n = nsteps - window; n < nsteps; ++n)
        for (int b = 0; b < nb; ++b) s += uz[(size_t)n * nb + b];
    const double ubar = s / ((double)window * nb);
    out[0] = ubar;
    out[1] = (ubar - target) * (ubar - target);
}

// ---- mapping weights and their derivatives, normalised units --------------
// z(t) = t^4 - 2 t^2 + 1 on [-1, 1] (Eq. 18 without 15/(16 n)); the cell
// integral of Z is 15/16 of the integral of z over the clipped cell.
__device__ __forceinline__ float zpoly(float t) {
    const float t2 = t * t;
    return (t2 - 2.0f) * t2 + 1.0f;
}

// Integral of z over [a, b] (clipped to [-1, 1]) and its derivatives with
// respect to the bubble coordinate x and the half-width n, for the cell
// [s0, s0 + 1] relative to the bubble (a = s0/n, b = (s0+1)/n).
struct AxisW {
    float w, dx, dn;
};

__device__ __forceinline__ AxisW axis_weight(float s0, float s1, float inv_n) {
    const float a = fmaxf(s0 * inv_n, -1.0f), b = fminf(s1 * inv_n, 1.0f);
    AxisW r{0.0f, 0.0f, 0.0f};
    if (!(b > a)) return r;
    const float a2 = a * a, b2 = b * b, ab = a * b;
    const float p4 = b2 * b2 + b2 * ab + ab * ab + ab * a2 + a2 * a2;
    r.w = (b - a) * (p4 * 0.2f - (b2 + ab + a2) * (2.0f / 3.0f) + 1.0f);
    const float za = zpoly(a), zb = zpoly(b);
    r.dx = -inv_n * (zb - za);                 // d/dx, s = i - x
    r.dn = -inv_n * (b * zb - a * za);         // d/dn
    return r;
}

// Per-axis normalisation over the in-box part of the window (walls) and its
// derivatives; 16/15 and zero derivatives on a periodic axis.
__device__ __forceinline__ AxisW axis_norm_d(double x, int L, float inv_n, bool periodic) {
    if (periodic) return AxisW{16.0f / 15.0f, 0.0f, 0.0f};
    return axis_weight((float)(-x), (float)((double)L - x), inv_n);
}

// The cells of a window at centre x, half-width n, per axis.
__device__ __forceinline__ void window_cells(const Geo& g, const double* x, double n, int lo[3],
                                             int cnt[3]) {
    const int L[3] = {g.nx, g.ny, g.nz};
    for (int a = 0; a < 3; ++a) {
        const bool periodic = !(g.walls & (1u << (2 * a)));
        int l = (int)floor(x[a] - n);
        int h = (int)ceil(x[a] + n) - 1;
        if (!periodic) {
            l = max(l, 0);
            h = min(h, L[a] - 1);
        }
        lo[a] = l;
        cnt[a] = min(max(h - l + 1, 0), 2 * (int)MAX_HALF_WIDTH + 2);
    }
}

// Window of one bubble: its cells, the centre as stored (two floats), 1/n, the
// reciprocal of the normalisation and, per axis, its derivative over itself
// with respect to the centre (rx) and, summed, to n (rn).
struct Window {
    int lo[3], cnt[3];
    float xh[3], xl[3];
    float inv_n, inv_norm, rx[3], rn;
    bool inner;   // no node has a neighbour beyond a face
};

__device__ __forceinline__ void make_window(const Geo& g, const double* x, const float* xh,
                                            const float* xl, double n, Window& w) {
    const int L[3] = {g.nx, g.ny, g.nz};
    window_cells(g, x, n, w.lo, w.cnt);
    w.inv_n = (float)(1.0 / n);
    float nrm = 1.0f;
    w.rn = 0.0f;
    w.inner = true;
    for (int a = 0; a < 3; ++a) {
        w.xh[a] = xh[a];
        w.xl[a] = xl[a];
        const AxisW q = axis_norm_d(x[a], L[a], w.inv_n, !(g.walls & (1u << (2 * a))));
        nrm *= q.w;
        w.rx[a] = q.dx / q.w;
        w.rn += q.dn / q.w;
        w.inner = w.inner && w.lo[a] >= 1 && w.lo[a] + w.cnt[a] < L[a];
    }
    w.inv_norm = 1.0f / nrm;
}

// The left end of cell c relative to the centre on axis a.
__device__ __forceinline__ float cell_left(const Window& w, int a, int c) {
    return ((float)c - w.xh[a]) - w.xl[a];
}

__device__ __forceinline__ int wrap1(int c, int L) { return c < 0 ? c + L : (c >= L ? c - L : c); }

__global__ void k_snapshot(Geo g, BubbleDev B, BubbleSnap* out, int post) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B.nb) return;
    BubbleSnap& s = out[b];
    for (int a = 0; a < 3; ++a) {
        s.xh[a] = B.xh[3 * b + a];
        s.xl[a] = B.xl[3 * b + a];
        s.x[a] = join_f2(s.xh[a], s.xl[a]);
        s.u[a] = B.u[3 * b + a];
        if (post) {
            s.ul[a] = B.ul[3 * b + a];
            s.psi[a] = B.psi[3 * b + a];
        } else {
            s.q[a] = B.ulprev[3 * b + a];
        }
    }
    if (post) {
        s.rec = B.rec[b];
        s.active = B.spread[b];   // 1 if it took part in the step
    } else {
        s.h = B.has_prev[b];
        s.active = B.active[b];
        window_cells(g, s.x, B.n[b], s.lo, s.cnt);
    }
}

// Weight W of window node m and its derivatives dW/dx (3) and dW/dn; the
// node's wrapped lattice coordinates in (i, j, k).
__device__ __forceinline__ float window_node(const Geo& g, const Window& w, int m, float dWdx[3],
                                             float& dWdn, int& i, int& j, int& k) {
    const int rest = m / w.cnt[0], iz = rest / w.cnt[1];
    const int c[3] = {w.lo[0] + m - rest * w.cnt[0], w.lo[1] + rest - iz * w.cnt[1], w.lo[2] + iz};
    AxisW ax[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float s0 = cell_left(w, a, c[a]);
        ax[a] = axis_weight(s0, s0 + 1.0f, w.inv_n);
    }
    const float W = ax[0].w * ax[1].w * ax[2].w * w.inv_norm;
    dWdn = -W * w.rn;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float others = ax[(a + 1) % 3].w * ax[(a + 2) % 3].w * w.inv_norm;
        dWdx[a] = ax[a].dx * others - W * w.rx[a];
        dWdn = fmaf(ax[a].dn, others, dWdn);
    }
    i = wrap1(c[0], g.nx);
    j = wrap1(c[1], g.ny);
    k = wrap1(c[2], g.nz);
    return W;
}

// Whether node (i, j, k) lies in a bubble's window, and its weight W there
// (window_node's).
__device__ __forceinline__ bool in_window(const Geo& g, const int lo[3], const int cnt[3], int i,
                                          int j, int k) {
    const int c[3] = {i, j, k}, L[3] = {g.nx, g.ny, g.nz};
    bool in = true;
#pragma unroll
    for (int a = 2; a >= 0; --a) in = in && wrap1(c[a] - lo[a], L[a]) < cnt[a];
    return in;
}

__device__ __forceinline__ float window_weight(const Geo& g, const Window& w, int i, int j,
                                               int k) {
    const int c[3] = {i, j, k}, L[3] = {g.nx, g.ny, g.nz};
    float v[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float s0 = cell_left(w, a, w.lo[a] + wrap1(c[a] - w.lo[a], L[a]));
        v[a] = axis_weight(s0, s0 + 1.0f, w.inv_n).w;
    }
    return v[0] * v[1] * v[2] * w.inv_norm;
}

__device__ __forceinline__ int node_index(const Geo& g, int i, int j, int k) {
    return (k * g.ny + j) * g.nx + i;
}

// Adjoint of the post-collision values gathered back through streaming:
// a_j(y) = Lambda^{n+1} at the node and direction that out_j(y) streams to.
// Element offset of the adjoint of population J leaving node (x,y,z): plane J
// at x + c_J, or, when that link crosses a wall, plane opp(J) at the node
// itself (the adjoint of half-way bounce-back); periodic axes wrap.  Written
// with selects so that a gather issues all 19 loads before using any.
template <int J>
__device__ __forceinline__ unsigned push_offset(const Geo& g, int x, int y, int z) {
    int tx = x + cx(J), ty = y + cy(J), tz = z + cz(J);
    bool bounce = false;
    if (cx(J) != 0) {
        const bool out = (unsigned)tx >= (unsigned)g.nx;
        bounce = bounce || (out && (g.walls & 0x01));
        tx = out ? (tx < 0 ? tx + g.nx : tx - g.nx) : tx;
    }
    if (cy(J) != 0) {
        const bool out = (unsigned)ty >= (unsigned)g.ny;
        bounce = bounce || (out && (g.walls & 0x04));
        ty = out ? (ty < 0 ? ty + g.ny : ty - g.ny) : ty;
    }
    if (cz(J) != 0) {
        const bool out = (unsigned)tz >= (unsigned)g.nz;
        bounce = bounce || (out && (g.walls & 0x10));
        tz = out ? (tz < 0 ? tz + g.nz : tz - g.nz) : tz;
    }
    const unsigned S = (unsigned)g.S;
    return bounce ? (unsigned)opp(J) * S + (unsigned)node_index(g, x, y, z)
                  : (unsigned)J * S + (unsigned)node_index(g, tx, ty, tz);
}

__device__ __forceinline__ void gather_push(const float* __restrict__ lam, const Geo& g, int x,
                                            int y, int z, float a[Q]) {
    unsigned o[Q];
#define LBM_PO(J) o[J] = push_offset<J>(g, x, y, z)
    LBM_PO(0); LBM_PO(1); LBM_PO(2); LBM_PO(3); LBM_PO(4); LBM_PO(5); LBM_PO(6);
    LBM_PO(7); LBM_PO(8); LBM_PO(9); LBM_PO(10); LBM_PO(11); LBM_PO(12); LBM_PO(13);
    LBM_PO(14); LBM_PO(15); LBM_PO(16); LBM_PO(17); LBM_PO(18);
#undef LBM_PO
#pragma unroll
    for (int j = 0; j < Q; ++j) a[j] = __ldg(lam + o[j]);
}

// Force at a node from all spreading records of the step (Eq. 21).
__device__ __forceinline__ void force_at(const Geo& g, const BubbleRec* recs, const int* spread,
                                         int nb, int x, int y, int z, float F[3]) {
    F[0] = F[1] = F[2] = 0.0f;
    for (int b = 0; b < nb; ++b) {
        if (!spread[b]) continue;
        const BubbleRec& r = recs[b];
        float rr[3] = {(float)(x - r.ax) + 0.5f - r.fx, (float)(y - r.ay) + 0.5f - r.fy,
                       (float)(z - r.az) + 0.5f - r.fz};
        const int L[3] = {g.nx, g.ny, g.nz};
        bool outside = false;
        for (int a = 0; a < 3; ++a) {
            if (!(g.walls & (1u << (2 * a)))) {
                if (rr[a] > 0.5f * L[a]) rr[a] -= (float)L[a];
                else if (rr[a] < -0.5f * L[a]) rr[a] += (float)L[a];
            }
            // cell_poly is zero once the cell [s - h, s + h] is outside [-1, 1]
            outside = outside || fabsf(rr[a] * r.inv_n) >= 1.0f + r.h;
        }
        if (outside) continue;
        float w = 1.0f;
        for (int a = 0; a < 3; ++a) w *= cell_poly(rr[a] * r.inv_n, r.h);
        F[0] = fmaf(w, r.px, F[0]);
        F[1] = fmaf(w, r.py, F[1]);
        F[2] = fmaf(w, r.pz, F[2]);
    }
}

// Bare Eq. 10 velocity and 1 / rho of shifted populations.
__device__ __forceinline__ void node_moments(const float gv[Q], float rho0, float u[3],
                                             float& inv_rho) {
    float drho = 0.0f, m[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        drho += gv[q];
        m[0] += (float)cx(q) * gv[q];
        m[1] += (float)cy(q) * gv[q];
        m[2] += (float)cz(q) * gv[q];
    }
    inv_rho = 1.0f / (rho0 + drho);
    for (int d = 0; d < 3; ++d) u[d] = m[d] * inv_rho;
}

// Linearised forced BGK at one node, transposed.  g: shifted pre-collision
// populations; a: adjoint of the post-collision values.  Returns the adjoint
// of the pre-collision populations in lam and of the force in lamF.
//   rho = rho0 + sum g, u = (sum c g + F/2) / rho
//   out_j = (1 - w) f_j + w f^eq_j(rho, u) + G_j(u, F)
//   dL/df_k = (1 - w) a_k + A_rho + A_u . (c_k - u) / rho
//   A_rho = w sum_j a_j w_j (1 + 3 cu + 9/2 cu^2 - 3/2 u^2)
//   A_u   = sum_j a_j [w w_j rho (3 c_j + 9 cu_j c_j - 3 u) + pref w_j (9 cF_j c_j - 3 F)]
//   dL/dF = A_u / (2 rho) + sum_j a_j pref w_j (3 (c_j - u) + 9 cu_j c_j)
__device__ __forceinline__ void collide_adjoint(const float g[Q], const float F[3], float rho0,
                                                float omega, float pref, const float a[Q],
                                                float lam[Q], float lamF[3]) {
    float drho = 0.0f, m[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int j = 0; j < Q; ++j) {
        drho += g[j];
        if (cx(j) != 0) m[0] += (float)cx(j) * g[j];
        if (cy(j) != 0) m[1] += (float)cy(j) * g[j];
        if (cz(j) != 0) m[2] += (float)cz(j) * g[j];
    }
    const float rho = rho0 + drho, inv_rho = 1.0f / rho;
    const float u[3] = {(m[0] + 0.5f * F[0]) * inv_rho, (m[1] + 0.5f * F[1]) * inv_rho,
                        (m[2] + 0.5f * F[2]) * inv_rho};
    const float usq = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    // With aw_j = a_j w_j, the sums over j that the adjoint needs:
    //   S0 = sum aw, S1 = sum aw c, S2 = sum aw (c.u) c, S3 = sum aw (c.F) c,
    //   Su = sum aw (c.u), Su2 = sum aw (c.u)^2.
    float S0 = 0.0f, Su = 0.0f, Su2 = 0.0f;
    float S1[3] = {0.0f, 0.0f, 0.0f}, S2[3] = {0.0f, 0.0f, 0.0f}, S3[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int j = 0; j < Q; ++j) {
        const int c[3] = {cx(j), cy(j), cz(j)};
        float cu = 0.0f, cF = 0.0f;
#pragma unroll
        for (int d = 0; d < 3; ++d)
            if (c[d] != 0) {
                cu += (float)c[d] * u[d];
                cF += (float)c[d] * F[d];
            }
        const float aw = a[j] * wf(j), awcu = aw * cu, awcF = aw * cF;
        S0 += aw;
        Su += awcu;
        Su2 = fmaf(awcu, cu, Su2);
#pragma unroll
        for (int d = 0; d < 3; ++d)
            if (c[d] != 0) {
                S1[d] += (float)c[d] * aw;
                S2[d] += (float)c[d] * awcu;
                S3[d] += (float)c[d] * awcF;
            }
    }
    // The density and velocity adjoints of the forced equilibrium (Eq. 6, 14,
    // 15): sum_j aw_j times the derivatives of f^eq_j and of the Guo term.
    const float A_rho = omega * (S0 * (1.0f - 1.5f * usq) + 3.0f * Su + 4.5f * Su2);
    float Au[3], base = A_rho;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const float A_u = omega * rho * (3.0f * S1[d] + 9.0f * S2[d] - 3.0f * u[d] * S0) +
                          pref * (9.0f * S3[d] - 3.0f * F[d] * S0);
        const float G_F = pref * (3.0f * S1[d] - 3.0f * u[d] * S0 + 9.0f * S2[d]);
        Au[d] = A_u * inv_rho;
        base -= u[d] * Au[d];
        lamF[d] = 0.5f * Au[d] + G_F;
    }
    // lam_k = (1 - omega) a_k + A_rho + (c_k - u) . A_u / rho
#pragma unroll
    for (int k = 0; k < Q; ++k) {
        float cA = base;
        if (cx(k) != 0) cA += (float)cx(k) * Au[0];
        if (cy(k) != 0) cA += (float)cy(k) * Au[1];
        if (cz(k) != 0) cA += (float)cz(k) * Au[2];
        lam[k] = (1.0f - omega) * a[k] + cA;
    }
}

// ---- two nodes per thread (even nx) -----------------------------------------
// Lambda^{n+1} of direction J at the places a row's pair (x0, x0 + 1) streams
// to: the row at (y, z) + c_J shifted against c_x, one aligned 2-wide load and,
// for the population leaving the pair, one scalar load; a row that bounces off
// a y or z wall takes the opposite plane of its own nodes.
template <int J>
__device__ __forceinline__ float2 push_pair(const float* __restrict__ lam, const Geo& g, int x0,
                                            int y, int z) {
    int ty = y + cy(J), tz = z + cz(J);
    bool bounce = false;
    if (cy(J) != 0) {
        const bool out = (unsigned)ty >= (unsigned)g.ny;
        bounce = out && (g.walls & 0x04);
        ty = out ? (ty < 0 ? ty + g.ny : ty - g.ny) : ty;
    }
    if (cz(J) != 0) {
        const bool out = (unsigned)tz >= (unsigned)g.nz;
        bounce = bounce || (out && (g.walls & 0x10));
        tz = out ? (tz < 0 ? tz + g.nz : tz - g.nz) : tz;
    }
    const unsigned S = (unsigned)g.S, nx = (unsigned)g.nx;
    const unsigned own = (unsigned)opp(J) * S + (unsigned)node_index(g, x0, y, z);
    const unsigned row = bounce ? own : (unsigned)J * S + (unsigned)node_index(g, x0, ty, tz);
    const float2 P = __ldg(reinterpret_cast<const float2*>(lam + row));
    if (cx(J) == 0) return P;
    const bool wallx = (g.walls & 0x01) != 0;
    unsigned e;
    if (cx(J) == 1) {   // node x0 sends to x0 + 1, node x0 + 1 to x0 + 2
        e = row + 2u;
        if ((unsigned)x0 + 2u >= nx) e = wallx ? own + 1u : row - (unsigned)x0;
    } else {            // node x0 sends to x0 - 1, node x0 + 1 to x0
        e = row - 1u;
        if (x0 == 0) e = wallx ? own : row + nx - 1u;
    }
    if (bounce) return P;
    const float v = __ldg(lam + e);
    return cx(J) == 1 ? make_float2(P.y, v) : make_float2(v, P.x);
}

// collide_adjoint without the force's adjoint on a pair of nodes, by sums s
// and differences d of opposite directions: S1 = sum aw c from the d, the
// second moments M = sum aw c c from the s, S2 = M u, S3 = M F, Su = S1 . u,
// Su2 = u . S2.
template <class Put>
__device__ __forceinline__ void collide_adjoint_pair(float2 drho, float2 jx, float2 jy, float2 jz,
                                                     const float2 F[3], float rho0, float omega,
                                                     float pref, const float2 a[Q], Put put) {
    const float2 rho = add2(f2(rho0), drho);
    const float2 inv_rho = make_float2(1.0f / rho.x, 1.0f / rho.y);
    const float2 u[3] = {mul2(fma2(f2(0.5f), F[0], jx), inv_rho),
                         mul2(fma2(f2(0.5f), F[1], jy), inv_rho),
                         mul2(fma2(f2(0.5f), F[2], jz), inv_rho)};
    const float2 usq = fma2(u[0], u[0], fma2(u[1], u[1], mul2(u[2], u[2])));
    float2 s[9], d[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        s[k] = add2(a[2 * k + 1], a[2 * k + 2]);
        d[k] = sub2(a[2 * k + 1], a[2 * k + 2]);
    }
    // Pairs: 0 x, 1 y, 2 z, 3 (1,1,0), 4 (1,-1,0), 5 (1,0,1), 6 (1,0,-1),
    // 7 (0,1,1), 8 (0,1,-1).
    const float2 wa = f2(wf(1)), we = f2(wf(7));
    const float2 exy = add2(s[3], s[4]), exz = add2(s[5], s[6]), eyz = add2(s[7], s[8]);
    const float2 S0 = fma2(f2(wf(0)), a[0],
                           fma2(wa, add2(add2(s[0], s[1]), s[2]), mul2(we, add2(add2(exy, exz), eyz))));
    const float2 S1[3] = {
        fma2(wa, d[0], mul2(we, add2(add2(d[3], d[4]), add2(d[5], d[6])))),
        fma2(wa, d[1], mul2(we, add2(sub2(d[3], d[4]), add2(d[7], d[8])))),
        fma2(wa, d[2], mul2(we, add2(sub2(d[5], d[6]), sub2(d[7], d[8]))))};
    const float2 Mxx = fma2(wa, s[0], mul2(we, add2(exy, exz)));
    const float2 Myy = fma2(wa, s[1], mul2(we, add2(exy, eyz)));
    const float2 Mzz = fma2(wa, s[2], mul2(we, add2(exz, eyz)));
    const float2 Mxy = mul2(we, sub2(s[3], s[4])), Mxz = mul2(we, sub2(s[5], s[6])),
                 Myz = mul2(we, sub2(s[7], s[8]));
    const float2 S2[3] = {fma2(Mxx, u[0], fma2(Mxy, u[1], mul2(Mxz, u[2]))),
                          fma2(Mxy, u[0], fma2(Myy, u[1], mul2(Myz, u[2]))),
                          fma2(Mxz, u[0], fma2(Myz, u[1], mul2(Mzz, u[2])))};
    const float2 S3[3] = {fma2(Mxx, F[0], fma2(Mxy, F[1], mul2(Mxz, F[2]))),
                          fma2(Mxy, F[0], fma2(Myy, F[1], mul2(Myz, F[2]))),
                          fma2(Mxz, F[0], fma2(Myz, F[1], mul2(Mzz, F[2])))};
    const float2 Su = fma2(S1[0], u[0], fma2(S1[1], u[1], mul2(S1[2], u[2])));
    const float2 Su2 = fma2(S2[0], u[0], fma2(S2[1], u[1], mul2(S2[2], u[2])));
    const float2 A_rho = mul2(f2(omega), fma2(S0, fma2(f2(-1.5f), usq, f2(1.0f)),
                                              fma2(f2(3.0f), Su, mul2(f2(4.5f), Su2))));
    const float2 wr = mul2(f2(omega), rho);
    float2 Au[3], base = A_rho;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float2 eq = fma2(f2(9.0f), S2[k], mul2(f2(3.0f), sub2(S1[k], mul2(u[k], S0))));
        const float2 guo = fma2(f2(9.0f), S3[k], mul2(f2(-3.0f), mul2(F[k], S0)));
        Au[k] = mul2(fma2(wr, eq, mul2(f2(pref), guo)), inv_rho);
        base = sub2(base, mul2(u[k], Au[k]));
    }
    // lam_k = (1 - omega) a_k + A_rho + (c_k - u) . A_u / rho
    const float2 om1 = f2(1.0f - omega);
    put(0, fma2(om1, a[0], base));
    const float2 cA[9] = {Au[0], Au[1], Au[2], add2(Au[0], Au[1]), sub2(Au[0], Au[1]),
                          add2(Au[0], Au[2]), sub2(Au[0], Au[2]), add2(Au[1], Au[2]),
                          sub2(Au[1], Au[2])};
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        put(2 * k + 1, fma2(om1, a[2 * k + 1], add2(base, cA[k])));
        put(2 * k + 2, fma2(om1, a[2 * k + 2], sub2(base, cA[k])));
    }
}

// What the per-node kernels need of the bubbles, in dynamic shared memory sized
// by their number (256 of them would hold back the CTAs of one): the spreading
// records, which bubbles spread, and the interpolation windows.
struct AdjBox {
    int lo[3], cnt[3];   // cnt = 0: not active
};

struct AdjView {
    static_assert(alignof(BubbleRec) == 16 && sizeof(BubbleRec) % alignof(AdjBox) == 0 &&
                  sizeof(AdjBox) % sizeof(int) == 0, "the shared buffer's declared alignment");
    BubbleRec* rec;
    AdjBox* box;
    int* spread;
    int nb;
    __device__ __forceinline__ AdjView(unsigned char* s, int n)
        : rec(reinterpret_cast<BubbleRec*>(s)), box(reinterpret_cast<AdjBox*>(rec + n)),
          spread(reinterpret_cast<int*>(box + n)), nb(n) {}
    __device__ __forceinline__ void load(const BubbleSnap* pre, const BubbleSnap* post,
                                         int two_way) {
        for (int b = threadIdx.x; b < nb; b += blockDim.x) {
            rec[b] = post[b].rec;
            spread[b] = two_way ? post[b].active : 0;
            for (int a = 0; a < 3; ++a) {
                box[b].lo[a] = pre[b].lo[a];
                box[b].cnt[a] = pre[b].active ? pre[b].cnt[a] : 0;
            }
        }
        __syncthreads();
    }
    static size_t bytes(int nb) { return (sizeof(BubbleRec) + sizeof(AdjBox) + sizeof(int)) * (size_t)nb; }
};

// Lambda^{n+1} at the places a node's populations stream to, for a node none of
// whose neighbours lies beyond a face.
__device__ __forceinline__ void gather_push_inner(const float* __restrict__ lam, const Geo& g,
                                                  int x, int y, int z, float a[Q]) {
    const unsigned S = (unsigned)g.S, nx = (unsigned)g.nx, nxy = nx * (unsigned)g.ny;
    const unsigned site = (unsigned)node_index(g, x, y, z);
#define LBM_PI(J)                                                                               \
    a[J] = __ldg(lam + ((unsigned)J * S + site + ((unsigned)cx(J) + (unsigned)cy(J) * nx +      \
                                                  (unsigned)cz(J) * nxy)))
    LBM_PI(0); LBM_PI(1); LBM_PI(2); LBM_PI(3); LBM_PI(4); LBM_PI(5); LBM_PI(6); LBM_PI(7);
    LBM_PI(8); LBM_PI(9); LBM_PI(10); LBM_PI(11); LBM_PI(12); LBM_PI(13); LBM_PI(14);
    LBM_PI(15); LBM_PI(16); LBM_PI(17); LBM_PI(18);
#undef LBM_PI
}

// One node of the reverse step: Lambda^n (out), the force's adjoint, and the
// bare Eq. 10 velocity with 1 / rho (the interpolation's adjoint).
__device__ __forceinline__ void adjoint_at(const float* __restrict__ fn,
                                           const float* __restrict__ lam_next, const Geo& g,
                                           const CollideParams& cp, const BubbleRec* recs,
                                           const int* spread, int nb, int x, int y, int z,
                                           bool inner, float out[Q], float lamF[3], float u[3],
                                           float& inv_rho) {
    float gv[Q], a[Q], F[3];
    if (inner) {
        gather_issue_inner<0>(fn, g, x, y, z, gv);   // FP32 storage: the values themselves
        gather_push_inner(lam_next, g, x, y, z, a);
    } else {
        gather<0>(fn, g, cp, x, y, z, gv);
        gather_push(lam_next, g, x, y, z, a);
    }
    force_at(g, recs, spread, nb, x, y, z, F);
    collide_adjoint(gv, F, cp.rho0, cp.omega, cp.pref, a, out, lamF);
    node_moments(gv, cp.rho0, u, inv_rho);
}

#ifndef LBM_ADJ_MINB
#define LBM_ADJ_MINB 4
#endif
// Lambda^n = C_f^T S^T Lambda^{n+1} at every node outside the bubbles'
// interpolation windows, whose nodes k_adj_window writes.
//
// Bound by HBM (228 B per node: f^n and Lambda^{n+1} read, Lambda^n written).
// A node per thread was bound by issue (0.172 ms on 128 x 128 x 256, 82 % of
// the copy peak, 1,200 warp instructions per 32 nodes); on even rows a thread
// takes an x-pair with 2-wide loads and packed arithmetic: 0.157 ms at 4 CTAs
// per SM (124 registers; 5 and 6 spill and lose).
__global__ void __launch_bounds__(128, LBM_ADJ_MINB)
k_adj_liquid_pair(const float* __restrict__ fn, const float* __restrict__ lam_next,
                  float* __restrict__ lam, Geo g, CollideParams cp,
                  const BubbleSnap* __restrict__ pre, const BubbleSnap* __restrict__ post, int nb,
                  int two_way) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    AdjView sh(s_dyn, nb);
    sh.load(pre, post, two_way);
    const unsigned half = (unsigned)g.nx / 2u;
    const unsigned p = blockIdx.x * blockDim.x + threadIdx.x;   // 19 S < 2^32
    if (p >= (unsigned)g.S / 2u) return;
    const unsigned xy = p / half;
    const int x0 = 2 * (int)(p - xy * half), y = (int)(xy % (unsigned)g.ny),
              z = (int)(xy / (unsigned)g.ny);
    float2 rv[Q], a[Q];
    gather_pair<0>(fn, g, x0, y, z, rv);
#define LBM_PP(J) a[J] = push_pair<J>(lam_next, g, x0, y, z)
    LBM_PP(0); LBM_PP(1); LBM_PP(2); LBM_PP(3); LBM_PP(4); LBM_PP(5); LBM_PP(6); LBM_PP(7);
    LBM_PP(8); LBM_PP(9); LBM_PP(10); LBM_PP(11); LBM_PP(12); LBM_PP(13); LBM_PP(14);
    LBM_PP(15); LBM_PP(16); LBM_PP(17); LBM_PP(18);
#undef LBM_PP
    float Fa[3], Fb[3];
    force_at(g, sh.rec, sh.spread, nb, x0, y, z, Fa);
    force_at(g, sh.rec, sh.spread, nb, x0 + 1, y, z, Fb);
    bool skip_a = false, skip_b = false;
    for (int b = 0; b < nb; ++b) {
        skip_a = skip_a || in_window(g, sh.box[b].lo, sh.box[b].cnt, x0, y, z);
        skip_b = skip_b || in_window(g, sh.box[b].lo, sh.box[b].cnt, x0 + 1, y, z);
    }
    const float2 F[3] = {make_float2(Fa[0], Fb[0]), make_float2(Fa[1], Fb[1]),
                         make_float2(Fa[2], Fb[2])};
    float2 drho, jx, jy, jz;
    pair_moments<0>(rv, cp, drho, jx, jy, jz);
    const unsigned S = (unsigned)g.S, site0 = (unsigned)node_index(g, x0, y, z);
    collide_adjoint_pair(drho, jx, jy, jz, F, cp.rho0, cp.omega, cp.pref, a,
                         [&](int j, float2 v) {
                             float* const at = lam + ((unsigned)j * S + site0);
                             if (!skip_a && !skip_b) *reinterpret_cast<float2*>(at) = v;
                             else if (!skip_a) at[0] = v.x;
                             else if (!skip_b) at[1] = v.y;
                         });
}

// The same, a node per thread (odd rows).
__global__ void __launch_bounds__(128)
k_adj_liquid(const float* __restrict__ fn, const float* __restrict__ lam_next,
             float* __restrict__ lam, Geo g, CollideParams cp, const BubbleSnap* __restrict__ pre,
             const BubbleSnap* __restrict__ post, int nb, int two_way) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    AdjView sh(s_dyn, nb);
    sh.load(pre, post, two_way);
    const unsigned s = blockIdx.x * blockDim.x + threadIdx.x;   // 19 S < 2^32
    if (s >= (unsigned)g.S) return;
    const unsigned xy = s / (unsigned)g.nx;
    const int x = (int)(s - xy * (unsigned)g.nx), y = (int)(xy % (unsigned)g.ny),
              z = (int)(xy / (unsigned)g.ny);
    for (int b = 0; b < nb; ++b)
        if (in_window(g, sh.box[b].lo, sh.box[b].cnt, x, y, z)) return;
    float out[Q], lamF[3], u[3], inv_rho;
    adjoint_at(fn, lam_next, g, cp, sh.rec, sh.spread, nb, x, y, z, false, out, lamF, u, inv_rho);
#pragma unroll
    for (int j = 0; j < Q; ++j) lam[(size_t)j * g.S + s] = out[j];
}

// One replayed sub-step (FP32, like the forward): slip v = u - u_l, |v|, Re,
// C_D |v|, the drag, Re^sn_exp and 1/|v|.
struct SubRec {
    float v[3], s, re, cdv, fd[3];
    float pw;        // Re^sn_exp
    float inv_s;     // 1 / |v| (0 at rest)
    int branch;      // 0: 8/3 Eo/(Eo+4) |v|, 1: 24 nu/d (1 + a Re^e), 2: 48 nu/d
    int xclamp[3], uclamp[3];
};

// The bubble part of one reverse step, a CTA per bubble (blockIdx.x).  It reads
// f^n, Lambda^{n+1} and the step's snapshots only, so it runs alongside
// k_adj_liquid; each CTA writes its own bubble's adjoint state, diameter
// gradient, drag-scale gradient part and interpolation seed lul_out.
//
// Bound by latency (one CTA's chain of dependent loads and FP64 arithmetic), and
// in a small column it is the reverse step.  So what does not wait for
// something runs at once: the worker warps sum the spreading adjoint over the
// window at x^{n+1} and the interpolation's velocity moments over the window
// at x^n, while the last warp forms the closure constants and replays the
// sub-steps, an axis per lane; then that warp adds up the workers' sums, a
// value per lane, and runs the sub-steps in reverse.  With the windows' nodes
// beside the sweep too, a reverse step of one bubble went from 0.252 to 0.157 ms
// on 128 x 128 x 256 (the sweep's own time) and from 0.080 to 0.041 ms on 32 x
// 32 x 64.
constexpr int ADJ_WORKERS = ADJ_THREADS;
constexpr int ADJ_BUBBLE_THREADS = ADJ_WORKERS + 32;
// The workers' sums: the spreading adjoint of psi (3), of x (3) and of n, the
// interpolation's sum u_c dW/dx_d (9) and sum u_c dW/dn (3).
constexpr int ADJ_SUMS = 19;

__device__ __forceinline__ float lane3_sum(float v) {
    const float a = __shfl_sync(0xffffffffu, v, 0), b = __shfl_sync(0xffffffffu, v, 1),
                c = __shfl_sync(0xffffffffu, v, 2);
    return a + b + c;
}

__device__ __forceinline__ double lane3_sum(double v) {
    const double a = __shfl_sync(0xffffffffu, v, 0), b = __shfl_sync(0xffffffffu, v, 1),
                 c = __shfl_sync(0xffffffffu, v, 2);
    return a + b + c;
}

__global__ void __launch_bounds__(ADJ_BUBBLE_THREADS)
k_adj_bubbles(const float* __restrict__ fn, const float* __restrict__ lam_next, Geo g,
              CollideParams cp, const BubbleSnap* __restrict__ pre,
              const BubbleSnap* __restrict__ post, const double* __restrict__ diam, int nb,
              AdjConst ac, BubbleAdj* __restrict__ adj, double* __restrict__ grad_sD,
              double* __restrict__ grad_d, double* __restrict__ lul_out, double loss_seed) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    __shared__ double s_sum[ADJ_WORKERS / 32][ADJ_SUMS];
    __shared__ SubRec sub[ADJ_MAX_SUB];
    __shared__ Window s_win[2];   // at x^{n+1} and at x^n
    const int tid = threadIdx.x, lane = tid & 31;
    const int b = blockIdx.x;
    if (!pre[b].active) {
        // Not updated this step: its adjoint state passes through unchanged.
        if (tid == 0 && loss_seed != 0.0) adj[b].lu[2] += loss_seed;
        return;
    }
    const double d = diam[b];
    const double n = ac.width_factor * d;
    AdjView sh(s_dyn, nb);
    if (tid == 0) make_window(g, post[b].x, post[b].xh, post[b].xl, n, s_win[0]);
    if (tid == 32) make_window(g, pre[b].x, pre[b].xh, pre[b].xl, n, s_win[1]);
    sh.load(pre, post, ac.two_way);   // synchronises the CTA

    if (tid < ADJ_WORKERS) {
        double sum[ADJ_SUMS];
#pragma unroll
        for (int i = 0; i < ADJ_SUMS; ++i) sum[i] = 0.0;
        if (sh.spread[b]) {
            const Window& w = s_win[0];
            const float psi[3] = {(float)post[b].psi[0], (float)post[b].psi[1],
                                  (float)post[b].psi[2]};   // FP32 in the forward
            const int M = w.cnt[0] * w.cnt[1] * w.cnt[2];
            for (int m = tid; m < M; m += ADJ_WORKERS) {
                float dWdx[3], dWdn, out[Q], lamF[3], u[3], inv_rho;
                int i, j, k;
                const float W = window_node(g, w, m, dWdx, dWdn, i, j, k);
                adjoint_at(fn, lam_next, g, cp, sh.rec, sh.spread, nb, i, j, k, w.inner, out, lamF,
                           u, inv_rho);
                const double pl = (double)psi[0] * lamF[0] + (double)psi[1] * lamF[1] +
                                  (double)psi[2] * lamF[2];
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    sum[c] += (double)W * lamF[c];
                    sum[3 + c] += pl * dWdx[c];
                }
                sum[6] += pl * dWdn;
            }
        }
        {
            const Window& w = s_win[1];
            const int M = w.cnt[0] * w.cnt[1] * w.cnt[2];
            for (int m = tid; m < M; m += ADJ_WORKERS) {
                float dWdx[3], dWdn, gv[Q], u[3], inv_rho;
                int i, j, k;
                window_node(g, w, m, dWdx, dWdn, i, j, k);
                if (w.inner) gather_issue_inner<0>(fn, g, i, j, k, gv);
                else gather<0>(fn, g, cp, i, j, k, gv);
                node_moments(gv, cp.rho0, u, inv_rho);
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const double uc = u[c];
#pragma unroll
                    for (int e = 0; e < 3; ++e) sum[7 + 3 * c + e] += uc * dWdx[e];
                    sum[16 + c] += uc * dWdn;
                }
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int i = 0; i < ADJ_SUMS; ++i) sum[i] += __shfl_xor_sync(0xffffffffu, sum[i], o);
        if (lane == 0)
#pragma unroll
            for (int i = 0; i < ADJ_SUMS; ++i) s_sum[tid >> 5][i] = sum[i];
        __syncwarp();
        asm volatile("bar.arrive 1, %0;" ::"n"(ADJ_BUBBLE_THREADS) : "memory");
        return;
    }

    // The last warp: lane c holds axis c (the lanes beyond mirror axis 2 and
    // write nothing).  The closure constants and their d-derivatives are
    // FP64, once per step.  The sub-step replay and the per-sub-step terms of
    // its reverse run in FP32, the precision of the forward they
    // differentiate; the centre (wall clamps) and the adjoint state carried
    // between sub-steps and steps stay FP64.
    const int c = min(lane, 2);
    const bool mine = lane < 3;
    const int K = min(ac.substeps, ADJ_MAX_SUB);
    const double r = 0.5 * d, vol = M_PI * d * d * d / 6.0, dvol = 0.5 * M_PI * d * d;
    const double meff = (ac.rho_b + ac.c_am * ac.rho_l) * vol;
    const double kdt = ac.dt_b / meff, dkdt = -kdt / vol * dvol;
    const double fb = (ac.rho_l - ac.rho_b) * vol * ac.g, dfb = (ac.rho_l - ac.rho_b) * ac.g * dvol;
    const double P = 0.5 * ac.rho_l * M_PI * r * r * ac.drag_scale;
    const double dP = 0.25 * ac.rho_l * M_PI * d * ac.drag_scale;
    const double A0 = 24.0 * ac.nu / d, dA0 = -A0 / d;
    const double Bv = 48.0 * ac.nu / d, dBv = -Bv / d;
    const double Eo = (ac.rho_l - ac.rho_b) * ac.g * d * d / ac.sigma, dEo = 2.0 * Eo / d;
    const double E = 8.0 / 3.0 * Eo / (Eo + 4.0), dE = 8.0 / 3.0 * 4.0 / ((Eo + 4.0) * (Eo + 4.0)) * dEo;
    const double Cf = ac.c_am * ac.rho_l * vol / ac.dt_l, dCf = ac.c_am * ac.rho_l * dvol / ac.dt_l;
    const float kdt_f = (float)kdt, fb_f = (float)fb, P_f = (float)P, A0_f = (float)A0,
                Bv_f = (float)Bv, E_f = (float)E;
    const float sn_coeff = (float)ac.sn_coeff, sn_exp = (float)ac.sn_exp;
    const float re_per_s = (float)(d / ac.nu), nu_over_d = (float)(ac.nu / d),
                inv_nu = (float)(1.0 / ac.nu), inv_K = 1.0f / (float)K;
    const double ul = post[b].ul[c], q = pre[b].q[c];
    const int h = pre[b].h;
    const float ulf = (float)ul, fvm = h ? (float)(Cf * (ul - q)) : 0.0f;
    const float fz = c == 2 ? fb_f : 0.0f;
    const double top = (double)(c == 0 ? g.nx : (c == 1 ? g.ny : g.nz)) - r;
    const bool wall = g.walls & (1u << (2 * c));
    // forward replay
    {
        float u = (float)pre[b].u[c];
        double x = pre[b].x[c];
        for (int kk = 0; kk < K; ++kk) {
            SubRec& sr = sub[kk];
            const float v = u - ulf;
            float s2 = 0.0f;
#pragma unroll
            for (int e = 0; e < 3; ++e) {
                const float ve = __shfl_sync(0xffffffffu, v, e);
                s2 = fmaf(ve, ve, s2);
            }
            const float sp = sqrtf(s2);
            const float re = sp * re_per_s;
            const float pw = re > 0.0f ? powf(re, sn_exp) : 0.0f;
            const float A = A0_f * (1.0f + sn_coeff * pw);
            const float vis = fminf(A, Bv_f);
            const bool eo = E_f * sp >= vis;
            const float cdv = eo ? E_f * sp : vis;
            const float fd = -P_f * cdv * v;
            u = u + (fz + fd + fvm) * kdt_f;
            x = x + (double)u * ac.dt_b;
            int xclamp = 0, uclamp = 0;
            if (wall) {
                if (x < r) {
                    x = r;
                    xclamp = 1;
                    if (u < 0.0f) { u = 0.0f; uclamp = 1; }
                }
                if (x > top) {
                    x = top;
                    xclamp = 1;
                    if (u > 0.0f) { u = 0.0f; uclamp = 1; }
                }
            }
            if (mine) {
                sr.v[c] = v;
                sr.fd[c] = fd;
                sr.xclamp[c] = xclamp;
                sr.uclamp[c] = uclamp;
            }
            if (lane == 0) {
                sr.s = sp;
                sr.inv_s = sp > 0.0f ? 1.0f / sp : 0.0f;
                sr.re = re;
                sr.pw = pw;
                sr.cdv = cdv;
                sr.branch = eo ? 0 : (A <= Bv_f ? 1 : 2);
            }
        }
    }
    // The workers' sums (and, within the warp, the replay).  The workers arrive
    // and only this warp waits: a named barrier, since the two are different
    // places in the code.
    __syncwarp();
    asm volatile("bar.sync 1, %0;" ::"n"(ADJ_BUBBLE_THREADS) : "memory");
    // The sums over the workers' warps, a value per lane.
    double tot = 0.0;
    if (lane < ADJ_SUMS)
        for (int w = 0; w < ADJ_WORKERS / 32; ++w) tot += s_sum[w][lane];
    const double lpsi = __shfl_sync(0xffffffffu, tot, c), gx = __shfl_sync(0xffffffffu, tot, 3 + c),
                 gn = __shfl_sync(0xffffffffu, tot, 6);
    // reverse
    const float lpsi_f = (float)lpsi;
    double lx = adj[b].lx[c] + gx, lu = adj[b].lu[c];
    double lul = adj[b].lq[c];   // u_l of this step is the next step's history
    double lq = 0.0;
    float lfvm = 0.0f, lkdt = 0.0f, lfb = 0.0f;   // this axis' parts
    float lP = 0.0f, lA0 = 0.0f, lB = 0.0f, lE = 0.0f, ld_re = 0.0f;
    if (c == 2) lu += loss_seed;
    for (int kk = K - 1; kk >= 0; --kk) {
        const SubRec& sr = sub[kk];
        // x_{k+1} = clamp(x_k + u_{k+1} dt_b), u_{k+1} = clamp(u_k + du)
        double lu_next = lu;
        if (!sr.xclamp[c]) lu_next += lx * ac.dt_b;
        else lx = 0.0;
        const double lpre = sr.uclamp[c] ? 0.0 : lu_next;
        const float lp = (float)lpre, v = sr.v[c];
        const float lfd = lp * kdt_f - lpsi_f * inv_K;
        lfvm += lp * kdt_f;
        lkdt += lp * (fz + sr.fd[c] + fvm);
        if (c == 2) lfb += lp * kdt_f;
        // fd = -P cdv v
        const float lfd_v = lane3_sum(lfd * v);
        const float lcdv = -P_f * lfd_v;
        lP += -sr.cdv * lfd_v;
        float lv = -P_f * sr.cdv * lfd, ls = 0.0f;
        if (sr.branch == 0) {
            lE += lcdv * sr.s;
            ls += lcdv * E_f;
        } else if (sr.branch == 1) {
            lA0 += lcdv * (1.0f + sn_coeff * sr.pw);
            if (sr.re > 0.0f) {
                // d(Re^e)/dRe = e Re^e / Re, with 1/Re = nu / (d |v|)
                const float lre = lcdv * A0_f * sn_coeff * sn_exp * sr.pw * nu_over_d * sr.inv_s;
                ls += lre * re_per_s;
                ld_re += lre * sr.s * inv_nu;
            }
        } else {
            lB += lcdv;
        }
        if (sr.s > 0.0f) lv += ls * v * sr.inv_s;
        lu = lpre + lv;
        lul -= lv;
    }
    double lCf = 0.0;
    if (h) {
        lul += lfvm * Cf;
        lq -= lfvm * Cf;
        lCf = lfvm * (ul - q);
    }
    lCf = lane3_sum(lCf);
    lkdt = lane3_sum(lkdt);
    lfb = __shfl_sync(0xffffffffu, lfb, 2);
    // The interpolation adjoint's part of the bubble: sum_c lul_c sum_nodes u_c
    // dW/dx_d (and dW/dn).
    double gx0 = 0.0, gn0 = 0.0;
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        const double le = __shfl_sync(0xffffffffu, lul, e);
        gx0 += le * __shfl_sync(0xffffffffu, tot, 7 + 3 * e + c);
        gn0 += le * __shfl_sync(0xffffffffu, tot, 16 + e);
    }
    if (mine) {
        adj[b].lx[c] = lx + gx0;
        adj[b].lu[c] = lu;
        adj[b].lq[c] = lq;
        lul_out[3 * b + c] = lul;
    }
    if (lane == 0) {
        grad_d[b] += lP * dP + lkdt * dkdt + lfb * dfb + lA0 * dA0 + lB * dBv + lE * dE + ld_re +
                     lCf * dCf + (gn + gn0) * ac.width_factor;
        grad_sD[b] += lP * P / ac.drag_scale;   // summed over bubbles at the end
    }
}

// Lambda^n at the nodes of the interpolation windows, after k_adj_bubbles,
// ADJ_WINDOW_CTAS CTAs per bubble.  A node in several windows belongs to the first active
// bubble whose window holds it; the interpolation adjoints of all of them are
// added to the collision's in bubble order: u(j) = m / rho, du / df_k = (c_k -
// u) / rho.  (One CTA after k_adj_liquid, bubble after bubble, took 20 us of
// every reverse step.)
constexpr int ADJ_WINDOW_CTAS = 8, ADJ_WINDOW_THREADS = 64;

__global__ void __launch_bounds__(ADJ_WINDOW_THREADS)
k_adj_window(const float* __restrict__ fn, const float* __restrict__ lam_next,
             float* __restrict__ lam, Geo g, CollideParams cp, const BubbleSnap* __restrict__ pre,
             const BubbleSnap* __restrict__ post, const double* __restrict__ diam, int nb,
             AdjConst ac, const double* __restrict__ lul_in) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    const int self = blockIdx.x / ADJ_WINDOW_CTAS, part = blockIdx.x % ADJ_WINDOW_CTAS;
    if (!pre[self].active) return;
    AdjView sh(s_dyn, nb);
    sh.load(pre, post, ac.two_way);
    const AdjBox& box = sh.box[self];
    const int M = box.cnt[0] * box.cnt[1] * box.cnt[2];
    for (int m = part * ADJ_WINDOW_THREADS + threadIdx.x; m < M;
         m += ADJ_WINDOW_CTAS * ADJ_WINDOW_THREADS) {
        const int r = m / box.cnt[0], ix = m - r * box.cnt[0];
        const int i = wrap1(box.lo[0] + ix, g.nx), j = wrap1(box.lo[1] + r % box.cnt[1], g.ny),
                  k = wrap1(box.lo[2] + r / box.cnt[1], g.nz);
        bool mine = true;
        for (int b = 0; b < self; ++b)
            mine = mine && !in_window(g, sh.box[b].lo, sh.box[b].cnt, i, j, k);
        if (!mine) continue;
        float out[Q], lamF[3], uj[3], inv_rho;
        const bool inner = i > 0 && i < g.nx - 1 && j > 0 && j < g.ny - 1 && k > 0 && k < g.nz - 1;
        adjoint_at(fn, lam_next, g, cp, sh.rec, sh.spread, nb, i, j, k, inner, out, lamF, uj, inv_rho);
        for (int b = self; b < nb; ++b) {
            if (!in_window(g, sh.box[b].lo, sh.box[b].cnt, i, j, k)) continue;
            Window w;
            make_window(g, pre[b].x, pre[b].xh, pre[b].xl, ac.width_factor * diam[b], w);
            const float W = window_weight(g, w, i, j, k);
            const float lw[3] = {(float)(W * lul_in[3 * b]) * inv_rho,
                                 (float)(W * lul_in[3 * b + 1]) * inv_rho,
                                 (float)(W * lul_in[3 * b + 2]) * inv_rho};
#pragma unroll
            for (int q = 0; q < Q; ++q)
                out[q] += ((float)cx(q) - uj[0]) * lw[0] + ((float)cy(q) - uj[1]) * lw[1] +
                          ((float)cz(q) - uj[2]) * lw[2];
        }
        const int node = node_index(g, i, j, k);
#pragma unroll
        for (int q = 0; q < Q; ++q) lam[(size_t)q * g.S + node] = out[q];
    }
}

// sum_k v_k c_k over the opposite pairs, an axis pair counted `axis` times
// (pairs as in collide_adjoint_pair).
__device__ __forceinline__ void pair_moment(const double v[9], double axis, double out[3]) {
    out[0] = fma(axis, v[0], (v[3] + v[4]) + (v[5] + v[6]));
    out[1] = fma(axis, v[1], (v[3] - v[4]) + (v[7] + v[8]));
    out[2] = fma(axis, v[2], (v[5] - v[6]) + (v[7] - v[8]));
}

// dL/du0 at every node for f^0 = f^eq(rho, u0):
//   dL/du0 = sum_j Lambda^0_j w_j rho (3 c_j + 9 (c_j . u0) c_j - 3 u0).
// Bound by the FP64 pipe (2 FMAs per clock and SM here), so the sums run on
// sums and differences of opposite directions, scaled by 36 so that the
// weights are 12, 2 and 1: about 165 operations per node instead of 545, 1.29 ms
// instead of 3.97 on 128 x 128 x 256, and fewer roundings (error at random
// populations up to 1.5e-16 of the sum of magnitudes, 3.4e-16 by the sum as
// written).  Sums in two floats took 0.55 ms but keep 48 bits (6.3e-16).
__global__ void k_adj_init(const float* __restrict__ f0, const float* __restrict__ lam, Geo g,
                           CollideParams cp, double* __restrict__ du0) {
    const unsigned s = blockIdx.x * blockDim.x + threadIdx.x;   // 19 S < 2^32
    if (s >= (unsigned)g.S) return;
    const unsigned xy = s / (unsigned)g.nx;
    const int x = (int)(s - xy * (unsigned)g.nx), y = (int)(xy % (unsigned)g.ny),
              z = (int)(xy / (unsigned)g.ny);
    float gv[Q], lv[Q];
    gather<0>(f0, g, cp, x, y, z, gv);
#pragma unroll
    for (int j = 0; j < Q; ++j) lv[j] = lam[(size_t)j * g.S + s];
    double v[9], m[3], S1[3];
#pragma unroll
    for (int k = 0; k < 9; ++k) v[k] = (double)gv[2 * k + 1] - (double)gv[2 * k + 2];
    pair_moment(v, 1.0, m);
#pragma unroll
    for (int k = 0; k < 9; ++k) v[k] = (double)gv[2 * k + 1] + (double)gv[2 * k + 2];
    const double drho = (double)gv[0] + ((v[0] + v[1]) + v[2]) +
                        (((v[3] + v[4]) + (v[5] + v[6])) + (v[7] + v[8]));
#pragma unroll
    for (int k = 0; k < 9; ++k) v[k] = (double)lv[2 * k + 1] - (double)lv[2 * k + 2];
    pair_moment(v, 2.0, S1);
#pragma unroll
    for (int k = 0; k < 9; ++k) v[k] = (double)lv[2 * k + 1] + (double)lv[2 * k + 2];
    const double exy = v[3] + v[4], exz = v[5] + v[6], eyz = v[7] + v[8];
    const double S0 = fma(12.0, (double)lv[0], fma(2.0, (v[0] + v[1]) + v[2], (exy + exz) + eyz));
    const double Mxx = fma(2.0, v[0], exy + exz), Myy = fma(2.0, v[1], exy + eyz),
                 Mzz = fma(2.0, v[2], exz + eyz);
    const double Mxy = v[3] - v[4], Mxz = v[5] - v[6], Myz = v[7] - v[8];
    const double rho = (double)cp.rho0 + drho, inv = 1.0 / rho, r12 = rho * (1.0 / 12.0);
    const double u[3] = {m[0] * inv, m[1] * inv, m[2] * inv};
    const double mu[3] = {fma(Mxx, u[0], fma(Mxy, u[1], Mxz * u[2])),
                          fma(Mxy, u[0], fma(Myy, u[1], Myz * u[2])),
                          fma(Mxz, u[0], fma(Myz, u[1], Mzz * u[2]))};
#pragma unroll
    for (int d = 0; d < 3; ++d)
        du0[(size_t)d * g.S + s] = r12 * (S1[d] + fma(3.0, mu[d], -u[d] * S0));
}

}  // namespace

// ---------------------------------------------------------------------------
// Host side: forward record with checkpoints, reverse sweep over segments.
// ---------------------------------------------------------------------------
struct AdjointTape {
    int nsteps = 0, every = 0, window = 0, nb = 0;
    double target = 0.0, ubar = 0.0, loss = 0.0;
    long long version = -1;         // ctx state version at the end of the forward
    size_t fbytes = 0;
    std::vector<void*> ck_f;        // populations at steps 0, every, 2 every, ...
    std::vector<BubbleSnap*> ck_b;  // bubble state there
    int cur0 = 0;                   // buffer index at step 0
    double* uz = nullptr;           // [nsteps * nb] u_b,z after each step
    double* lossbuf = nullptr;      // {ubar, loss}
    void* final_f = nullptr;        // state after the forward, restored after backward
    BubbleSnap* final_b = nullptr;
    int final_cur = 0;
};

void adjoint_free(lbm_ctx* c) {
    AdjointTape* t = c->adj;
    if (!t) return;
    for (void* p : t->ck_f) dfree(c, p);
    for (BubbleSnap* p : t->ck_b) dfree(c, p);
    dfree(c, t->uz);
    dfree(c, t->lossbuf);
    dfree(c, t->final_f);
    dfree(c, t->final_b);
    delete t;
    c->adj = nullptr;
}

extern "C" int lbm_adj_forward(lbm_ctx* c, int nsteps, int checkpoint_every, int window,
                               double target, double* loss) {
    if (!c || nsteps < 1 || checkpoint_every < 1 || window < 1 || window > nsteps)
        return LBM_ERR_ARG;
    int rc = ensure_device(c);
    if (rc) return rc;
    const bool timing = c->timing;   // forward launches are not timed
    c->timing = false;
    struct Restore { lbm_ctx* c; bool t; ~Restore() { c->timing = t; } } restore_timing{c, timing};
    if (c->storage != LBM_STORE_F32)
        return fail(c, LBM_ERR_STATE, "the adjoint needs FP32 population storage");
    if (c->walls & WALL_TOP_FREE)
        return fail(c, LBM_ERR_STATE, "the adjoint covers no-slip and periodic faces only");
    if (c->p.forces != 0)
        return fail(c, LBM_ERR_STATE, "the adjoint covers buoyancy, drag and virtual mass only");
    if (c->p.mapping != LBM_MAP_CELL || c->p.reaction != LBM_REACTION_DRAG_LIFT)
        return fail(c, LBM_ERR_STATE, "the adjoint covers the cell-integral map and the "
                    "-(F_D + F_L) reaction only");
    const int nb = c->bub.nb;
    if (nb < 1 || nb > ADJ_MAX_BUBBLES)
        return fail(c, LBM_ERR_STATE, "the adjoint needs 1..%d bubbles", ADJ_MAX_BUBBLES);
    if (c->p.substeps > ADJ_MAX_SUB)
        return fail(c, LBM_ERR_STATE, "the adjoint supports at most %d sub-steps", ADJ_MAX_SUB);
    if (c->unstable) return fail(c, LBM_ERR_UNSTABLE, "liquid solver is unstable (sticky)");
    adjoint_free(c);
    AdjointTape* t = new AdjointTape();
    c->adj = t;
    t->nsteps = nsteps;
    t->every = checkpoint_every;
    t->window = window;
    t->target = target;
    t->nb = nb;
    const Geo g = geo_of(c);
    t->fbytes = (size_t)Q * (size_t)g.S * sizeof(float);
    t->uz = (double*)dalloc(c, sizeof(double) * (size_t)nsteps * nb);
    t->lossbuf = (double*)dalloc(c, sizeof(double) * 2);
    t->final_f = dalloc(c, t->fbytes);
    t->final_b = (BubbleSnap*)dalloc(c, sizeof(BubbleSnap) * nb);
    if (!t->uz || !t->lossbuf || !t->final_f || !t->final_b) {
        adjoint_free(c);
        return fail(c, LBM_ERR_ALLOC, "adjoint tape");
    }
    const int sb = (nb + 127) / 128;
    cudaStream_t s = c->stream;
    t->cur0 = c->cur;
    for (int n = 0; n < nsteps; ++n) {
        if (n % checkpoint_every == 0) {
            void* ck = dalloc(c, t->fbytes);
            BubbleSnap* cb = (BubbleSnap*)dalloc(c, sizeof(BubbleSnap) * nb);
            if (!ck || !cb) {
                dfree(c, ck);
                dfree(c, cb);
                adjoint_free(c);
                return fail(c, LBM_ERR_ALLOC, "checkpoint of %zu bytes", t->fbytes);
            }
            t->ck_f.push_back(ck);
            t->ck_b.push_back(cb);
            LBM_CUDA(cudaMemcpyAsync(ck, c->f[c->cur], t->fbytes, cudaMemcpyDeviceToDevice, s),
                     "checkpoint");
            k_snapshot<<<sb, 128, 0, s>>>(g, c->bub, cb, 0);
            c->launches += 1;
        }
        rc = enqueue_one_step(c);
        if (rc) return rc;
        k_record_uz<<<sb, 128, 0, s>>>(c->bub, t->uz + (size_t)n * nb);
        c->launches += 1;
    }
    LBM_CUDA(cudaMemcpyAsync(t->final_f, c->f[c->cur], t->fbytes, cudaMemcpyDeviceToDevice, s),
             "final state");
    k_snapshot<<<sb, 128, 0, s>>>(g, c->bub, t->final_b, 0);
    t->final_cur = c->cur;
    k_adj_loss<<<1, 32, 0, s>>>(t->uz, nsteps, nb, window, target, t->lossbuf);
    c->launches += 2;   // the final snapshot and the loss
    LBM_CUDA(cudaGetLastError(), "adjoint forward");
    rc = finish_steps(c);
    if (rc) return rc;
    double lb[2];
    LBM_CUDA(cudaMemcpy(lb, t->lossbuf, sizeof(lb), cudaMemcpyDeviceToHost), "loss");
    t->ubar = lb[0];
    t->loss = lb[1];
    if (loss) *loss = t->loss;
    return LBM_OK;
}

extern "C" int lbm_adj_backward(lbm_ctx* c, double dloss, double* grad_drag_scale,
                                double* grad_diam, double* grad_u0) {
    if (!c) return LBM_ERR_ARG;
    AdjointTape* t = c->adj;
    if (!t) return fail(c, LBM_ERR_STATE, "lbm_adj_backward needs a preceding lbm_adj_forward");
    const Geo g = geo_of(c);
    const CollideParams cp = collide_params(c);
    const int nb = t->nb, N = t->nsteps, K = t->every;
    cudaStream_t s = c->stream;
    const int sb = (nb + 127) / 128;
    // Scratch: the segment's populations and bubble snapshots, two adjoint fields.
    const size_t fb = t->fbytes;
    std::vector<void*> seg_f(K, nullptr);
    for (int k = 0; k < K; ++k) seg_f[k] = dalloc(c, fb);
    BubbleSnap* seg_pre = (BubbleSnap*)dalloc(c, sizeof(BubbleSnap) * (size_t)K * nb);
    BubbleSnap* seg_post = (BubbleSnap*)dalloc(c, sizeof(BubbleSnap) * (size_t)K * nb);
    float* lam[2] = {(float*)dalloc(c, fb), (float*)dalloc(c, fb)};
    BubbleAdj* adj = (BubbleAdj*)dalloc(c, sizeof(BubbleAdj) * nb);
    // grads[0, nb): dL/dd_b; grads[nb, 2 nb): each bubble's part of dL/ds_D
    // (summed over the bubbles in order at the end); lul: the interpolation's
    // seed, from k_adj_bubbles to k_adj_window.
    double* grads = (double*)dalloc(c, sizeof(double) * 2 * (size_t)nb);
    double* lul = (double*)dalloc(c, sizeof(double) * 3 * (size_t)nb);
    double* du0 = grad_u0 ? (double*)dalloc(c, sizeof(double) * 3 * (size_t)g.S) : nullptr;
    auto release = [&]() {
        for (void* p : seg_f) dfree(c, p);
        dfree(c, seg_pre);
        dfree(c, seg_post);
        dfree(c, lam[0]);
        dfree(c, lam[1]);
        dfree(c, adj);
        dfree(c, grads);
        dfree(c, lul);
        dfree(c, du0);
    };
    bool ok = seg_pre && seg_post && lam[0] && lam[1] && adj && grads && lul && (!grad_u0 || du0);
    for (void* p : seg_f) ok = ok && p;
    if (!ok) {
        release();
        return fail(c, LBM_ERR_ALLOC, "adjoint segment storage");
    }
    AdjConst ac;
    ac.nu = (2.0 / c->omega - 1.0) / 6.0;   // Eq. 9
    ac.dt_l = 1.0;
    ac.dt_b = 1.0 / c->p.substeps;
    ac.sn_coeff = c->p.sn_coeff;
    ac.sn_exp = c->p.sn_exp;
    ac.width_factor = c->p.width_factor;
    ac.drag_scale = c->p.drag_scale;
    ac.rho_l = c->p.rho_l;
    ac.rho_b = c->p.rho_ratio * c->p.rho_l;
    ac.g = c->p.g;
    ac.sigma = c->p.sigma;
    ac.c_am = c->p.c_added_mass;
    ac.substeps = c->p.substeps;
    ac.two_way = c->p.two_way;
    const double seed = dloss * 2.0 * (t->ubar - t->target) / ((double)t->window * nb);
    // Kernel timing covers the adjoint sweep only, not the recomputed forward.
    const bool time_adjoint = c->timing;
    c->timing = false;
    struct Restore { lbm_ctx* c; bool t; ~Restore() { c->timing = t; } } restore_timing{c, time_adjoint};
    int lc = 0;   // lam[lc] holds Lambda^{n+1}
    int rc = LBM_OK;
    auto step_rc = [&](cudaError_t e, const char* what) {
        if (e != cudaSuccess && rc == LBM_OK) rc = cuda_fail(c, e, what);
    };
    step_rc(cudaMemsetAsync(lam[lc], 0, fb, s), "lambda");
    step_rc(cudaMemsetAsync(adj, 0, sizeof(BubbleAdj) * nb, s), "bubble adjoint");
    step_rc(cudaMemsetAsync(grads, 0, sizeof(double) * 2 * (size_t)nb, s), "grads");
    // The bubble adjoint and the windows' nodes run on a second stream
    // alongside the liquid adjoint of the other nodes; the step joins both.
    cudaStream_t s2 = nullptr;
    cudaEvent_t ev_in = nullptr, ev_ab = nullptr;
    // (High priority: their few CTAs take the first slots the sweep frees.)
    int least = 0, greatest = 0;
    step_rc(cudaDeviceGetStreamPriorityRange(&least, &greatest), "stream priorities");
    step_rc(cudaStreamCreateWithPriority(&s2, cudaStreamNonBlocking, greatest), "adjoint stream");
    step_rc(cudaEventCreateWithFlags(&ev_in, cudaEventDisableTiming), "event");
    step_rc(cudaEventCreateWithFlags(&ev_ab, cudaEventDisableTiming), "event");
    struct Side {
        cudaStream_t& s2;
        cudaEvent_t& a;
        cudaEvent_t& b;
        ~Side() {
            if (s2) {
                cudaStreamSynchronize(s2);
                cudaStreamDestroy(s2);
            }
            if (a) cudaEventDestroy(a);
            if (b) cudaEventDestroy(b);
        }
    } side{s2, ev_in, ev_ab};
    const unsigned blocks = (unsigned)((g.S + 127) / 128);
    const unsigned pair_blocks = (unsigned)((g.S / 2 + 127) / 128);
    const size_t shared = AdjView::bytes(nb);
    const int nseg = (N + K - 1) / K;
    for (int seg = nseg - 1; seg >= 0 && rc == LBM_OK; --seg) {
        const int n0 = seg * K, n1 = std::min(N, n0 + K);
        // Recompute the segment forward from its checkpoint.  Step n reads its
        // populations from slot n - n0 and writes slot n - n0 + 1 directly, so
        // no state is copied per step; the last step writes into a context
        // buffer, which the final restore overwrites.
        void* const f_ctx[2] = {c->f[0], c->f[1]};
        step_rc(cudaMemcpyAsync(seg_f[0], t->ck_f[seg], fb, cudaMemcpyDeviceToDevice, s), "restore");
        k_restore<<<sb, 128, 0, s>>>(c->bub, t->ck_b[seg]);
        c->launches += 1;
        c->cover_valid = false;
        guard_invalidate(c);
        for (int n = n0; n < n1 && rc == LBM_OK; ++n) {
            c->cur = 0;
            c->f[0] = seg_f[n - n0];
            c->f[1] = n + 1 < n1 ? seg_f[n + 1 - n0] : f_ctx[0];
            k_snapshot<<<sb, 128, 0, s>>>(g, c->bub, seg_pre + (size_t)(n - n0) * nb, 0);
            int r2 = enqueue_one_step(c);
            if (r2) rc = r2;
            k_snapshot<<<sb, 128, 0, s>>>(g, c->bub, seg_post + (size_t)(n - n0) * nb, 1);
            c->launches += 2;   // the two snapshots around the recomputed step
        }
        c->f[0] = f_ctx[0];
        c->f[1] = f_ctx[1];
        // Reverse through the segment.
        for (int n = n1 - 1; n >= n0 && rc == LBM_OK; --n) {
            const float* fn = (const float*)seg_f[n - n0];
            const BubbleSnap* pre = seg_pre + (size_t)(n - n0) * nb;
            const BubbleSnap* post = seg_post + (size_t)(n - n0) * nb;
            cudaEvent_t e1 = nullptr;
            if (time_adjoint) {
                if (c->events_used == c->events.size()) {
                    cudaEvent_t ea, eb;
                    step_rc(cudaEventCreate(&ea), "event");
                    step_rc(cudaEventCreate(&eb), "event");
                    c->events.emplace_back(ea, eb);
                }
                step_rc(cudaEventRecord(c->events[c->events_used].first, s), "event");
                e1 = c->events[c->events_used].second;
                ++c->events_used;
            }
            const double ls = n >= N - t->window ? seed : 0.0;
            step_rc(cudaEventRecord(ev_in, s), "event");
            step_rc(cudaStreamWaitEvent(s2, ev_in, 0), "event wait");
            k_adj_bubbles<<<nb, ADJ_BUBBLE_THREADS, shared, s2>>>(fn, lam[lc], g, cp, pre, post, c->bub.d,
                                                                  nb, ac, adj, grads + nb, grads, lul, ls);
            step_rc(cudaGetLastError(), "bubble adjoint");
            if (g.nx & 1)
                k_adj_liquid<<<blocks, 128, shared, s>>>(fn, lam[lc], lam[lc ^ 1], g, cp, pre, post, nb,
                                                         ac.two_way);
            else
                k_adj_liquid_pair<<<pair_blocks, 128, shared, s>>>(fn, lam[lc], lam[lc ^ 1], g, cp, pre,
                                                                   post, nb, ac.two_way);
            if (e1) step_rc(cudaEventRecord(e1, s), "event");
            step_rc(cudaGetLastError(), "adjoint step");
            // Enqueued after the sweep it runs beside: ahead of it, its wait
            // for the bubble adjoint can hold the sweep back where the two
            // streams share a hardware queue.
            k_adj_window<<<nb * ADJ_WINDOW_CTAS, ADJ_WINDOW_THREADS, shared, s2>>>(fn, lam[lc], lam[lc ^ 1], g, cp, pre, post,
                                                          c->bub.d, nb, ac, lul);
            step_rc(cudaGetLastError(), "window adjoint");
            step_rc(cudaEventRecord(ev_ab, s2), "event");
            step_rc(cudaStreamWaitEvent(s, ev_ab, 0), "event wait");
            c->launches += 3;
            lc ^= 1;
        }
    }
    if (rc == LBM_OK && du0) {
        k_adj_init<<<blocks, 128, 0, s>>>((const float*)t->ck_f[0], lam[lc], g, cp, du0);
        c->launches += 1;
        step_rc(cudaGetLastError(), "initial-field adjoint");
        step_rc(cudaMemcpyAsync(grad_u0, du0, sizeof(double) * 3 * (size_t)g.S, cudaMemcpyDeviceToHost, s),
                "du0");
    }
    std::vector<double> hg(2 * (size_t)nb, 0.0);
    if (rc == LBM_OK)
        step_rc(cudaMemcpyAsync(hg.data(), grads, sizeof(double) * 2 * (size_t)nb,
                                cudaMemcpyDeviceToHost, s),
                "grads");
    // Back to the state after the forward.
    c->cur = t->final_cur;
    step_rc(cudaMemcpyAsync(c->f[c->cur], t->final_f, fb, cudaMemcpyDeviceToDevice, s), "final");
    k_restore<<<sb, 128, 0, s>>>(c->bub, t->final_b);
    c->launches += 1;
    c->cover_valid = false;
    guard_invalidate(c);
    step_rc(cudaStreamSynchronize(s), "adjoint");
    if (s2) step_rc(cudaStreamSynchronize(s2), "adjoint side stream");
    release();
    if (rc) return rc;
    if (grad_drag_scale) {
        double sum = 0.0;
        for (int b = 0; b < nb; ++b) sum += hg[nb + b];
        *grad_drag_scale = sum;
    }
    if (grad_diam)
        for (int b = 0; b < nb; ++b) grad_diam[b] = hg[b];
    return LBM_OK;
}
