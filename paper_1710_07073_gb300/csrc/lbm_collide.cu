// Fused collide-stream sweep (one liquid step of Sec. 2.2 with the bubble
// reaction force of Sec. 3.2).
//
// One thread per lattice node, pull scheme on two structure-of-arrays buffers:
// the thread gathers the 19 populations arriving at its node (Eq. 16 with
// half-way bounce-back, Sec. 3.3), gathers the node's force Phi from the
// bubbles binned to its tile (Eq. 21, fixed order, no atomics), applies the
// first forcing (Eq. 13), BGK collision towards Eq. 6 (Eq. 14) and the second
// forcing with the Guo term (Eq. 12, 15), and writes the post-collision
// populations of its own node.  All arithmetic is FP32 on populations shifted
// by w_j rho0.
//
// The sweep is bound by issue as much as by HBM, so the common case is kept
// short: nodes away from the box faces address their 19 sources with one
// 32-bit offset each, tiles without bubbles skip the forcing terms, and each
// pair of opposite directions shares its equilibrium terms.
#include <climits>
#include "lbm_device.cuh"

namespace lbm {

// Force Phi at node (x,y,z) from one bubble record: tensor product of cell
// integrals (Eq. 19) times psi_b / normalisation.
__device__ __forceinline__ void add_bubble_force(const BubbleRec& r, const Geo& g, int x, int y,
                                                 int z, float& Fx, float& Fy, float& Fz) {
    float rx = (float)(x - r.ax) + 0.5f - r.fx;
    float ry = (float)(y - r.ay) + 0.5f - r.fy;
    float rz = (float)(z - r.az) + 0.5f - r.fz;
    if (!(g.walls & 0x01)) {
        if (rx > 0.5f * g.nx) rx -= (float)g.nx;
        else if (rx < -0.5f * g.nx) rx += (float)g.nx;
    }
    if (!(g.walls & 0x04)) {
        if (ry > 0.5f * g.ny) ry -= (float)g.ny;
        else if (ry < -0.5f * g.ny) ry += (float)g.ny;
    }
    if (!(g.walls & 0x10)) {
        if (rz > 0.5f * g.nz) rz -= (float)g.nz;
        else if (rz < -0.5f * g.nz) rz += (float)g.nz;
    }
    float wx = cell_poly(rx * r.inv_n, r.h);
    if (wx == 0.0f) return;
    float wy = cell_poly(ry * r.inv_n, r.h);
    if (wy == 0.0f) return;
    float wz = cell_poly(rz * r.inv_n, r.h);
    float w = wx * wy * wz;
    Fx = fmaf(w, r.px, Fx);
    Fy = fmaf(w, r.py, Fy);
    Fz = fmaf(w, r.pz, Fz);
}

// Offset of the source of direction J from the receiving node, x fastest.
template <int J>
__device__ __forceinline__ unsigned src_delta(unsigned nx, unsigned nxy) {
    return (unsigned)cx(J) + (unsigned)cy(J) * nx + (unsigned)cz(J) * nxy;
}

// Pull-gather of raw stored values for a node whose y and z neighbours are
// inside the box (all rows but the first and last of each face).  Indices are
// 32-bit (19 S < 2^32 is enforced at creation): the source of J is
// J*S + site - (c_J . (1, nx, nx ny)).  A node on an x face takes its
// x-crossing populations from the opposite plane at its own site (wall) or
// from the other end of the row (periodic), by selects rather than branches.
template <int ST, int J>
__device__ __forceinline__ float pull_raw(const typename Store<ST>::T* __restrict__ f,
                                          unsigned S, unsigned site, unsigned nx, unsigned nxy,
                                          bool xlo, bool xhi, bool wallx) {
    unsigned idx = (unsigned)J * S + site - src_delta<J>(nx, nxy);
    if (cx(J) == 1 && xlo) idx = wallx ? (unsigned)opp(J) * S + site : idx + nx;
    if (cx(J) == -1 && xhi) idx = wallx ? (unsigned)opp(J) * S + site : idx - nx;
    return Store<ST>::load_raw(f + idx);
}

template <int ST>
__device__ __forceinline__ void gather_rows(const typename Store<ST>::T* __restrict__ f,
                                            unsigned S, unsigned site, unsigned nx,
                                            unsigned nxy, bool xlo, bool xhi, bool wallx,
                                            float rv[Q]) {
#define LBM_PULL(J) rv[J] = pull_raw<ST, J>(f, S, site, nx, nxy, xlo, xhi, wallx)
    LBM_PULL(0); LBM_PULL(1); LBM_PULL(2); LBM_PULL(3); LBM_PULL(4);
    LBM_PULL(5); LBM_PULL(6); LBM_PULL(7); LBM_PULL(8); LBM_PULL(9);
    LBM_PULL(10); LBM_PULL(11); LBM_PULL(12); LBM_PULL(13); LBM_PULL(14);
    LBM_PULL(15); LBM_PULL(16); LBM_PULL(17); LBM_PULL(18);
#undef LBM_PULL
}

// General pull-gather of raw values (any node, any walls).
template <int ST, int J>
__device__ __forceinline__ float pull_raw_any(const typename Store<ST>::T* __restrict__ f,
                                              const Geo& g, int x, int y, int z) {
    int plane, idx;
    pull_source<J>(g, x, y, z, plane, idx);
    return Store<ST>::load_raw(f + (size_t)plane * (size_t)g.S + idx);
}

template <int ST>
__device__ __forceinline__ void gather_any(const typename Store<ST>::T* __restrict__ f,
                                           const Geo& g, int x, int y, int z, float rv[Q]) {
#define LBM_PULL(J) rv[J] = pull_raw_any<ST, J>(f, g, x, y, z)
    LBM_PULL(0); LBM_PULL(1); LBM_PULL(2); LBM_PULL(3); LBM_PULL(4);
    LBM_PULL(5); LBM_PULL(6); LBM_PULL(7); LBM_PULL(8); LBM_PULL(9);
    LBM_PULL(10); LBM_PULL(11); LBM_PULL(12); LBM_PULL(13); LBM_PULL(14);
    LBM_PULL(15); LBM_PULL(16); LBM_PULL(17); LBM_PULL(18);
#undef LBM_PULL
}

// One pair of opposite directions (J, J+1 = opp(J)) in raw storage units.
// Eq. 6 is split into its even part (shared by the pair) and odd part (sign
// flips); g^eq_j / w_j = base + 9/2 rho cu^2 +- 3 rho cu.  BGK relaxation
// (Eq. 14) is r' = (1 - omega) r + C [omega g^eq / w], and the Guo term of
// Eq. 12 adds C pref [(9 cu cF - 3 u.F) +- 3 cF], where C = w_J for FP32
// storage and C = scale for the 16-bit formats (r = g scale / w).
template <int ST, int J, bool FORCED>
__device__ __forceinline__ void relax_pair(typename Store<ST>::T* __restrict__ fout, unsigned S,
                                           unsigned site, const float rv[Q], float base,
                                           float rho, float ux, float uy, float uz, float Fx,
                                           float Fy, float Fz, float uF,
                                           const CollideParams& cp) {
    const float C = Store<ST>::kScaled ? cp.scale : wf(J);
    const float cu = (float)cx(J) * ux + (float)cy(J) * uy + (float)cz(J) * uz;
    float even = cp.omega * fmaf(4.5f * rho * cu, cu, base);
    float odd = cp.omega * 3.0f * rho * cu;
    if (FORCED) {
        const float cF = (float)cx(J) * Fx + (float)cy(J) * Fy + (float)cz(J) * Fz;
        even = fmaf(cp.pref, 9.0f * cu * cF - 3.0f * uF, even);
        odd = fmaf(cp.pref, 3.0f * cF, odd);
    }
    const float om1 = 1.0f - cp.omega;
    Store<ST>::store_raw(fout + ((unsigned)J * S + site), fmaf(om1, rv[J], C * (even + odd)));
    Store<ST>::store_raw(fout + ((unsigned)(J + 1) * S + site),
                         fmaf(om1, rv[J + 1], C * (even - odd)));
}

template <int ST, bool FORCED>
__device__ __forceinline__ void collide_store(typename Store<ST>::T* __restrict__ fout,
                                              unsigned S, unsigned site, const float rv[Q],
                                              float Fx, float Fy, float Fz,
                                              const CollideParams& cp, int* flag) {
    // Eq. 10 / Eq. 13 moments of g = r k, k = 1 (FP32) or w_j / scale
    // (16-bit); sum_j w_j c_j = 0 so the shift drops out of the momentum.
    const float s_rest = rv[0];
    const float s_axis = (rv[1] + rv[2]) + (rv[3] + rv[4]) + (rv[5] + rv[6]);
    const float s_edge = ((rv[7] + rv[8]) + (rv[9] + rv[10])) + ((rv[11] + rv[12]) + (rv[13] + rv[14])) +
                         ((rv[15] + rv[16]) + (rv[17] + rv[18]));
    const float ax_x = rv[1] - rv[2], ax_y = rv[3] - rv[4], ax_z = rv[5] - rv[6];
    const float ed_x = (rv[7] - rv[8]) + (rv[9] - rv[10]) + (rv[11] - rv[12]) + (rv[13] - rv[14]);
    const float ed_y = (rv[7] - rv[8]) + (rv[10] - rv[9]) + (rv[15] - rv[16]) + (rv[17] - rv[18]);
    const float ed_z = (rv[11] - rv[12]) + (rv[14] - rv[13]) + (rv[15] - rv[16]) + (rv[18] - rv[17]);
    float drho, jx, jy, jz;
    if (Store<ST>::kScaled) {
        const float k0 = wf(0) * cp.inv_scale, ka = wf(1) * cp.inv_scale, ke = wf(7) * cp.inv_scale;
        drho = fmaf(k0, s_rest, fmaf(ka, s_axis, ke * s_edge));
        jx = fmaf(ka, ax_x, ke * ed_x);
        jy = fmaf(ka, ax_y, ke * ed_y);
        jz = fmaf(ka, ax_z, ke * ed_z);
    } else {
        drho = s_rest + s_axis + s_edge;
        jx = ax_x + ed_x;
        jy = ax_y + ed_y;
        jz = ax_z + ed_z;
    }
    const float rho = cp.rho0 + drho;
    const float inv_rho = 1.0f / rho;
    float ux, uy, uz;
    if (FORCED) {
        ux = fmaf(0.5f, Fx, jx) * inv_rho;
        uy = fmaf(0.5f, Fy, jy) * inv_rho;
        uz = fmaf(0.5f, Fz, jz) * inv_rho;
    } else {
        ux = jx * inv_rho;
        uy = jy * inv_rho;
        uz = jz * inv_rho;
    }
    const float usq = ux * ux + uy * uy + uz * uz;
    if (!(usq < 0.09f)) atomicOr(flag, 1);   // non-finite or beyond |u| = 0.3
    const float uF = FORCED ? (ux * Fx + uy * Fy + uz * Fz) : 0.0f;
    // Common part of g^eq_j / w_j: drho - 3/2 rho u^2.
    const float base = fmaf(-1.5f * rho, usq, drho);
    float e0 = cp.omega * base;
    if (FORCED) e0 = fmaf(cp.pref, -3.0f * uF, e0);   // Eq. 12 with c_0 = 0
    const float C0 = Store<ST>::kScaled ? cp.scale : wf(0);
    Store<ST>::store_raw(fout + site, fmaf(1.0f - cp.omega, rv[0], C0 * e0));
#define LBM_PAIR(J) relax_pair<ST, J, FORCED>(fout, S, site, rv, base, rho, ux, uy, uz, Fx, Fy, Fz, uF, cp)
    LBM_PAIR(1); LBM_PAIR(3); LBM_PAIR(5); LBM_PAIR(7); LBM_PAIR(9);
    LBM_PAIR(11); LBM_PAIR(13); LBM_PAIR(15); LBM_PAIR(17);
#undef LBM_PAIR
}

// Odd rows: a CTA is 32 x 4 nodes of one z-plane, a node per thread (rows of odd
// length leave no aligned 2-wide access).  127 x 127 x 255, FP32: 0.115 ms, 80 %
// of the copy peak.  Two planes per thread, all rows loaded first, took 0.122 ms:
// it is not the loads in flight that bound it but the sectors that unaligned
// rows share between warps.  Overlapped with the bubble update as the even
// rows' sweep is (126 us a step before, in stream order).  The 16-bit formats,
// whose loads are half as long, take 10 CTAs per SM (48 registers): a step in
// FP16 82.6 us against 88.1 at 8 (12: 83.8), 201 x 150 x 300 193 against 199;
// FP32 loses by it (117.5 us at 10, 115.3 at 6).
constexpr int ODD_PZ = 1;
constexpr int ODD_CHUNK = 32;   // bubble records staged per pass

// The pre-collision populations of a node (a warp is one row), its site.
template <int ST>
__device__ __forceinline__ unsigned odd_gather(const typename Store<ST>::T* __restrict__ fin,
                                               const Geo& g, int x, int y, int z, float rv[Q]) {
    const unsigned nx = (unsigned)g.nx, nxy = (unsigned)g.nx * (unsigned)g.ny;
    const unsigned site = (unsigned)z * nxy + (unsigned)y * nx + (unsigned)x;
    // Rows away from the y and z faces (uniform over a warp).
    if (y > 0 && y < g.ny - 1 && z > 0 && z < g.nz - 1)
        gather_rows<ST>(fin, (unsigned)g.S, site, nx, nxy, x == 0, x == g.nx - 1,
                        (g.walls & 0x01) != 0, rv);
    else
        gather_any<ST>(fin, g, x, y, z, rv);
    return site;
}

template <int ST>
__global__ void __launch_bounds__(TX * TY, ST == 0 ? 8 : 10)
k_collide_stream(const typename Store<ST>::T* __restrict__ fin,
                 typename Store<ST>::T* __restrict__ fout, Geo g, CollideParams cp,
                 const int* tile_start, const int* tile_count, const int* items, int cap,
                 const BubbleRec* recs, int nb, int* __restrict__ flag, const unsigned* safe,
                 unsigned epoch, const int* zperm) {
    __shared__ BubbleRec srec[ODD_CHUNK];
    pdl_trigger();
    const int z = zperm != nullptr ? __ldcg(zperm + blockIdx.z) : (int)blockIdx.z;
    const bool lead = (blockIdx.x | blockIdx.y | blockIdx.z) == 0;
    const int x = blockIdx.x * TX + threadIdx.x;
    const int y = blockIdx.y * TY + threadIdx.y;
    const bool inside = (x < g.nx) && (y < g.ny);
    const unsigned S = (unsigned)g.S;
    // No lists: left at once.  Behind the force gather the 16-bit formats took
    // 16.7 us a step on 63 x 64 x 128, 14.7 here.
    if (tile_count == nullptr) {
        if (!inside) return;
        float rv[Q];
        const unsigned site = odd_gather<ST>(fin, g, x, y, z, rv);
        collide_store<ST, false>(fout, S, site, rv, 0.0f, 0.0f, 0.0f, cp, flag);
        return;
    }
    const int t = ((z / TZ) * g.nty + blockIdx.y) * g.ntx + blockIdx.x;
    // The order of the tile count, the population loads and the wait for an
    // overlapped update is sweep_block's.
    int n_t = 0;
    bool skip = false;
    if (safe == nullptr) n_t = __ldcg(tile_count + t);
    else skip = !lead && __ldcg(safe + z / TZ) == epoch;
    // Threads beyond the box gather at a valid node and store nothing.
    float rv[Q];
    const unsigned site = odd_gather<ST>(fin, g, min(x, g.nx - 1), min(y, g.ny - 1), z, rv);
    if (safe != nullptr && !skip) {
        pdl_wait();
        n_t = __ldcg(tile_count + t);
    }
    float Fx = 0.0f, Fy = 0.0f, Fz = 0.0f;
    if (n_t > 0) {   // uniform over the CTA (one tile)
        const int beg = __ldcg(tile_start + t);
        const int end = min(beg + n_t, cap);
        const int tid = threadIdx.y * TX + threadIdx.x;
        for (int c0 = beg; c0 < end; c0 += ODD_CHUNK) {
            const int cnt = min(ODD_CHUNK, end - c0);
            __syncthreads();
            if (tid < cnt) {
                const int id = __ldcg(items + c0 + tid);
                if (id >= 0 && id < nb) srec[tid] = load_rec(recs + id);
                else srec[tid] = BubbleRec{0, 0, 0, 0, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            }
            __syncthreads();
            if (inside)
                for (int k = 0; k < cnt; ++k) add_bubble_force(srec[k], g, x, y, z, Fx, Fy, Fz);
        }
    }
    if (!inside) return;
    if (n_t > 0) collide_store<ST, true>(fout, S, site, rv, Fx, Fy, Fz, cp, flag);
    else collide_store<ST, false>(fout, S, site, rv, 0.0f, 0.0f, 0.0f, cp, flag);
}

// ---------------------------------------------------------------------------
// Two nodes per thread (even nx).  Each thread owns the x-pair (x0, x0 + 1),
// x0 even, so every plane row is read and written with aligned 2-wide vector
// accesses (float2, half2, bfloat162) and the collision runs on packed FP32
// pairs (FFMA2 / FADD2 / FMUL2).  A CTA is 16 x 4 x 2 threads = 32 x 4 x 2
// nodes, inside one binning tile.
// ---------------------------------------------------------------------------
// Resident CTAs per SM the register budget is sized for: FP32 rows move twice
// the bytes per thread and keep more registers; the 16-bit formats need more
// warps in flight to cover memory latency.  Measured on GB300 (FP16 sweep,
// 256x256x512, rows kept packed until use): 8 CTAs (64 registers) 0.439 ms,
// 7 CTAs 0.448 ms, 9 CTAs 0.461 ms.
#ifndef LBM_PAIR_MINB_16
#define LBM_PAIR_MINB_16 8
#endif
template <int ST> struct PairOccupancy {
    static constexpr int kMinBlocks = ST == 0 ? 6 : LBM_PAIR_MINB_16;
};
constexpr int PX = TX / 2;   // threads along x
// Bubbles staged per pass of the sweep's force gather (records and per-axis
// weight tables in shared memory).
constexpr int FORCE_CHUNK = 32;
constexpr int PZ = SWEEP_PZ;      // z-planes per CTA (divides TZ)
static_assert(TZ % PZ == 0, "a CTA's z-planes must lie in one binning tile");


// Force of one bubble record on the pair (x0, x0 + 1) at (y, z), Eq. 19 and 21.
__device__ __forceinline__ void add_bubble_force_pair(const BubbleRec& r, const Geo& g, int x0,
                                                      int y, int z, float2& Fx, float2& Fy,
                                                      float2& Fz) {
    float ry = (float)(y - r.ay) + 0.5f - r.fy;
    float rz = (float)(z - r.az) + 0.5f - r.fz;
    if (!(g.walls & 0x04)) {
        if (ry > 0.5f * g.ny) ry -= (float)g.ny;
        else if (ry < -0.5f * g.ny) ry += (float)g.ny;
    }
    if (!(g.walls & 0x10)) {
        if (rz > 0.5f * g.nz) rz -= (float)g.nz;
        else if (rz < -0.5f * g.nz) rz += (float)g.nz;
    }
    const float wy = cell_poly(ry * r.inv_n, r.h);
    if (wy == 0.0f) return;
    const float wyz = wy * cell_poly(rz * r.inv_n, r.h);
    if (wyz == 0.0f) return;
    float w[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        float rx = (float)(x0 + k - r.ax) + 0.5f - r.fx;
        if (!(g.walls & 0x01)) {
            if (rx > 0.5f * g.nx) rx -= (float)g.nx;
            else if (rx < -0.5f * g.nx) rx += (float)g.nx;
        }
        w[k] = cell_poly(rx * r.inv_n, r.h) * wyz;
    }
    const float2 wv = make_float2(w[0], w[1]);
    Fx = fma2(wv, f2(r.px), Fx);
    Fy = fma2(wv, f2(r.py), Fy);
    Fz = fma2(wv, f2(r.pz), Fz);
}

// c_j . v for direction J (J odd; J + 1 is its opposite), written with adds
// only: no multiply by +-1.
template <int J>
__device__ __forceinline__ float2 c_dot(float2 vx, float2 vy, float2 vz) {
    constexpr int X = cx(J), Y = cy(J), Z = cz(J);
    static_assert((J & 1) && (X == 1 || (X == 0 && Y == 1) || (X == 0 && Y == 0 && Z == 1)),
                  "odd directions lead with a +1 component");
    if (Y == 0 && Z == 0) return vx;                    // J = 1 (+x)
    if (X == 0 && Z == 0) return vy;                    // J = 3 (+y)
    if (X == 0 && Y == 0) return vz;                    // J = 5 (+z)
    if (Z == 0) return Y > 0 ? add2(vx, vy) : sub2(vx, vy);
    if (Y == 0) return Z > 0 ? add2(vx, vz) : sub2(vx, vz);
    return Z > 0 ? add2(vy, vz) : sub2(vy, vz);
}

// Per-class coefficients of the relaxation in stored units: with K = C omega
// (C = w_j for FP32, the storage scale for 16 bits), the post-collision value
// of J and of its opposite is
//   (1 - omega) r_{J or J+1} + K base + 4.5 K rho (c.u)^2  +-  3 K rho (c.u)
// (Eq. 6 and 14 with f^eq - w rho0 written around base = drho - 1.5 rho u^2).
struct RelaxK {
    float2 base, r45, r3;
};

__device__ __forceinline__ RelaxK relax_k(float K, float2 base, float2 rho) {
    return RelaxK{mul2(f2(K), base), mul2(f2(4.5f * K), rho), mul2(f2(3.0f * K), rho)};
}

// Where a collided pair goes: the pair kernels store it 2-wide in plane J at
// site0.
template <int ST>
struct PairStore {
    typename Store<ST>::T* fout;
    unsigned S, site0;
    bool store;
    template <int J>
    __device__ __forceinline__ void put(float2 v) const {
        if (store) Vec2<ST>::store(fout + ((unsigned)J * S + site0), v);
    }
};

template <int ST, int J, bool FORCED, class Sink>
__device__ __forceinline__ void relax_pair2(Sink& sink, const typename Raw2<ST>::T rv[Q],
                                            const RelaxK& k,
                                            float2 ux, float2 uy, float2 uz, float2 Fx, float2 Fy,
                                            float2 Fz, float2 uF, const CollideParams& cp) {
    const float2 cu = c_dot<J>(ux, uy, uz);
    float2 even = fma2(mul2(k.r45, cu), cu, k.base);
    float2 odd = mul2(k.r3, cu);
    if (FORCED) {
        // Guo term (Eq. 15), (1 - omega/2) w_j [3 (c - u) + 9 (c.u) c] . F
        const float C = Store<ST>::kScaled ? cp.scale : wf(J);
        const float2 cF = c_dot<J>(Fx, Fy, Fz);
        even = fma2(f2(C * cp.pref), fma2(mul2(f2(9.0f), cu), cF, mul2(f2(-3.0f), uF)), even);
        odd = fma2(f2(3.0f * C * cp.pref), cF, odd);
    }
    const float2 om1 = f2(1.0f - cp.omega);
    sink.template put<J>(fma2(om1, Raw2<ST>::widen(rv[J]), add2(even, odd)));
    sink.template put<J + 1>(fma2(om1, Raw2<ST>::widen(rv[J + 1]), sub2(even, odd)));
}

// Collision of one x-pair of nodes (Eq. 13, 6, 14, 12, 15) from its
// pre-collision values rr (stored units, as loaded); `live` pairs take part in
// the stability flag.
template <int ST, bool FORCED, class Sink>
__device__ __forceinline__ void collide_pair(Sink& sink, const typename Raw2<ST>::T rr[Q],
                                             float2 Fx, float2 Fy, float2 Fz,
                                             const CollideParams& cp, int* flag, bool live) {
    float2 drho, jx, jy, jz;
    pair_moments<ST>(rr, cp, drho, jx, jy, jz);
    const float2 rho = add2(f2(cp.rho0), drho);
    const float2 inv_rho = make_float2(1.0f / rho.x, 1.0f / rho.y);
    float2 ux, uy, uz;
    if (FORCED) {
        ux = mul2(fma2(f2(0.5f), Fx, jx), inv_rho);
        uy = mul2(fma2(f2(0.5f), Fy, jy), inv_rho);
        uz = mul2(fma2(f2(0.5f), Fz, jz), inv_rho);
    } else {
        ux = mul2(jx, inv_rho);
        uy = mul2(jy, inv_rho);
        uz = mul2(jz, inv_rho);
    }
    const float2 usq = fma2(ux, ux, fma2(uy, uy, mul2(uz, uz)));
    if (live && !(usq.x < 0.09f && usq.y < 0.09f)) atomicOr(flag, 1);
    const float2 uF = FORCED ? fma2(ux, Fx, fma2(uy, Fy, mul2(uz, Fz))) : f2(0.0f);
    const float2 base = fma2(mul2(f2(-1.5f), rho), usq, drho);
    float2 e0 = mul2(f2(cp.omega), base);
    if (FORCED) e0 = fma2(f2(-3.0f * cp.pref), uF, e0);
    const float C0 = Store<ST>::kScaled ? cp.scale : wf(0);
    sink.template put<0>(fma2(f2(1.0f - cp.omega), Raw2<ST>::widen(rr[0]), mul2(f2(C0), e0)));
    // One coefficient class for the 16-bit formats (C = scale); FP32 has
    // the axis and the diagonal weights.
    const RelaxK ka = relax_k((Store<ST>::kScaled ? cp.scale : wf(1)) * cp.omega, base, rho);
    const RelaxK ke = Store<ST>::kScaled ? ka : relax_k(wf(7) * cp.omega, base, rho);
#define LBM_PAIR2(J, K) relax_pair2<ST, J, FORCED>(sink, rr, K, ux, uy, uz, Fx, Fy, Fz, uF, cp)
    LBM_PAIR2(1, ka); LBM_PAIR2(3, ka); LBM_PAIR2(5, ka); LBM_PAIR2(7, ke); LBM_PAIR2(9, ke);
    LBM_PAIR2(11, ke); LBM_PAIR2(13, ke); LBM_PAIR2(15, ke); LBM_PAIR2(17, ke);
#undef LBM_PAIR2
}

// Eq. 21 at the pair (x0, x0 + 1), (y, z) of a block whose tile lists n_t > 0
// bubbles, for long tile lists (many bubbles).  Every thread of the CTA calls
// it (it synchronises the CTA).
struct Force2 {
    float2 x, y, z;
};

template <int ST>
__device__ __forceinline__ Force2 gather_force_tab(const Geo& g, const int* __restrict__ tile_start,
                                                 const int* __restrict__ items, int cap,
                                                 const BubbleRec* __restrict__ recs, int nb,
                                                 int n_t, int bx, int by, int bz, int x0, int y,
                                                 int z, bool active, BubbleRec* srec, bool point) {
    float2 Fx = f2(0.0f), Fy = f2(0.0f), Fz = f2(0.0f);
    // Chunks of FB bubbles: the CTA first tabulates each bubble's per-axis
    // cell integrals over the block (TX columns, TY rows, PZ planes), then
    // every node forms wx (wy wz) from the tables.  Same products, zero test
    // and order as add_bubble_force_pair.
    constexpr int FB = FORCE_CHUNK, NAX = TX + TY + PZ;
    __shared__ float s_w[FB][NAX];   // x: [0, TX), y: [TX, TX + TY), z: the rest
    const int t = (((bz * PZ) / TZ) * g.nty + by) * g.ntx + bx;
    const int beg = __ldcg(tile_start + t);
    const int end = min(beg + n_t, cap);
    const int tid = (threadIdx.z * TY + threadIdx.y) * PX + threadIdx.x;
    constexpr int NT = PX * TY * PZ;
    const int xb0 = bx * TX, yb0 = by * TY, zb0 = bz * PZ;
    for (int c0 = beg; c0 < end; c0 += FB) {
        const int cnt = min(FB, end - c0);
        __syncthreads();
        if (tid < cnt) {
            const int id = __ldcg(items + c0 + tid);
            if (id >= 0 && id < nb) srec[tid] = load_rec(recs + id);
            else srec[tid] = BubbleRec{0, 0, 0, 0, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        }
        __syncthreads();
        // The mapping mode is the same for every bubble: one loop per mode.
        auto tabulate = [&](auto mode) {
            constexpr int PM = decltype(mode)::value;
            for (int e = tid; e < cnt * NAX; e += NT) {
                const int k = e / NAX, q = e - k * NAX;
                const BubbleRec& r = srec[k];
                if (q < TX)
                    s_w[k][q] = axis_weight<PM>(r, xb0 + q, r.ax, r.fx, g.nx, !(g.walls & 0x01));
                else if (q < TX + TY)
                    s_w[k][q] = axis_weight<PM>(r, yb0 + q - TX, r.ay, r.fy, g.ny, !(g.walls & 0x04));
                else
                    s_w[k][q] =
                        axis_weight<PM>(r, zb0 + q - TX - TY, r.az, r.fz, g.nz, !(g.walls & 0x10));
            }
        };
        // (FP32 keeps the one loop with the mode read per weight: its sweep
        // has the slack, and the smaller code measured faster.)
        if (ST == 0) tabulate(MapMode<MAP_ANY>{});
        else if (point) tabulate(MapMode<MAP_POINT>{});
        else tabulate(MapMode<MAP_CELL>{});
        __syncthreads();
        if (active) {
            const int xi = 2 * threadIdx.x, yi = TX + threadIdx.y, zi = TX + TY + threadIdx.z;
            for (int k = 0; k < cnt; ++k) {
                const float wyz = s_w[k][yi] * s_w[k][zi];
                if (wyz == 0.0f) continue;
                const float2 wv = make_float2(s_w[k][xi] * wyz, s_w[k][xi + 1] * wyz);
                const BubbleRec& r = srec[k];
                Fx = fma2(wv, f2(r.px), Fx);
                Fy = fma2(wv, f2(r.py), Fy);
                Fz = fma2(wv, f2(r.pz), Fz);
            }
        }
    }
    __syncthreads();   // srec and s_w are reused by the CTA's next block
    return Force2{Fx, Fy, Fz};
}

// One CTA's block of the sweep: x-pairs of 32 nodes, TY rows, PZV planes at
// block coordinates (bx, by, bz).  `srec` is the CTA's staging of bubble
// records; every thread of the CTA must call this with the same block.
template <int ST, bool TAB, int PZV = PZ>
__device__ __forceinline__ void sweep_block(const typename Store<ST>::T* __restrict__ fin,
                                            typename Store<ST>::T* __restrict__ fout,
                                            const Geo& g, const CollideParams& cp,
                                            const int* __restrict__ tile_start,
                                            const int* __restrict__ tile_count,
                                            const int* __restrict__ items, int cap,
                                            const BubbleRec* __restrict__ recs, int nb,
                                            int* __restrict__ flag, int bx, int by, int bz,
                                            BubbleRec* srec, const unsigned* safe = nullptr,
                                            unsigned epoch = 0, bool lead = false) {
    static_assert(TZ % PZV == 0 && (!TAB || PZV == PZ), "a block lies in one tile layer");
    const int x0 = bx * TX + 2 * threadIdx.x;
    const int y = by * TY + threadIdx.y;
    const int z = bz * PZV + threadIdx.z;
    const bool active = (x0 < g.nx) && (y < g.ny) && (z < g.nz);
    // Inactive threads gather at a valid node and store nothing.
    const int xa = active ? x0 : 0;
    const int ya = min(y, g.ny - 1), za = min(z, g.nz - 1);

    const int t = (((bz * PZV) / TZ) * g.nty + by) * g.ntx + bx;
    // Read before the population loads: in plain stream order the tile count;
    // overlapped with the bubble update, the guard tag of this z layer (written
    // by the update before, which has completed).  The launch's first CTA
    // (`lead`) never skips, so the sweep cannot complete before the update.
    int n_t = 0;
    bool skip = false;
    if (tile_count != nullptr) {
        if (safe == nullptr) n_t = __ldcg(tile_count + t);
        else skip = !lead && __ldcg(safe + (bz * PZV) / TZ) == epoch;
    }

    const unsigned S = (unsigned)g.S;
    const unsigned nx = (unsigned)g.nx, nxy = (unsigned)g.nx * (unsigned)g.ny;
    const unsigned site0 = (unsigned)za * nxy + (unsigned)ya * nx + (unsigned)xa;
    typename Raw2<ST>::T rv[Q];
    gather_pair<ST>(fin, g, xa, ya, za, rv);
    if (tile_count != nullptr && safe != nullptr && !skip) {
        // Overlapped, and the update before did not clear this layer: wait
        // for this step's update, then read its tile lists.
        pdl_wait();
        n_t = __ldcg(tile_count + t);
    }
    // The force gather (Eq. 21) runs after the population loads are issued,
    // so the tile-list lookup does not delay them.
    float2 Fx = f2(0.0f), Fy = f2(0.0f), Fz = f2(0.0f);
    const bool forced = n_t > 0;   // uniform over the CTA (one tile)
    if (forced && TAB) {
        const Force2 F = gather_force_tab<ST>(g, tile_start, items, cap, recs, nb, n_t, bx, by, bz,
                                          x0, y, z, active, srec, cp.point != 0);
        Fx = F.x;
        Fy = F.y;
        Fz = F.z;
    } else if (forced) {
        // Few bubbles per tile: each node evaluates its listed bubbles directly.
        const int beg = __ldcg(tile_start + t);
        const int end = min(beg + n_t, cap);
        const int tid = (threadIdx.z * TY + threadIdx.y) * PX + threadIdx.x;
        for (int c0 = beg; c0 < end; c0 += FORCE_CHUNK) {
            const int cnt = min(FORCE_CHUNK, end - c0);
            __syncthreads();
            if (tid < cnt) {
                const int id = __ldcg(items + c0 + tid);
                if (id >= 0 && id < nb) srec[tid] = load_rec(recs + id);
                else srec[tid] = BubbleRec{0, 0, 0, 0, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            }
            __syncthreads();
            if (active)
                for (int k = 0; k < cnt; ++k)
                    add_bubble_force_pair(srec[k], g, x0, y, z, Fx, Fy, Fz);
        }
        __syncthreads();   // srec is reused by the CTA's next block
    }

    PairStore<ST> sink{fout, S, site0, active};
    if (forced) collide_pair<ST, true>(sink, rv, Fx, Fy, Fz, cp, flag, active);
    else collide_pair<ST, false>(sink, rv, Fx, Fy, Fz, cp, flag, active);
}

// ---------------------------------------------------------------------------
// Four nodes per thread: 16-bit storage on rows whose length is a multiple of
// 4.  A CTA is 8 x 4 x 4 threads = one 32 x 4 x 4 binning tile.
//
// The 16-bit sweep moves half the bytes of FP32 per node, so with two nodes per
// thread it was bound by its load latency and instructions (82 % of the copy
// peak, 256 x 256 x 512).  Four nodes halve the row loads, the x-crossing loads
// and the address arithmetic per node and double the bytes a thread has in
// flight.  The raw values wait in shared memory (QuadSlot): kept in registers
// the kernel spilled at 80 registers and lost (0.476 ms).  At 6 CTAs per SM
// (80 registers, no spills without force; 4: 0.410, 5: 0.396, 7: 0.427,
// 8: 0.476 ms) the 256 x 256 x 512 FP16 step takes 0.391 ms against 0.444 ms
// with two nodes (96 % of the copy peak), the 384 x 384 x 768 swarm's FP16 step
// 1.953 against 2.116 ms, its whole listed sweep 1.660 against 1.777 ms (1.647
// with a tile's first records staged before the rows are used).
// ---------------------------------------------------------------------------
constexpr int QX = TX / 4;      // threads along x
constexpr int QUAD_PZ = TZ;     // z-planes per CTA
constexpr int QUAD_THREADS = QX * TY * QUAD_PZ;
#ifndef LBM_QUAD_MINB
#define LBM_QUAD_MINB 6
#endif
// CTA shape and residency of the sweep kernels, by nodes per thread.
template <int ST, int NODES> struct SweepShape {
    static constexpr int kThreads = PX * TY * PZ, kPlanes = PZ;
    static constexpr int kMinBlocks = PairOccupancy<ST>::kMinBlocks;
};
template <int ST> struct SweepShape<ST, 4> {
    static constexpr int kThreads = QUAD_THREADS, kPlanes = QUAD_PZ;
    static constexpr int kMinBlocks = LBM_QUAD_MINB;
};

// The raw values of a thread's quads wait in shared memory between the moments
// and the relaxation (a slot per thread, so no synchronisation): held in
// registers, packed and widened, they spill at any occupancy that hides the
// load latency.
template <int PZV>
struct QuadSlot {
    unsigned at;   // shared-space address of direction 0
    static constexpr unsigned STRIDE = QX * TY * PZV * 8;
    template <int J>
    __device__ __forceinline__ void put(unsigned a, unsigned b) const {
        asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(at + J * STRIDE), "r"(a), "r"(b));
    }
    template <int J>
    __device__ __forceinline__ void put_a(unsigned a) const {
        asm volatile("st.shared.u32 [%0], %1;" ::"r"(at + J * STRIDE), "r"(a));
    }
    // Half H (0: first pair, 1: second) of direction J.
    template <int J, int H>
    __device__ __forceinline__ unsigned get_half() const {
        unsigned v;
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(at + J * STRIDE + 4 * H));
        return v;
    }
    template <int H>
    __device__ __forceinline__ void get_all(unsigned v[Q]) const {
#define LBM_GH(J) v[J] = get_half<J, H>()
        LBM_GH(0); LBM_GH(1); LBM_GH(2); LBM_GH(3); LBM_GH(4); LBM_GH(5); LBM_GH(6);
        LBM_GH(7); LBM_GH(8); LBM_GH(9); LBM_GH(10); LBM_GH(11); LBM_GH(12); LBM_GH(13);
        LBM_GH(14); LBM_GH(15); LBM_GH(16); LBM_GH(17); LBM_GH(18);
#undef LBM_GH
    }
    template <int J>
    __device__ __forceinline__ Quad get() const {
        Quad q;
        asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];"
                     : "=r"(q.a), "=r"(q.b)
                     : "r"(at + J * STRIDE));
        return q;
    }
};

// What the relaxation of one pair needs (collide_pair's values).
struct PairState {
    float2 ux, uy, uz, uF;
    RelaxK k;
    float2 rest;   // C0 e0
};

template <int ST, bool FORCED>
__device__ __forceinline__ PairState pair_state(const unsigned rr[Q], float2 Fx, float2 Fy,
                                                float2 Fz, const CollideParams& cp, int* flag,
                                                bool live) {
    static_assert(Store<ST>::kScaled, "16-bit storage: one coefficient class");
    PairState p;
    float2 drho, jx, jy, jz;
    pair_moments<ST>(rr, cp, drho, jx, jy, jz);
    const float2 rho = add2(f2(cp.rho0), drho);
    const float2 inv_rho = make_float2(1.0f / rho.x, 1.0f / rho.y);
    if (FORCED) {
        p.ux = mul2(fma2(f2(0.5f), Fx, jx), inv_rho);
        p.uy = mul2(fma2(f2(0.5f), Fy, jy), inv_rho);
        p.uz = mul2(fma2(f2(0.5f), Fz, jz), inv_rho);
    } else {
        p.ux = mul2(jx, inv_rho);
        p.uy = mul2(jy, inv_rho);
        p.uz = mul2(jz, inv_rho);
    }
    const float2 usq = fma2(p.ux, p.ux, fma2(p.uy, p.uy, mul2(p.uz, p.uz)));
    if (live && !(usq.x < 0.09f && usq.y < 0.09f)) atomicOr(flag, 1);
    p.uF = FORCED ? fma2(p.ux, Fx, fma2(p.uy, Fy, mul2(p.uz, Fz))) : f2(0.0f);
    const float2 base = fma2(mul2(f2(-1.5f), rho), usq, drho);
    float2 e0 = mul2(f2(cp.omega), base);
    if (FORCED) e0 = fma2(f2(-3.0f * cp.pref), p.uF, e0);
    p.rest = mul2(f2(cp.scale), e0);
    p.k = relax_k(cp.scale * cp.omega, base, rho);
    return p;
}

// One pair's post-collision values of J and its opposite (relax_pair2).
template <int ST>
struct PackedPair {
    unsigned v[2];
    template <int J>
    __device__ __forceinline__ void put(float2 x) { v[(J + 1) & 1] = Raw2<ST>::pack(x); }
};

template <int ST, int J, bool FORCED, class Slot>
__device__ __forceinline__ void relax_quad(typename Store<ST>::T* __restrict__ fout, unsigned S,
                                           unsigned site0, const Slot& slot,
                                           const PairState& pa, const PairState& pb,
                                           const float2 F[6], const CollideParams& cp,
                                           bool active) {
    unsigned ra[Q], rb[Q];   // only [J] and [J + 1] are used
    const Quad q0 = slot.template get<J>(), q1 = slot.template get<J + 1>();
    ra[J] = q0.a;
    ra[J + 1] = q1.a;
    rb[J] = q0.b;
    rb[J + 1] = q1.b;
    PackedPair<ST> a, b;
    relax_pair2<ST, J, FORCED>(a, ra, pa.k, pa.ux, pa.uy, pa.uz, F[0], F[1], F[2], pa.uF, cp);
    relax_pair2<ST, J, FORCED>(b, rb, pb.k, pb.ux, pb.uy, pb.uz, F[3], F[4], F[5], pb.uF, cp);
    if (active) {
        __stcs(reinterpret_cast<uint2*>(fout + ((unsigned)J * S + site0)), make_uint2(a.v[0], b.v[0]));
        __stcs(reinterpret_cast<uint2*>(fout + ((unsigned)(J + 1) * S + site0)),
               make_uint2(a.v[1], b.v[1]));
    }
}

// Forced relaxation of one pair of a quad: the first pair's results go back
// into the slot, the second's are stored together with them.
template <int ST, int J, bool SECOND, class Slot>
__device__ __forceinline__ void relax_half(typename Store<ST>::T* __restrict__ fout, unsigned S,
                                           unsigned site0, const Slot& slot,
                                           const PairState& p, const float2* F,
                                           const CollideParams& cp, bool active) {
    unsigned r[Q];   // only [J] and [J + 1] are used
    const Quad q0 = slot.template get<J>(), q1 = slot.template get<J + 1>();
    r[J] = SECOND ? q0.b : q0.a;
    r[J + 1] = SECOND ? q1.b : q1.a;
    PackedPair<ST> v;
    relax_pair2<ST, J, true>(v, r, p.k, p.ux, p.uy, p.uz, F[0], F[1], F[2], p.uF, cp);
    if (!SECOND) {
        slot.template put_a<J>(v.v[0]);
        slot.template put_a<J + 1>(v.v[1]);
    } else if (active) {
        __stcs(reinterpret_cast<uint2*>(fout + ((unsigned)J * S + site0)), make_uint2(q0.a, v.v[0]));
        __stcs(reinterpret_cast<uint2*>(fout + ((unsigned)(J + 1) * S + site0)),
               make_uint2(q1.a, v.v[1]));
    }
}

// Collision of a quad whose raw values are in A, B and in the slot.  Without
// force the two pairs' states fit the registers side by side; with it the raw
// values are read back (none are held through the force gather) and one pair
// is finished before the other begins.
template <int ST, bool FORCED, class Slot>
__device__ __forceinline__ void collide_quad(typename Store<ST>::T* __restrict__ fout, unsigned S,
                                             unsigned site0, const unsigned A[Q],
                                             const unsigned B[Q], const Slot& slot,
                                             const float2 F[6], const CollideParams& cp,
                                             int* flag, bool active) {
    const float2 om1 = f2(1.0f - cp.omega);
    if (!FORCED) {
        const PairState pa = pair_state<ST, false>(A, F[0], F[1], F[2], cp, flag, active);
        const PairState pb = pair_state<ST, false>(B, F[3], F[4], F[5], cp, flag, active);
        const Quad q = slot.template get<0>();
        if (active)
            __stcs(reinterpret_cast<uint2*>(fout + site0),
                   make_uint2(Raw2<ST>::pack(fma2(om1, Raw2<ST>::widen(q.a), pa.rest)),
                              Raw2<ST>::pack(fma2(om1, Raw2<ST>::widen(q.b), pb.rest))));
#define LBM_RQ(J) relax_quad<ST, J, false>(fout, S, site0, slot, pa, pb, F, cp, active)
        LBM_RQ(1); LBM_RQ(3); LBM_RQ(5); LBM_RQ(7); LBM_RQ(9);
        LBM_RQ(11); LBM_RQ(13); LBM_RQ(15); LBM_RQ(17);
#undef LBM_RQ
        return;
    }
#define LBM_RH(J, N) relax_half<ST, J, N>(fout, S, site0, slot, p, F + 3 * N, cp, active)
    {
        unsigned v[Q];
        slot.template get_all<0>(v);
        const PairState p = pair_state<ST, true>(v, F[0], F[1], F[2], cp, flag, active);
        slot.template put_a<0>(Raw2<ST>::pack(fma2(om1, Raw2<ST>::widen(slot.template get<0>().a), p.rest)));
        LBM_RH(1, 0); LBM_RH(3, 0); LBM_RH(5, 0); LBM_RH(7, 0); LBM_RH(9, 0);
        LBM_RH(11, 0); LBM_RH(13, 0); LBM_RH(15, 0); LBM_RH(17, 0);
    }
    {
        unsigned v[Q];
        slot.template get_all<1>(v);
        const PairState p = pair_state<ST, true>(v, F[3], F[4], F[5], cp, flag, active);
        const Quad q = slot.template get<0>();
        if (active)
            __stcs(reinterpret_cast<uint2*>(fout + site0),
                   make_uint2(q.a, Raw2<ST>::pack(fma2(om1, Raw2<ST>::widen(q.b), p.rest))));
        LBM_RH(1, 1); LBM_RH(3, 1); LBM_RH(5, 1); LBM_RH(7, 1); LBM_RH(9, 1);
        LBM_RH(11, 1); LBM_RH(13, 1); LBM_RH(15, 1); LBM_RH(17, 1);
    }
#undef LBM_RH
}

// The slot of this thread in s_raw[Q][threads of the CTA], filled with its raw
// values.
template <int PZV>
__device__ __forceinline__ QuadSlot<PZV> fill_slot(uint2* s_raw, const unsigned A[Q],
                                                   const unsigned B[Q]) {
    const int tid = (threadIdx.z * TY + threadIdx.y) * QX + threadIdx.x;
    const QuadSlot<PZV> slot{(unsigned)__cvta_generic_to_shared(s_raw + tid)};
#define LBM_SP(J) slot.template put<J>(A[J], B[J])
    LBM_SP(0); LBM_SP(1); LBM_SP(2); LBM_SP(3); LBM_SP(4); LBM_SP(5); LBM_SP(6);
    LBM_SP(7); LBM_SP(8); LBM_SP(9); LBM_SP(10); LBM_SP(11); LBM_SP(12); LBM_SP(13);
    LBM_SP(14); LBM_SP(15); LBM_SP(16); LBM_SP(17); LBM_SP(18);
#undef LBM_SP
    return slot;
}

// Eq. 21 of a tile with long lists, as gather_force_tab (same products and
// order) over the whole tile, in three parts per chunk of FORCE_CHUNK listed
// bubbles.  The first stages the records, straight into shared memory: for
// the first chunk it runs between the population loads and their use, so that
// its chain of dependent loads (list start, ids, records) hides behind theirs.
constexpr int QUAD_NAX = TX + TY + TZ;   // x: [0, TX), y: [TX, TX + TY), z: the rest
static_assert(FORCE_CHUNK == 32 && QX * TY == 32, "a lane per staged bubble, a warp per plane");

__device__ __forceinline__ void quad_force_stage(const int* __restrict__ items,
                                                 const BubbleRec* __restrict__ recs, int nb,
                                                 int c0, int cnt, BubbleRec* srec) {
    const int tid = (threadIdx.z * TY + threadIdx.y) * QX + threadIdx.x;
    if (tid < cnt) {
        const int id = __ldcg(items + c0 + tid);
        if (id >= 0 && id < nb) {
            const unsigned to = (unsigned)__cvta_generic_to_shared(srec + tid);
            const char* from = reinterpret_cast<const char*>(recs + id);
#pragma unroll
            for (int k = 0; k < (int)sizeof(BubbleRec); k += 16)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + k),
                             "l"(from + k) : "memory");
        } else {
            srec[tid] = BubbleRec{0, 0, 0, 0, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        }
    }
}

// The second tabulates their per-axis weights over the tile.  Every thread of
// the CTA calls it; the caller synchronises after it.
__device__ __forceinline__ void quad_force_tables(const Geo& g, int cnt, int bx, int by, int bz,
                                                  bool point, const BubbleRec* srec,
                                                  float (*s_w)[QUAD_NAX]) {
    const int tid = (threadIdx.z * TY + threadIdx.y) * QX + threadIdx.x;
    const int xb0 = bx * TX, yb0 = by * TY, zb0 = bz * TZ;
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    auto tabulate = [&](auto mode) {
        constexpr int PM = decltype(mode)::value;
        for (int e = tid; e < cnt * QUAD_NAX; e += QUAD_THREADS) {
            const int k = e / QUAD_NAX, q = e - k * QUAD_NAX;
            const BubbleRec& r = srec[k];
            if (q < TX)
                s_w[k][q] = axis_weight<PM>(r, xb0 + q, r.ax, r.fx, g.nx, !(g.walls & 0x01));
            else if (q < TX + TY)
                s_w[k][q] = axis_weight<PM>(r, yb0 + q - TX, r.ay, r.fy, g.ny, !(g.walls & 0x04));
            else
                s_w[k][q] =
                    axis_weight<PM>(r, zb0 + q - TX - TY, r.az, r.fz, g.nz, !(g.walls & 0x10));
        }
    };
    if (point) tabulate(MapMode<MAP_POINT>{});
    else tabulate(MapMode<MAP_CELL>{});
}

// The third adds the chunk to the force F on the thread's quad.  A warp is
// one z-plane, so it visits only the bubbles whose z weight there is not zero.
__device__ __forceinline__ void quad_force_add(int cnt, const BubbleRec* srec,
                                               const float (*s_w)[QUAD_NAX], float2 F[6]) {
    const int lane = threadIdx.y * QX + threadIdx.x;
    const int yi = TX + threadIdx.y, zi = TX + TY + threadIdx.z;
    unsigned todo = __ballot_sync(0xffffffffu, lane < cnt && s_w[lane < cnt ? lane : 0][zi] != 0.0f);
    while (todo) {
        const int k = __ffs(todo) - 1;
        todo &= todo - 1;
        const float wyz = s_w[k][yi] * s_w[k][zi];
        if (wyz == 0.0f) continue;
        const float4 wx = *reinterpret_cast<const float4*>(&s_w[k][4 * threadIdx.x]);
        const BubbleRec& r = srec[k];
        const float2 wa = make_float2(wx.x * wyz, wx.y * wyz);
        const float2 wb = make_float2(wx.z * wyz, wx.w * wyz);
        F[0] = fma2(wa, f2(r.px), F[0]);
        F[1] = fma2(wa, f2(r.py), F[1]);
        F[2] = fma2(wa, f2(r.pz), F[2]);
        F[3] = fma2(wb, f2(r.px), F[3]);
        F[4] = fma2(wb, f2(r.py), F[4]);
        F[5] = fma2(wb, f2(r.pz), F[5]);
    }
}

// One CTA's block of the sweep (sweep_block with four nodes per thread): 32 x 4
// nodes of PZV planes, a whole tile at PZV = 4.
template <int ST, bool TAB, int PZV = QUAD_PZ>
__device__ __forceinline__ void quad_block(const typename Store<ST>::T* __restrict__ fin,
                                           typename Store<ST>::T* __restrict__ fout,
                                           const Geo& g, const CollideParams& cp,
                                           const int* __restrict__ tile_start,
                                           const int* __restrict__ tile_count,
                                           const int* __restrict__ items, int cap,
                                           const BubbleRec* __restrict__ recs, int nb,
                                           int* __restrict__ flag, int bx, int by, int bz,
                                           BubbleRec* srec, const unsigned* safe,
                                           unsigned epoch, bool lead) {
    static_assert(TZ % PZV == 0 && (!TAB || PZV == QUAD_PZ), "a block lies in one tile layer");
    __shared__ uint2 s_raw[Q * QX * TY * PZV];
    const int x0 = bx * TX + 4 * threadIdx.x;
    const int y = by * TY + threadIdx.y;
    const int z = bz * PZV + threadIdx.z;
    const bool active = (x0 < g.nx) && (y < g.ny) && (z < g.nz);
    // Inactive threads gather at a valid node and store nothing.
    const int xa = active ? x0 : 0;
    const int ya = min(y, g.ny - 1), za = min(z, g.nz - 1);
    const int t = (((bz * PZV) / TZ) * g.nty + by) * g.ntx + bx;
    // The order of the tile count, the population loads and the wait for an
    // overlapped update is sweep_block's.
    int n_t = 0;
    bool skip = false;
    if (tile_count != nullptr) {
        if (safe == nullptr) n_t = __ldcg(tile_count + t);
        else skip = !lead && __ldcg(safe + (bz * PZV) / TZ) == epoch;
    }
    unsigned A[Q], B[Q];
    gather_quad<ST>(fin, g, xa, ya, za, A, B);
    if (tile_count != nullptr && safe != nullptr && !skip) {
        pdl_wait();
        n_t = __ldcg(tile_count + t);
    }
    __shared__ __align__(16) float s_w[TAB ? FORCE_CHUNK : 1][QUAD_NAX];
    int beg = 0, end = 0;
    if (n_t > 0) {   // uniform over the CTA (one tile)
        beg = __ldcg(tile_start + t);
        end = min(beg + n_t, cap);
        if (TAB) quad_force_stage(items, recs, nb, beg, min(FORCE_CHUNK, end - beg), srec);
    }
    const QuadSlot<PZV> slot = fill_slot<PZV>(s_raw, A, B);
    const unsigned S = (unsigned)g.S;
    const unsigned site0 = (unsigned)site_index(g, xa, ya, za);
    float2 F[6] = {f2(0.0f), f2(0.0f), f2(0.0f), f2(0.0f), f2(0.0f), f2(0.0f)};
    if (n_t > 0) {
        if (TAB) {
            for (int c0 = beg; c0 < end; c0 += FORCE_CHUNK) {
                const int cnt = min(FORCE_CHUNK, end - c0);
                if (c0 > beg) {
                    __syncthreads();   // the chunk before is done with
                    quad_force_stage(items, recs, nb, c0, cnt, srec);
                }
                quad_force_tables(g, cnt, bx, by, bz, cp.point != 0, srec, s_w);
                __syncthreads();
                quad_force_add(cnt, srec, s_w, F);
            }
        } else {
            const int tid = (threadIdx.z * TY + threadIdx.y) * QX + threadIdx.x;
            for (int c0 = beg; c0 < end; c0 += FORCE_CHUNK) {
                const int cnt = min(FORCE_CHUNK, end - c0);
                __syncthreads();
                if (tid < cnt) {
                    const int id = __ldcg(items + c0 + tid);
                    if (id >= 0 && id < nb) srec[tid] = load_rec(recs + id);
                    else srec[tid] = BubbleRec{0, 0, 0, 0, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
                }
                __syncthreads();
                if (active)
                    for (int k = 0; k < cnt; ++k) {
                        add_bubble_force_pair(srec[k], g, x0, y, z, F[0], F[1], F[2]);
                        add_bubble_force_pair(srec[k], g, x0 + 2, y, z, F[3], F[4], F[5]);
                    }
            }
        }
        collide_quad<ST, true>(fout, S, site0, A, B, slot, F, cp, flag, active);
    } else {
        collide_quad<ST, false>(fout, S, site0, A, B, slot, F, cp, flag, active);
    }
}

// The same of a block no bubble force reaches.
template <int ST>
__device__ __forceinline__ void quad_block_free(const typename Store<ST>::T* __restrict__ fin,
                                                typename Store<ST>::T* __restrict__ fout,
                                                const Geo& g, const CollideParams& cp,
                                                int* __restrict__ flag, int bx, int by, int bz) {
    __shared__ uint2 s_raw[Q * QUAD_THREADS];
    const int x0 = bx * TX + 4 * threadIdx.x;
    const int y = by * TY + threadIdx.y;
    const int z = bz * QUAD_PZ + threadIdx.z;
    const bool active = (x0 < g.nx) && (y < g.ny) && (z < g.nz);
    const int xa = active ? x0 : 0;
    const int ya = min(y, g.ny - 1), za = min(z, g.nz - 1);
    unsigned A[Q], B[Q];
    gather_quad<ST>(fin, g, xa, ya, za, A, B);
    const float2 F[6] = {f2(0.0f), f2(0.0f), f2(0.0f), f2(0.0f), f2(0.0f), f2(0.0f)};
    const QuadSlot<QUAD_PZ> slot = fill_slot<QUAD_PZ>(s_raw, A, B);
    collide_quad<ST, false>(fout, (unsigned)g.S, (unsigned)site_index(g, xa, ya, za), A, B, slot,
                            F, cp, flag, active);
}

// The form of a sweep kernel from its parameters behind ST, of which there are
// as many as lbm_sweep_kernel's names show: [4,] TAB for the listed sweep, [4]
// for the force-free one.
template <int... P> struct ListedForm;
template <int TAB> struct ListedForm<TAB> {
    static constexpr int kNodes = 2;
    static constexpr bool kTab = TAB != 0;
};
template <int NODES, int TAB> struct ListedForm<NODES, TAB> {
    static constexpr int kNodes = NODES;
    static constexpr bool kTab = TAB != 0;
};
template <int... N> struct FreeForm { static constexpr int kNodes = 2; };
template <int NODES> struct FreeForm<NODES> { static constexpr int kNodes = NODES; };

// kTab: the force gather of long tile lists (per-axis weight tables).  kNodes:
// nodes per thread along x (four: quad_block below).
template <int ST, int... P>
__global__ void __launch_bounds__(SweepShape<ST, ListedForm<P...>::kNodes>::kThreads,
                                  SweepShape<ST, ListedForm<P...>::kNodes>::kMinBlocks)
k_collide_stream_pair(const typename Store<ST>::T* __restrict__ fin,
                      typename Store<ST>::T* __restrict__ fout, Geo g, CollideParams cp,
                      const int* tile_start, const int* tile_count, const int* items, int cap,
                      const BubbleRec* recs, int nb, int* __restrict__ flag,
                      const unsigned* safe, unsigned epoch, const int* zperm, ZSpan zs) {
    constexpr bool TAB = ListedForm<P...>::kTab;
    __shared__ __align__(16) BubbleRec srec[FORCE_CHUNK];
    // The next bubble update may be scheduled once every CTA of the sweep has
    // started; it waits for the sweep to complete before it reads anything.
    pdl_trigger();
    // z blocks in the order the bubble update before chose (cleared layers
    // first; written by an update that has completed), else the span's.
    int bz = zs.first + (int)blockIdx.z;
    if (bz >= zs.hole) bz += zs.skip;
    if (zperm != nullptr) bz = __ldcg(zperm + blockIdx.z);
    const bool lead = (blockIdx.x | blockIdx.y | blockIdx.z) == 0;
    if constexpr (ListedForm<P...>::kNodes == 4)
        quad_block<ST, TAB>(fin, fout, g, cp, tile_start, tile_count, items, cap, recs, nb, flag,
                            blockIdx.x, blockIdx.y, bz, srec, safe, epoch, lead);
    else
        sweep_block<ST, TAB>(fin, fout, g, cp, tile_start, tile_count, items, cap, recs, nb, flag,
                             blockIdx.x, blockIdx.y, bz, srec, safe, epoch, lead);
}

// Sweeps without tile lists (no two-way coupling, or the blocks no bubble
// force reaches): the same gather and the same collision without force
// (collide_pair<ST, false>, as k_collide_stream_pair runs it for a block with
// an empty list), in a kernel without the force-gather code: the 16-bit
// sweep runs about 3 % faster in it than in k_collide_stream_pair.
template <int ST, int... N>
__global__ void __launch_bounds__(SweepShape<ST, FreeForm<N...>::kNodes>::kThreads,
                                  SweepShape<ST, FreeForm<N...>::kNodes>::kMinBlocks)
k_collide_stream_free(const typename Store<ST>::T* __restrict__ fin,
                      typename Store<ST>::T* __restrict__ fout, Geo g, CollideParams cp,
                      int* __restrict__ flag, ZSpan zs) {
    int bz = zs.first + (int)blockIdx.z;
    if (bz >= zs.hole) bz += zs.skip;
    if constexpr (FreeForm<N...>::kNodes == 4) {
        quad_block_free<ST>(fin, fout, g, cp, flag, blockIdx.x, blockIdx.y, bz);
        return;
    }
    const int x0 = blockIdx.x * TX + 2 * threadIdx.x;
    const int y = blockIdx.y * TY + threadIdx.y;
    const int z = bz * PZ + threadIdx.z;
    const bool active = (x0 < g.nx) && (y < g.ny) && (z < g.nz);
    // Inactive threads gather at a valid node and store nothing.
    const int xa = active ? x0 : 0;
    const int ya = min(y, g.ny - 1), za = min(z, g.nz - 1);
    const unsigned nx = (unsigned)g.nx, nxy = (unsigned)g.nx * (unsigned)g.ny;
    const unsigned site0 = (unsigned)za * nxy + (unsigned)ya * nx + (unsigned)xa;
    typename Raw2<ST>::T rv[Q];
    gather_pair<ST>(fin, g, xa, ya, za, rv);
    PairStore<ST> sink{fout, (unsigned)g.S, site0, active};
    collide_pair<ST, false>(sink, rv, f2(0.0f), f2(0.0f), f2(0.0f), cp, flag, active);
}

// ---------------------------------------------------------------------------
// Batched sweep: many independent columns in one persistent launch.  Each CTA
// takes work items -- `depth` consecutive z-blocks of one (column, x-block,
// y-block) -- from a global counter until all are done; columns keep their
// own size, omega and walls.  Results do not depend on which CTA takes which
// item.
// ---------------------------------------------------------------------------
constexpr int MAX_BATCH_COLUMNS = 256;

// NODES: nodes per thread along x, as the single sweep's (four where every
// column's rows are a multiple of 4 of 16-bit values).
template <int ST, int PZV, int NODES>
__global__ void __launch_bounds__(SweepShape<ST, NODES>::kThreads / SweepShape<ST, NODES>::kPlanes * PZV,
                                  SweepShape<ST, NODES>::kMinBlocks * SweepShape<ST, NODES>::kPlanes / PZV)
k_collide_batch(const typename Store<ST>::T* __restrict__ fin,
                typename Store<ST>::T* __restrict__ fout, const BatchColumn* __restrict__ cols,
                int ncols, int total_items, int depth, int* __restrict__ work_counter,
                const int* __restrict__ tile_start, const int* __restrict__ tile_count,
                const int* __restrict__ items, int cap, const BubbleRec* __restrict__ recs,
                int nb, int* __restrict__ flag) {
    __shared__ BubbleRec srec[FORCE_CHUNK];
    __shared__ int s_item_base[MAX_BATCH_COLUMNS + 1];
    __shared__ int s_item;
    const int tid = (threadIdx.z * TY + threadIdx.y) * (TX / NODES) + threadIdx.x;
    for (int c = tid; c <= ncols; c += TX / NODES * TY * PZV)
        s_item_base[c] = c < ncols ? cols[c].item_base : total_items;
    for (;;) {
        __syncthreads();
        if (tid == 0) s_item = atomicAdd(work_counter, 1);
        __syncthreads();
        const int item = s_item;
        if (item >= total_items) break;
        int lo = 0, hi = ncols - 1;   // column with item_base <= item < next base
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (s_item_base[mid] <= item) lo = mid;
            else hi = mid - 1;
        }
        const BatchColumn& col = cols[lo];
        const int local = item - s_item_base[lo];
        const int bx = local % col.g.ntx;
        const int rest = local / col.g.ntx;
        const int by = rest % col.g.nty;
        const int bz0 = (rest / col.g.nty) * depth;
        const int nbz = (col.g.nz + PZV - 1) / PZV;
        // No lists (no two-way coupling): null stays null.
        const int* const start = tile_start ? tile_start + col.tile_base : nullptr;
        const int* const count = tile_count ? tile_count + col.tile_base : nullptr;
        for (int bz = bz0; bz < min(bz0 + depth, nbz); ++bz) {
            if constexpr (NODES == 4)
                quad_block<ST, false, PZV>(fin + col.pop_offset, fout + col.pop_offset, col.g,
                                           col.cp, start, count, items, cap, recs, nb, flag, bx, by,
                                           bz, srec, nullptr, 0, false);
            else
                sweep_block<ST, false, PZV>(fin + col.pop_offset, fout + col.pop_offset, col.g,
                                            col.cp, start, count, items, cap, recs, nb, flag, bx,
                                            by, bz, srec);
        }
    }
}

cudaError_t launch_collide_batch(int storage, const void* fin, void* fout,
                                 const BatchColumn* cols, int ncols, int total_items, int depth,
                                 int grid, int planes, bool quad, int* work_counter,
                                 const TileLists& tl, const BubbleRec* recs, int nb, int* flag,
                                 cudaStream_t st) {
    if (ncols > MAX_BATCH_COLUMNS) return cudaErrorInvalidValue;
    if (quad && storage != 0) {
        switch (storage * 8 + planes) {
#define LBM_LAUNCH_BATCH4(SI, PV, T)                                                              \
    case SI * 8 + PV:                                                                             \
        k_collide_batch<SI, PV, 4><<<grid, dim3(QX, TY, PV), 0, st>>>(                            \
            (const T*)fin, (T*)fout, cols, ncols, total_items, depth, work_counter, tl.start,    \
            tl.count, tl.items, tl.cap, recs, nb, flag);                                         \
        break;
            LBM_LAUNCH_BATCH4(1, 1, __half)
            LBM_LAUNCH_BATCH4(1, 2, __half)
            LBM_LAUNCH_BATCH4(1, 4, __half)
            LBM_LAUNCH_BATCH4(2, 1, __nv_bfloat16)
            LBM_LAUNCH_BATCH4(2, 2, __nv_bfloat16)
            LBM_LAUNCH_BATCH4(2, 4, __nv_bfloat16)
#undef LBM_LAUNCH_BATCH4
            default:
                return cudaErrorInvalidValue;
        }
        return cudaGetLastError();
    }
    switch (storage * 8 + planes) {
#define LBM_LAUNCH_BATCH(SI, PV, T)                                                               \
    case SI * 8 + PV:                                                                             \
        k_collide_batch<SI, PV, 2><<<grid, dim3(PX, TY, PV), 0, st>>>(                            \
            (const T*)fin, (T*)fout, cols, ncols, total_items, depth, work_counter, tl.start,    \
            tl.count, tl.items, tl.cap, recs, nb, flag);                                         \
        break;
        LBM_LAUNCH_BATCH(0, 1, float)
        LBM_LAUNCH_BATCH(0, 2, float)
        LBM_LAUNCH_BATCH(0, 4, float)
        LBM_LAUNCH_BATCH(1, 1, __half)
        LBM_LAUNCH_BATCH(1, 2, __half)
        LBM_LAUNCH_BATCH(1, 4, __half)
        LBM_LAUNCH_BATCH(2, 1, __nv_bfloat16)
        LBM_LAUNCH_BATCH(2, 2, __nv_bfloat16)
        LBM_LAUNCH_BATCH(2, 4, __nv_bfloat16)
#undef LBM_LAUNCH_BATCH
        default:
            return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

int sweep_planes(int storage, int nx, const void* fa, const void* fb) {
    // Four nodes per thread wherever rows of 16-bit values can be read 8
    // bytes at a time.
    const bool quad = storage != 0 && (nx & 3) == 0 && ((uintptr_t)fa & 7) == 0 &&
                      ((uintptr_t)fb & 7) == 0;
    return (nx & 1) ? ODD_PZ : (quad ? QUAD_PZ : PZ);
}
int batch_min_blocks(int storage, int planes, bool quad) {
    if (quad) return SweepShape<1, 4>::kMinBlocks * QUAD_PZ / planes;
    const int k = storage == 0 ? PairOccupancy<0>::kMinBlocks : PairOccupancy<1>::kMinBlocks;
    return k * PZ / planes;
}

cudaError_t launch_collide_stream(int storage, const void* fin, void* fout, const Geo& g,
                                  const CollideParams& cp, const TileLists* tl,
                                  const BubbleRec* recs, int nb, int* flag, const unsigned* safe,
                                  unsigned epoch, bool overlap, const int* zperm,
                                  cudaStream_t st, const ZSpan* span) {
    const int* start = tl ? tl->start : nullptr;
    const int* count = tl ? tl->count : nullptr;
    const int* items = tl ? tl->items : nullptr;
    const int cap = tl ? tl->cap : 0;
    if (overlap && (safe == nullptr || tl == nullptr)) return cudaErrorInvalidValue;
    if (!overlap) safe = nullptr;
    const int planes = sweep_planes(storage, g.nx, fin, fout);
    const bool quad = planes == QUAD_PZ;
    const int nbz = (g.nz + planes - 1) / planes;
    ZSpan zs{0, nbz, INT_MAX, 0};
    if (span) {
        if ((g.nx & 1) || zperm || span->count < 0 || span->first < 0 || span->skip < 0 ||
            span->first + span->count + span->skip > nbz)
            return cudaErrorInvalidValue;
        zs = *span;
        if (zs.count == 0) return cudaSuccess;
    }
    if ((g.nx & 1) == 0) {
        // Even rows: two nodes per thread with aligned vector accesses.  Tile
        // lists longer than the few-bubble path's (many bubbles per tile)
        // take the tabulated force gather.
        cudaLaunchConfig_t cfg = {};
        cfg.blockDim = quad ? dim3(QX, TY, QUAD_PZ) : dim3(PX, TY, PZ);
        cfg.gridDim = dim3((g.nx + TX - 1) / TX, (g.ny + TY - 1) / TY, (unsigned)zs.count);
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = overlap ? 1 : 0;
        if (tl == nullptr && zperm == nullptr && !overlap) {
            // No bubble force reaches these blocks.
            if (quad && storage == 1)
                return cudaLaunchKernelEx(&cfg, k_collide_stream_free<1, 4>, (const __half*)fin,
                                          (__half*)fout, g, cp, flag, zs);
            if (quad)
                return cudaLaunchKernelEx(&cfg, k_collide_stream_free<2, 4>,
                                          (const __nv_bfloat16*)fin, (__nv_bfloat16*)fout, g, cp,
                                          flag, zs);
            switch (storage) {
                case 0:
                    return cudaLaunchKernelEx(&cfg, k_collide_stream_free<0>, (const float*)fin,
                                              (float*)fout, g, cp, flag, zs);
                case 1:
                    return cudaLaunchKernelEx(&cfg, k_collide_stream_free<1>, (const __half*)fin,
                                              (__half*)fout, g, cp, flag, zs);
                default:
                    return cudaLaunchKernelEx(&cfg, k_collide_stream_free<2>,
                                              (const __nv_bfloat16*)fin, (__nv_bfloat16*)fout, g,
                                              cp, flag, zs);
            }
        }
        const bool tab = tl != nullptr && tl->cap > SMALL_MAX_PAIRS;
        if (quad) {
            switch (storage * 2 + (tab ? 1 : 0)) {
#define LBM_LAUNCH_QUAD(SI, TB, T)                                                                \
    case SI * 2 + TB:                                                                             \
        return cudaLaunchKernelEx(&cfg, k_collide_stream_pair<SI, 4, TB>, (const T*)fin, (T*)fout,   \
                                  g, cp, start, count, items, cap, recs, nb, flag, safe, epoch,  \
                                  zperm, zs);
                LBM_LAUNCH_QUAD(1, 0, __half)
                LBM_LAUNCH_QUAD(1, 1, __half)
                LBM_LAUNCH_QUAD(2, 0, __nv_bfloat16)
                LBM_LAUNCH_QUAD(2, 1, __nv_bfloat16)
#undef LBM_LAUNCH_QUAD
                default:
                    return cudaErrorInvalidValue;
            }
        }
        switch (storage * 2 + (tab ? 1 : 0)) {
#define LBM_LAUNCH_PAIR(SI, TB, T)                                                                \
    case SI * 2 + TB:                                                                             \
        return cudaLaunchKernelEx(&cfg, k_collide_stream_pair<SI, TB>, (const T*)fin, (T*)fout,   \
                                  g, cp, start, count, items, cap, recs, nb, flag, safe, epoch,  \
                                  zperm, zs);
            LBM_LAUNCH_PAIR(0, 0, float)
            LBM_LAUNCH_PAIR(0, 1, float)
            LBM_LAUNCH_PAIR(1, 0, __half)
            LBM_LAUNCH_PAIR(1, 1, __half)
            LBM_LAUNCH_PAIR(2, 0, __nv_bfloat16)
            LBM_LAUNCH_PAIR(2, 1, __nv_bfloat16)
#undef LBM_LAUNCH_PAIR
            default:
                return cudaErrorInvalidValue;
        }
    }
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(TX, TY, 1);
    cfg.gridDim = dim3((g.nx + TX - 1) / TX, (g.ny + TY - 1) / TY, (unsigned)nbz);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = overlap ? 1 : 0;
    switch (storage) {
        case 0:
            return cudaLaunchKernelEx(&cfg, k_collide_stream<0>, (const float*)fin, (float*)fout, g,
                                      cp, start, count, items, cap, recs, nb, flag, safe, epoch,
                                      zperm);
        case 1:
            return cudaLaunchKernelEx(&cfg, k_collide_stream<1>, (const __half*)fin, (__half*)fout,
                                      g, cp, start, count, items, cap, recs, nb, flag, safe, epoch,
                                      zperm);
        default:
            return cudaLaunchKernelEx(&cfg, k_collide_stream<2>, (const __nv_bfloat16*)fin,
                                      (__nv_bfloat16*)fout, g, cp, start, count, items, cap, recs,
                                      nb, flag, safe, epoch, zperm);
    }
}

}  // namespace lbm
