// godunov_fine on a complete level, FP32 path: the column-per-thread ("pencil") form of
// the z-column update.
//
// A CTA owns a 16 x 16-cell footprint of the level and marches segments of its column in z
// one cell plane at a time.  Twelve warps in three roles, one barrier per plane:
//   eight interior warps, a thread per (x, y) column.  Plane p, before the barrier:
//     B  slopes and MUSCL-Hancock predictor of plane p from a ring of four planes of
//        primitives (20 x 20 cells); the -x, -y, +z and -z face states stay in registers, +x
//        and +y go to shared memory;
//     C  the z face below plane p from two states the thread holds (no shared memory);
//   after it:
//     D  the x and y faces on the left of and below the thread's cell of plane p (left states
//        from shared memory, right states from registers), published;
//     E  FP64 update of plane p-1: x and y fluxes from shared memory, z fluxes from registers;
//   two gathering warps: the FP64 states of stencil plane p+2 to FP32 primitives in the ring,
//     loads three items ahead of the conversions;
//   two warps: the restriction of the planes updated before (children in cell order), the
//     predictor of the four one-cell strips around the footprint and the faces on its right
//     and top edges, the last 16 gather items, the oct ids of the layers ahead.
// Shared buffers alternate with the plane's parity.  Per cell the arithmetic is the tile
// kernel's, in the same order (gather conversion, predictor, face states, Riemann solve, flux
// sum x-left, x-right, y-left, y-right, z-below, z-above, FP64 update, CFL candidate,
// restriction), so the states are bitwise those of the other kernels.
//
// Bound: latency and issue, not bandwidth (0.83 ms for 1.34 GB of algorithmic traffic at 256^3;
// issue 52% active, 31.2 warp instructions per update, 24 warps per SM at 80 registers).  A
// single role of 256 threads needed 128 registers (the gather's FP64 loads live across the
// predictor): 16 warps per SM, 37.9 warp instructions per update.  256^3 step on a GB300: 1.137
// ms with one role; 1.03 with the roles; 0.97 with look-ups a plane ahead of their use and the
// L2 prefetch; 0.93 without a branch in the Riemann solver; 0.91 with the range clamps of the
// conversions in one instruction and the CFL step from the largest signal speed; 0.88 with the
// restriction first in its warps' iteration (0.866 with the restriction launches below it by
// variable).  At 0.91, without the gather's loads it would take 0.80, without restriction 0.80,
// without the old states' loads 0.85, without x and y faces 0.86.
#pragma once
#include <type_traits>
#include "godunov_col.cuh"

namespace amr {

struct PenGeo {
    static constexpr int FX = 16, FY = 16;            // footprint (cells)
    static constexpr int SX = FX + 4, SY = FY + 4;    // stencil plane (cells)
    static constexpr int NS = SX * SY;                // 400
    static constexpr int NI = FX * FY;                // 256 interior columns = interior threads
    static constexpr int OX = SX / 2, NO = OX * (SY / 2);   // footprint oct columns (10 x 10)
    static constexpr int NA = 64, NB = 64;            // gathering threads; edge, strip and restriction threads
    static constexpr int NT = NI + NA + NB;
};

template <bool FINER> struct PenSmem {
    using G = PenGeo;
    // primitive stencil planes, ring slot = plane & 3: (rho, u, v, w) and p
    float4 Wv[4][G::NS];
    float Wp[4][G::NS];
    // face states in the face-normal frame, by plane parity:
    //   Sx: +x states of interior cell x + 16 y, the left strip's at NI + y;
    //   Sy: +y states of interior cells, the bottom strip's at NI + x;
    //   Sr: -x states of the right strip (row y at y), -y of the top strip (column x at 16 + x)
    float4 Sx4[2][G::NI + 16];
    float Sx1[2][G::NI + 16];
    float4 Sy4[2][G::NI + 16];
    float Sy1[2][G::NI + 16];
    float4 Sr4[2][32];
    float Sr1[2][32];
    // fluxes (face-normal frame) by plane parity: the face on the left of x (x = 16: the right
    // edge) at x + 17 y; the face below y (y = 16: the top edge) at x + 16 y
    float4 Gx4[2][G::NI + 16];
    float Gx1[2][G::NI + 16];
    float4 Gy4[2][G::NI + 16];
    float Gy1[2][G::NI + 16];
    double Ur[2][NV][G::NI];                          // new states by plane parity, [variable][x + 16 y]
    int32_t oct[8][G::NO];                            // oct id per footprint oct column, slot = layer & 7
    uint8_t ref[FINER ? 8 : 1][FINER ? G::NS : 1];    // refined flag per stencil cell, slot = plane & 7
};

__device__ __forceinline__ void pen_ld(const float4 *a4, const float *a1, int i, float W[NV])
{
    const float4 q = a4[i];
    W[0] = q.x; W[1] = q.y; W[2] = q.z; W[3] = q.w; W[4] = a1[i];
}

__device__ __forceinline__ void pen_st(float4 *a4, float *a1, int i, const float W[NV])
{
    a4[i] = make_float4(W[0], W[1], W[2], W[3]);
    a1[i] = W[4];
}

// dU += s F for the face-normal flux Fn of a face of direction D
template <int D> __device__ __forceinline__ void pen_acc(float dU[NV], const float Fn[NV], bool plus)
{
    constexpr int N0 = D + 1, T1 = D == 0 ? 2 : 1, T2 = D == 2 ? 2 : 3;
    float F[NV];
    F[0] = Fn[0]; F[N0] = Fn[1]; F[T1] = Fn[2]; F[T2] = Fn[3]; F[4] = Fn[4];
#pragma unroll
    for (int v = 0; v < NV; ++v) dU[v] = plus ? dU[v] + F[v] : dU[v] - F[v];
}

// One barrier per plane, for both roles
__device__ __forceinline__ void pen_barrier() { asm volatile("bar.sync 1, %0;" ::"n"(PenGeo::NT) : "memory"); }

// BATCH: the box batch (its own instantiation: in octree mode the segment's geometry is then
// the same for every thread as far as the compiler can see, and stays out of the threads'
// registers)
template <int RS, bool FINER, bool BATCH>
__global__ void __launch_bounds__(PenGeo::NT, 2) k_godunov_pen(ColArgs a)
{
    using G = PenGeo;
    using S = PenSmem<FINER>;
    constexpr int SX = G::SX;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    S &sm = *reinterpret_cast<S *>(smem_raw);
    const TreeView &tv = a.tv;
    const int tid = threadIdx.x, lane = tid & 31;
    Prm<float> pr;
    pr.gamma = d2f_bits(a.gamma); pr.rho_floor = d2f_bits(a.rho_floor); pr.p_floor = d2f_bits(a.p_floor);
    const bool per[3] = {tv.bc[0] == AMR_BC_PERIODIC, tv.bc[2] == AMR_BC_PERIODIC, tv.bc[4] == AMR_BC_PERIODIC};
    unsigned long long my_dt = ~0ull;

    const int64_t gend = min((int64_t(blockIdx.x) + 1) * a.share, a.planes);
    for (int64_t g = blockIdx.x * a.share; g < gend;) {
        // ---- geometry of this segment: the level (or box), footprint and z range
        int64_t n = a.n, plane0 = 0;
        int32_t obase = 0;
        double dx, lam;
        double *dtn = a.dt_next;
        if constexpr (BATCH) {
            // box offsets in planes of 16 x 16 columns: four per 8 x 8 x 16 item of the tree
            int lo = 0, hi = a.n_inst - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (a.inst_col_off[mid] * 4 <= g) lo = mid; else hi = mid - 1;
            }
            n = tv.inst_n[lo];
            plane0 = a.inst_col_off[lo] * 4;
            obase = int32_t(a.inst_oct_off[lo]);
            dx = tv.inst_dx[lo];
            lam = a.dt[lo] * double(n);
            dtn = a.dt_next ? a.dt_next + lo : nullptr;
        } else {
            dx = pow2(-a.level);
            lam = scale_pow2(*a.dt, a.level);   // dt / dx, exact
        }
        const float lamR = d2f_bits(lam), hl = 0.5f * lamR;
        const int ni = int(n), nf = ni / G::FX;
        const ColSeg seg = next_segment(plane0, g, gend, ni, a.zc);
        g = a.zc > 0 ? gend : g + (seg.z1 - seg.z0);                           // zc: one segment per CTA
        const int X0 = (seg.col % nf) * G::FX - 2, Y0 = (seg.col / nf) * G::FY - 2;   // stencil index 0
        const int z0 = seg.z0, z1 = seg.z1;                                    // planes [z0, z1)
        const int32_t Mi = ni / 2;
        auto wrap = [&](int c, int axis) -> int {
            if (c >= 0 && c < ni) return c;
            if (per[axis]) return c < 0 ? c + ni : c - ni;
            return c < 0 ? 0 : ni - 1;
        };
        // oct ids of the footprint's oct columns at oct layer L (wrapped or clamped like the cells)
        auto oct_of = [&](int L, int o) -> int32_t {
            const int wx = wrap(X0 + 2 * (o % G::OX), 0), wy = wrap(Y0 + 2 * (o / G::OX), 1);
            const int32_t oi = (wx >> 1) + Mi * ((wy >> 1) + Mi * (wrap(2 * L, 2) >> 1));
            return BATCH ? obase + oi : a.grid[oi];
        };
        // gather items: stencil cell q (quads of the 2 x 2 cells of one oct column, so four
        // lanes read 32 contiguous bytes of a variable): packed stencil index | oct column
        // << 9 | x-y cell bits << 16
        auto gitem = [&](int q) -> int {
            const int o = q >> 2, sub = q & 3;
            const int i = 2 * (o % G::OX) + (sub & 1), j = 2 * (o / G::OX) + (sub >> 1);
            const int cb = (wrap(X0 + i, 0) & 1) + 2 * (wrap(Y0 + j, 1) & 1);
            return (i + SX * j) | (o << 9) | (cb << 16);
        };
        // load of gather item pk of stencil plane z (FP64 state), then conversion and store
        auto gload = [&](int pk, int z, double U[NV]) -> int32_t {
            const int o = (pk >> 9) & 127, cb = pk >> 16;
            const int32_t cid = sm.oct[(z >> 1) & 7][o] * 8 + cb + 4 * (wrap(z, 2) & 1);
#pragma unroll
            for (int v = 0; v < NV; ++v) U[v] = a.uo[v][cid];
            return cid;
        };
        auto gstore = [&](int pk, int z, const double U[NV], int32_t cid) {
            const int si = pk & 511;
            float Uw[NV], Wc[NV];
#pragma unroll
            for (int v = 0; v < NV; ++v) Uw[v] = d2f_ftz(U[v]);
            cons_to_prim_w(Uw, pr, Wc);
            pen_st(sm.Wv[z & 3], sm.Wp[z & 3], si, Wc);
            if constexpr (FINER) sm.ref[z & 7][si] = (tv.refmask[cid >> 3] >> (cid & 7)) & 1;
        };
        // slopes + predictor of stencil cell si of plane p
        auto predict = [&](int p, int si, float Wt[NV], float Dl[3][NV]) {
            const int s0 = p & 3, sm1 = (p - 1) & 3, sp1 = (p + 1) & 3;
            float Wc[NV], Wa[NV], Wb[NV];
            pen_ld(sm.Wv[s0], sm.Wp[s0], si, Wc);
            pen_ld(sm.Wv[s0], sm.Wp[s0], si - 1, Wa);
            pen_ld(sm.Wv[s0], sm.Wp[s0], si + 1, Wb);
#pragma unroll
            for (int v = 0; v < NV; ++v) Dl[0][v] = minmod(Wc[v] - Wa[v], Wb[v] - Wc[v]);
            pen_ld(sm.Wv[s0], sm.Wp[s0], si - SX, Wa);
            pen_ld(sm.Wv[s0], sm.Wp[s0], si + SX, Wb);
#pragma unroll
            for (int v = 0; v < NV; ++v) Dl[1][v] = minmod(Wc[v] - Wa[v], Wb[v] - Wc[v]);
            pen_ld(sm.Wv[sm1], sm.Wp[sm1], si, Wa);
            pen_ld(sm.Wv[sp1], sm.Wp[sp1], si, Wb);
#pragma unroll
            for (int v = 0; v < NV; ++v) Dl[2][v] = minmod(Wc[v] - Wa[v], Wb[v] - Wc[v]);
            muscl_predict(Wc, Dl, hl, pr.gamma, Wt);
        };

        // ---- prologue, all threads: oct tables of layers z0/2-1 .. z0/2+3, planes z0-2 .. z0
        for (int w = tid; w < 5 * G::NO; w += G::NT) {
            const int L = z0 / 2 - 1 + w / G::NO;
            sm.oct[L & 7][w % G::NO] = oct_of(L, w % G::NO);
        }
        pen_barrier();
        for (int w = tid; w < 3 * G::NS; w += G::NT) {
            const int pk = gitem(w % G::NS), z = z0 - 2 + w / G::NS;
            double U[NV];
            const int32_t cid = gload(pk, z, U);
            gstore(pk, z, U, cid);
        }
        pen_barrier();

        if (tid >= G::NI + G::NA) {
            const int ht = tid - G::NI - G::NA, hw = ht >> 5;
            const int gpk = gitem(6 * G::NA + (ht & 15));
            // edge faces of plane p, first warp: lane l < 16 the right face of row l, else the top
            // face of column l - 16
            auto edges = [&](int p) {
                const int pb = p & 1, r = lane & 15;
                float WL[NV], WR[NV], Fn[NV];
                if (lane < 16) pen_ld(sm.Sx4[pb], sm.Sx1[pb], (G::FX - 1) + G::FX * r, WL);
                else pen_ld(sm.Sy4[pb], sm.Sy1[pb], r + G::FX * (G::FY - 1), WL);
                pen_ld(sm.Sr4[pb], sm.Sr1[pb], lane, WR);
                col_solve<float, RS>(WL, WR, pr, a.status, Fn);
                if (lane < 16) pen_st(sm.Gx4[pb], sm.Gx1[pb], G::FX + (G::FX + 1) * r, Fn);
                else pen_st(sm.Gy4[pb], sm.Gy1[pb], r + G::FX * G::FY, Fn);
            };
            // strips of plane p, a warp per axis: the left (lanes 0-15, +x state) and right (-x)
            // neighbour of row lane & 15; the bottom (+y) and top (-y) neighbour of column lane & 15
            auto strips = [&](int p) {
                const bool lo = lane < 16;
                const float half = lo ? 0.5f : -0.5f;
                const int r = lane & 15, pb = p & 1;
                float Wt[NV], Dl[3][NV], st[NV];
                if (hw == 0) {
                    predict(p, (lo ? 1 : G::FX + 2) + SX * (2 + r), Wt, Dl);
                    face_state<0>(Wt, Dl[0], half, pr, st);
                    if (lo) pen_st(sm.Sx4[pb], sm.Sx1[pb], G::NI + r, st);
                    else pen_st(sm.Sr4[pb], sm.Sr1[pb], r, st);
                } else {
                    predict(p, (2 + r) + SX * (lo ? 1 : G::FY + 2), Wt, Dl);
                    face_state<1>(Wt, Dl[1], half, pr, st);
                    if (lo) pen_st(sm.Sy4[pb], sm.Sy1[pb], G::NI + r, st);
                    else pen_st(sm.Sr4[pb], sm.Sr1[pb], 16 + r, st);
                }
            };
            // restriction: thread ht takes oct ht of the layer; the four children of plane q
            // added in cell order, the mean written after the layer's second plane
            const int ox = ht & 7, oy = ht >> 3;
            double acc[NV];
            int32_t father = 0;                        // of the layer's oct
            uint8_t fused = 0;                         // whether it is restricted here
            auto restrict_plane = [&](int q) {
                if (!(q & 1)) {
                    // looked up a plane before it is used
                    const int32_t oct = sm.oct[(q >> 1) & 7][(ox + 1) + G::OX * (oy + 1)];
                    father = tv.father[oct];
                    fused = tv.fused[oct];
                }
                const double *U = sm.Ur[q & 1][0] + 2 * ox + G::FX * 2 * oy;
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    const double2 c0 = *reinterpret_cast<const double2 *>(U + v * G::NI);
                    const double2 c2 = *reinterpret_cast<const double2 *>(U + v * G::NI + G::FX);
                    // (0 + c0) + c1 ... in cell order: the first addition changes nothing
                    const double s = (q & 1) ? (acc[v] + c0.x) + c0.y : c0.x + c0.y;
                    acc[v] = (s + c2.x) + c2.y;
                }
                if ((q & 1) && fused) {
#pragma unroll
                    for (int v = 0; v < NV; ++v) a.un[v][father] = 0.125 * acc[v];
                }
            };
            int32_t oct0 = 0, oct1 = 0;
            for (int p = z0 - 1; p <= z1; ++p) {
                double Ug[NV];
                int32_t cid = 0;
                const bool last_items = hw == 1 && lane < 16 && p < z1;
                if (last_items) cid = gload(gpk, p + 2, Ug);
                // oct table of layer (p+7)/2 (p odd), looked up in one plane, stored in the next,
                // read by the gather four planes on
                if (p & 1) {
                    const int L = min((p + 7) >> 1, (z1 + 1) >> 1);
                    oct0 = oct_of(L, ht);
                    if (ht < G::NO - G::NB) oct1 = oct_of(L, ht + G::NB);
                } else if (p + 6 <= z1 + 1) {
                    sm.oct[((p + 6) >> 1) & 7][ht] = oct0;
                    if (ht < G::NO - G::NB) sm.oct[((p + 6) >> 1) & 7][ht + G::NB] = oct1;
                }
                if (!BATCH && p - 3 >= z0) restrict_plane(p - 3);
                if (hw == 0 && p > z0) edges(p - 1);
                if (p >= z0 && p < z1) strips(p);
                if (last_items) gstore(gpk, p + 2, Ug, cid);
                pen_barrier();
            }
            if (!BATCH) restrict_plane(z1 - 2);
            pen_barrier();
            if (!BATCH) restrict_plane(z1 - 1);
        } else if (tid >= G::NI) {
            // gather, two warps: six items a thread and plane, loads three items ahead of the
            // conversions, across planes too
            const int ht = tid - G::NI;
            int gpk[6];
#pragma unroll
            for (int i = 0; i < 6; ++i) gpk[i] = gitem(ht + G::NA * i);
            double Ug[3][NV];
            int32_t cid[3];
#pragma unroll
            for (int i = 0; i < 3; ++i) cid[i] = gload(gpk[i], z0 + 1, Ug[i]);
            for (int p = z0 - 1; p <= z1; ++p) {
                if (p < z1) {
                    const int z = p + 2;
#pragma unroll
                    for (int i = 0; i < 6; ++i) {
                        gstore(gpk[i], z, Ug[i % 3], cid[i % 3]);
                        if (i < 3) cid[i] = gload(gpk[i + 3], z, Ug[i]);
                        else if (z <= z1) cid[i - 3] = gload(gpk[i - 3], z + 1, Ug[i - 3]);
                    }
                }
                pen_barrier();
            }
            pen_barrier();
        } else {
            const int x = lane & 15, y = 2 * (tid >> 5) + (lane >> 4);    // interior column
            const int ci = x + G::FX * y;                                   // its interior index
            const int sio = (x + 2) + SX * (y + 2);                         // its stencil index
            const int oo = ((x + 2) >> 1) + G::OX * ((y + 2) >> 1);         // its footprint oct column
            const int cxy = (x & 1) + 2 * (y & 1);                          // its cell bits in x and y
            const float cflR = d2f_bits(a.cfl), dxR = d2f_bits(dx);
            float pz[NV], fz[NV];                                           // thread state between planes
#pragma unroll
            for (int v = 0; v < NV; ++v) { pz[v] = 0.f; fz[v] = 0.f; }
            float sig = 0.f;                                                // largest signal speed met
            // plane p: MID: its faces are solved; UPD: plane p - 1 is updated
            auto plane = [&](auto upd_c, auto mid_c, int p) {
                constexpr bool UPD = decltype(upd_c)::value, MID = decltype(mid_c)::value;
                const int q = p - 1, pb = p & 1, qb = q & 1;
                float mx[NV], my[NV], fzp[NV];
                {
                    // ---- B: predictor of the thread's cell
                    float Wt[NV], Dl[3][NV];
                    predict(p, sio, Wt, Dl);
                    if (MID) {
                        float st[NV];
                        face_state<0>(Wt, Dl[0], 0.5f, pr, st);
                        pen_st(sm.Sx4[pb], sm.Sx1[pb], ci, st);
                        face_state<1>(Wt, Dl[1], 0.5f, pr, st);
                        pen_st(sm.Sy4[pb], sm.Sy1[pb], ci, st);
                        face_state<0>(Wt, Dl[0], -0.5f, pr, mx);
                        face_state<1>(Wt, Dl[1], -0.5f, pr, my);
                    }
                    if (UPD || MID) {
                        // ---- C: the z face below plane p
                        float mz[NV], Fn[NV];
                        face_state<2>(Wt, Dl[2], -0.5f, pr, mz);
                        col_solve<float, RS>(pz, mz, pr, a.status, Fn);
#pragma unroll
                        for (int v = 0; v < NV; ++v) { fzp[v] = fz[v]; fz[v] = Fn[v]; }
                    }
                    if (!UPD || MID) face_state<2>(Wt, Dl[2], 0.5f, pr, pz);
                }
                // L2 prefetch of oct layer (p+4)/2 (stencil planes p+4 and p+5): the two 32-byte
                // sectors of each oct's 64-byte row per variable
                if (!(p & 1) && p + 4 <= z1 + 1 && tid < G::NO) {
                    const int32_t c0 = sm.oct[((p + 4) >> 1) & 7][tid] * 8;
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(a.uo[v] + c0));
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(a.uo[v] + c0 + 4));
                    }
                }
                pen_barrier();
                // the old state of the cell to update: loaded between the two solves, early
                // enough for its latency and late enough for the registers
                double Uo[NV];
                int32_t ucid = 0;
                auto uload = [&]() {
                    ucid = sm.oct[(q >> 1) & 7][oo] * 8 + cxy + 4 * (q & 1);
#pragma unroll
                    for (int v = 0; v < NV; ++v) Uo[v] = a.uo[v][ucid];
                };
                // ---- D: the x and y faces on the left of and below the thread's cell
                if (MID) {
                    float WL[NV], Fx[NV], Fy[NV];
                    pen_ld(sm.Sx4[pb], sm.Sx1[pb], x ? ci - 1 : G::NI + y, WL);
                    col_solve<float, RS>(WL, mx, pr, a.status, Fx);
                    pen_st(sm.Gx4[pb], sm.Gx1[pb], ci + y, Fx);
                    __syncwarp();
                    if (UPD) uload();
                    pen_ld(sm.Sy4[pb], sm.Sy1[pb], y ? ci - G::FX : G::NI + x, WL);
                    col_solve<float, RS>(WL, my, pr, a.status, Fy);
                    pen_st(sm.Gy4[pb], sm.Gy1[pb], ci, Fy);
                }
                // ---- E: FP64 update of plane q
                if (UPD && !MID) uload();
                if (UPD) {
                    bool sk[6] = {false, false, false, false, false, false};
                    bool skip = false;
                    if constexpr (FINER) {
                        const uint8_t *rp = sm.ref[q & 7];
                        skip = rp[sio] != 0;
                        sk[0] = rp[sio - 1]; sk[1] = rp[sio + 1]; sk[2] = rp[sio - SX]; sk[3] = rp[sio + SX];
                        sk[4] = sm.ref[(q - 1) & 7][sio]; sk[5] = sm.ref[(q + 1) & 7][sio];
                    }
                    if (!skip) {
                        float F[NV], dU[NV] = {0.f, 0.f, 0.f, 0.f, 0.f};
                        // the order of the other kernels: x-left, x-right, y-left, y-right, z-below, z-above
                        pen_ld(sm.Gx4[qb], sm.Gx1[qb], ci + y, F);
                        if (!sk[0]) pen_acc<0>(dU, F, true);
                        pen_ld(sm.Gx4[qb], sm.Gx1[qb], ci + y + 1, F);
                        if (!sk[1]) pen_acc<0>(dU, F, false);
                        pen_ld(sm.Gy4[qb], sm.Gy1[qb], ci, F);
                        if (!sk[2]) pen_acc<1>(dU, F, true);
                        pen_ld(sm.Gy4[qb], sm.Gy1[qb], ci + G::FX, F);
                        if (!sk[3]) pen_acc<1>(dU, F, false);
                        if (!sk[4]) pen_acc<2>(dU, fzp, true);
                        if (!sk[5]) pen_acc<2>(dU, fz, false);
                        double Un[NV];
#pragma unroll
                        for (int v = 0; v < NV; ++v) {
                            Un[v] = add_f32(Uo[v], lamR * dU[v]);
                            a.un[v][ucid] = Un[v];
                            if (!BATCH) sm.Ur[qb][v][ci] = Un[v];
                        }
                        if (!state_finite<float>(Un)) set_error(a.status, AMR_ENONPHYSICAL);
                        const bool nbref = sk[0] || sk[1] || sk[2] || sk[3] || sk[4] || sk[5];
                        if (!nbref) sig = fmaxf(sig, cfl_signal(Un, pr));
                    }
                }
            };
            using T = std::true_type;
            using N = std::false_type;
            plane(N(), N(), z0 - 1);
            plane(N(), T(), z0);
            for (int p = z0 + 1; p < z1; ++p) plane(T(), T(), p);
            plane(T(), N(), z1);
            pen_barrier();
            if (dtn && sig > 0.f) my_dt = min(my_dt, (unsigned long long)__double_as_longlong(cfl_step(sig, cflR, dxR)));
            if (BATCH && dtn) {
                for (int off = 16; off > 0; off >>= 1) my_dt = min(my_dt, __shfl_xor_sync(0xffffffffu, my_dt, off));
                if (lane == 0 && my_dt != ~0ull) atomicMin(reinterpret_cast<unsigned long long *>(dtn), my_dt);
                my_dt = ~0ull;
            }
        }
        pen_barrier();
    }
    if (tid < G::NI && a.dt_next) {
        for (int off = 16; off > 0; off >>= 1) my_dt = min(my_dt, __shfl_xor_sync(0xffffffffu, my_dt, off));
        if (lane == 0 && my_dt != ~0ull) atomicMin(reinterpret_cast<unsigned long long *>(a.dt_next), my_dt);
    }
}

// Launch of the pencil kernel for the deepest complete level (or the box batch): zc is
// the z segment of a CTA, ragged at the top when it does not divide the level (octree mode),
// 0: equal shares of all z planes, one per resident CTA.  Requires 16 | n (every box, in
// batch mode).
template <int RS>
amr_status launch_pen(const amr_tree *t, const hydro_params *p, const double *u_old, double *u_new, const double *dt,
                      double *dt_next, int zc, cudaStream_t st)
{
    using G = PenGeo;
    ColArgs a;
    a.tv = make_view(t);
    a.grid = t->grid;
    a.n_inst = t->n_inst;
    a.inst_col_off = t->inst_col_off;
    a.inst_oct_off = t->inst_oct_off;
    a.finer = t->n_inst == 0 && t->grid_level < t->levelmax;
    a.zc = a.long_zc = 0;
    a.share_max = INT64_MAX;
    if (t->n_inst > 0) {
        if (t->col_work <= 0 || t->col_work % 4) return AMR_EINVAL;
        a.level = 0;
        a.n = 0;
        a.planes = t->col_work * 4;
    } else {
        a.level = t->grid_level;
        a.n = int64_t(1) << t->grid_level;
        if (a.n % G::FX) return AMR_EINVAL;
        const int64_t cols = (a.n / G::FX) * (a.n / G::FY);
        a.planes = cols * a.n;
        if (zc > 0) {
            zc = (zc + 1) & ~1;                          // whole oct layers
            a.zc = zc < a.n ? zc : int(a.n);
            a.planes = cols * ((a.n + a.zc - 1) / a.zc) * a.zc;
        }
    }
    a.state(t, u_old, u_new);
    a.dt = dt; a.dt_next = dt_next;
    a.scheme(p);
    const bool finer = a.finer != 0;
    const size_t bytes = finer ? sizeof(PenSmem<true>) : sizeof(PenSmem<false>);
    auto kern = t->n_inst > 0 ? k_godunov_pen<RS, false, true>
                              : finer ? k_godunov_pen<RS, true, false> : k_godunov_pen<RS, false, false>;
    return launch_kernel(kern, G::NT, bytes, true, st, a, column_grid);
}

}  // namespace amr
