// The fused field step of open grids (Ampere of step n with Faraday of step
// n + 1) over runs of consecutive nodes. Bodies of the separate updates:
// fields_node.cuh; the same step over tiles: fields_fused.cuh.
//
// A warp takes 31 consecutive nodes of a plane and marches up H planes. Each
// thread evaluates E_{n+3/2} at its node, plane by plane; of the three
// neighbours' E that Faraday reads, the +x one comes from the next lane (lane
// 31 only serves lane 30), the +z one is the thread's own next plane, and the
// +y one (E_x, E_z) the thread evaluates itself, which costs nine more loads
// per plane (24 instead of the tiles' 15, mostly L1 hits) and saves the
// block barrier, the tile fit and the set-up of a 32 x 8 block: what a grid
// that fits in L2, and that few large tiles cannot spread over the GPU, is
// bound by. B of the plane below and J_z of the plane above stay in
// registers. The arithmetic helpers are the separate kernels', so the state
// is theirs bit for bit.
#pragma once

#include "fields_node.cuh"

namespace pwfa {

constexpr int kARThreads = 128;
// nodes a warp owns: its last lane is the +x neighbour of the one before
constexpr int kARNodes = 31;

// What a thread reads for E_{n+3/2} of its column's plane: its own node, and
// E_x, E_z of the +y neighbour (y...).
struct ARPlane {
    float e0, e1, e2, bx, by, bz, bz_i, by_i, bz_j, bx_j, j0, j0_i, j1, j1_j, j2_k;
    float ye0, ye2, ybx, yby, ybz, yby_i, yj0, yj0_i, yj2_k;
};

template <bool HALO>
__device__ __forceinline__ void ar_load(const StepArgs& a, int o, int xp, int yp, int zp, ARPlane& v) {
    const float *Bx = a.Bn[0], *By = a.Bn[1], *Bz = a.Bn[2];
    const int nx = a.g.nx;
#ifdef PWFA_DEBUG
    o = PWFA_CHECK(a.dbg, o, 0, a.g.N, 6u);
    zp = PWFA_CHECK(a.dbg, o + yp + zp, 0, a.g.N, 6u) - o - yp;
    xp = PWFA_CHECK(a.dbg, o + yp + xp, 0, a.g.N, 6u) - o - yp;
    PWFA_CHECK(a.dbg, o - nx, -guard_elems(a.g), a.g.N, 6u);
#endif
    v.e0 = __ldg(a.E[0] + o);
    v.e1 = __ldg(a.E[1] + o);
    v.bx = __ldg(Bx + o);
    v.by = __ldg(By + o);
    v.bz = __ldg(Bz + o);
    v.bz_i = __ldg(Bz + o - 1);
    v.bz_j = __ldg(Bz + o - nx);
    v.j0 = __ldg(a.J[0] + o);
    v.j0_i = __ldg(a.J[0] + o + xp);
    v.j1 = __ldg(a.J[1] + o);
    v.j1_j = __ldg(a.J[1] + o + yp);
    if (HALO) {
        v.e2 = __ldg(a.E[2] + o);
        v.by_i = __ldg(By + o - 1);
        v.bx_j = __ldg(Bx + o - nx);
        v.j2_k = __ldg(a.J[2] + o + zp);
        v.ye0 = __ldg(a.E[0] + o + yp);
        v.ye2 = __ldg(a.E[2] + o + yp);
        v.ybx = __ldg(Bx + o + yp);
        v.yby = __ldg(By + o + yp);
        v.ybz = __ldg(Bz + o + yp);
        v.yby_i = __ldg(By + o + yp - 1);
        v.yj0 = __ldg(a.J[0] + o + yp);
        v.yj0_i = __ldg(a.J[0] + o + yp + xp);
        v.yj2_k = __ldg(a.J[2] + o + yp + zp);
    }
}

// The fused step of the calling warp's kARNodes nodes [n0, n0 + 31) of a
// plane (n = y nx + x) and planes [k0, k0 + H).
template <int H>
__device__ __forceinline__ void ampere_faraday_rows(const StepArgs& a, const FieldPair& out, int n0, int k0, float zc) {
    const Grid& g = a.g;
    const int nx = g.nx, ny = g.ny, nz = g.nz, nxy = nx * ny;
    const int lane = threadIdx.x & 31;
    const int n = min(n0 + lane, nxy - 1);
    const bool own = lane < kARNodes && n0 + lane < nxy;
    const int y = n / nx, x = n - y * nx;
    const int xp = x < nx - 1 ? 1 : 0, yp = y < ny - 1 ? nx : 0;
    const bool mEx = x <= nx - 2 && y >= 1 && y <= ny - 2;   // E_x and B_y
    const bool mEy = x >= 1 && x <= nx - 2 && y <= ny - 2;   // E_y and B_x
    const bool mEz = x >= 1 && x <= nx - 2 && y >= 1 && y <= ny - 2;
    const bool mBz = x <= nx - 2 && y <= ny - 2;
    const bool yEx = x <= nx - 2 && y + 1 <= ny - 2, yEz = yEx && x >= 1;
    const float c = a.cdt, dt = a.dt;
    const float gT = a.alpha != 0.0f ? driver_transverse(a, x, y) : 0.0f;
    const float gTy = a.alpha != 0.0f ? driver_transverse(a, x, y + 1) : 0.0f;
    const float glane = a.alpha != 0.0f && lane <= H ? driver_longitudinal(a, k0 + lane, zc) : 0.0f;
    const int kend = min(k0 + H, nz);
    int o = k0 * nxy + n;
    float by_k, bx_k, yby_k, j2, yj2;
    {
#ifdef PWFA_DEBUG
        PWFA_CHECK(a.dbg, o - nxy, -guard_elems(g), g.N, 6u);
#endif
        by_k = __ldg(a.Bn[1] + o - nxy);
        bx_k = __ldg(a.Bn[0] + o - nxy);
        yby_k = __ldg(a.Bn[1] + o + yp - nxy);
        j2 = __ldg(a.J[2] + o);
        yj2 = __ldg(a.J[2] + o + yp);
    }
    ARPlane v;
    ar_load<true>(a, o, xp, yp, k0 < nz - 1 ? nxy : 0, v);
    for (int k = k0; k < kend; ++k) {
        const bool kin = k >= 1 && k <= nz - 2, klo = k <= nz - 2;
        const float gl = __shfl_sync(0xffffffffu, glane, k - k0);
        const float jb = a.alpha != 0.0f ? -(gT * gl) : 0.0f, yjb = a.alpha != 0.0f ? -(gTy * gl) : 0.0f;
        float e0 = v.e0, e1 = v.e1, e2 = v.e2, ex_j = v.ye0, ez_j = v.ye2;
        if (mEx && kin) e0 = ampere_arith(c, dt, e0, v.bz - v.bz_j, v.by - by_k, 0.5f * (v.j0 + v.j0_i));
        if (mEy && kin) e1 = ampere_arith(c, dt, e1, v.bx - bx_k, v.bz - v.bz_i, 0.5f * (v.j1 + v.j1_j));
        if (mEz && klo) e2 = ampere_arith(c, dt, e2, v.by - v.by_i, v.bx - v.bx_j, 0.5f * (j2 + v.j2_k) + jb);
        if (yEx && kin) ex_j = ampere_arith(c, dt, ex_j, v.ybz - v.bz, v.yby - yby_k, 0.5f * (v.yj0 + v.yj0_i));
        if (yEz && klo) ez_j = ampere_arith(c, dt, ez_j, v.yby - v.yby_i, v.ybx - v.bx, 0.5f * (yj2 + v.yj2_k) + yjb);
        const float b[3] = {v.bx, v.by, v.bz};
        by_k = v.by;
        bx_k = v.bx;
        yby_k = v.yby;
        j2 = v.j2_k;
        yj2 = v.yj2_k;
        // plane k + 1: its E_x, E_y now, the rest of it in the next pass
        const int on = o + nxy;
        float ex_k = 0.0f, ey_k = 0.0f;
        if (klo) {
            if (k + 1 < kend) ar_load<true>(a, on, xp, yp, k + 1 < nz - 1 ? nxy : 0, v);
            else ar_load<false>(a, on, xp, yp, 0, v);
            const bool kin1 = k + 1 <= nz - 2;
            ex_k = v.e0;
            ey_k = v.e1;
            if (mEx && kin1) ex_k = ampere_arith(c, dt, ex_k, v.bz - v.bz_j, v.by - by_k, 0.5f * (v.j0 + v.j0_i));
            if (mEy && kin1) ey_k = ampere_arith(c, dt, ey_k, v.bx - bx_k, v.bz - v.bz_i, 0.5f * (v.j1 + v.j1_j));
        }
        const float ez_i = __shfl_down_sync(0xffffffffu, e2, 1), ey_i = __shfl_down_sync(0xffffffffu, e1, 1);
        if (own) {
#ifdef PWFA_DEBUG
            o = PWFA_CHECK(a.dbg, o, 0, g.N, 6u);
#endif
            float bn[3];
            faraday_arith(c, b, e0, e1, e2, ez_j, ey_k, ex_k, ez_i, ey_i, ex_j, mEy && klo, mEx && klo, mBz && kin,
                          bn);
            out.E[0][o] = e0;
            out.E[1][o] = e1;
            out.E[2][o] = e2;
            out.B[0][o] = bn[0];
            out.B[1][o] = bn[1];
            out.B[2][o] = bn[2];
        }
        o = on;
    }
}

}  // namespace pwfa
