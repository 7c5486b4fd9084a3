// The fused field step of open grids (Ampere of step n with Faraday of step
// n + 1) over runs of consecutive nodes. Bodies of the separate updates:
// fields_node.cuh; the same step over tiles: fields_fused.cuh.
//
// A warp takes 31 V consecutive nodes of a plane, V (1 or 2; a divisor of
// nx) per thread, and marches up H planes. Each thread evaluates E_{n+3/2} at
// its nodes, plane by plane; of the three neighbours' E that Faraday reads,
// the +x one comes from the thread itself or the next lane (lane 31 only
// serves lane 30), the +z one is the thread's own next plane, and the +y one
// (E_x, E_z) the thread evaluates itself, which costs more loads per plane
// (19 for a pair of nodes, 24 for a single one, instead of the tiles' 15 per
// node; mostly L1 and L2 hits) and saves the block barrier, the tile fit and
// the set-up of a 32 x 8 block. B of the
// plane below, E_x, E_y of the plane above and J_z stay in registers. The
// arithmetic helpers are the separate kernels', so the state is theirs bit
// for bit.
#pragma once

#include "fields_node.cuh"

namespace pwfa {

constexpr int kARThreads = 128;
// lanes of a warp that own nodes: the last is the +x neighbour of the one before
constexpr int kARLanes = 31;

// V consecutive nodes' values as one load or store (p aligned to V floats)
template <int V>
__device__ __forceinline__ void row_ld(float (&d)[V], const float* p) {
    if constexpr (V == 2) {
        const float2 t = ld_state(reinterpret_cast<const float2*>(p));
        d[0] = t.x; d[1] = t.y;
    } else {
        d[0] = ld_state(p);
    }
}
template <int V>
__device__ __forceinline__ void row_st(float* p, const float (&d)[V]) {
    if constexpr (V == 2) *reinterpret_cast<float2*>(p) = make_float2(d[0], d[1]);
    else *p = d[0];
}
// The +x / -x neighbours' values of V consecutive ones. With V = 1 what was
// loaded is loaded again one node on, an L1 hit that a small grid waits for
// less than for a shuffle behind the load; with V > 1 the neighbours are
// the thread's own and, at the ends, the next lane's (last: what lane 31
// makes of it is not used) or the one before's (first: lane 0 reads it).
template <int V>
__device__ __forceinline__ void row_next(float (&d)[V], const float (&v)[V]) {
#pragma unroll
    for (int j = 0; j < V - 1; ++j) d[j] = v[j + 1];
    d[V - 1] = __shfl_down_sync(0xffffffffu, v[0], 1);
}
template <int V>
__device__ __forceinline__ void row_next(float (&d)[V], const float (&v)[V], float last) {
    if constexpr (V == 1) d[0] = last;
    else row_next(d, v);
}
template <int V>
__device__ __forceinline__ void row_prev(float (&d)[V], const float (&v)[V], float first) {
    if constexpr (V == 1) {
        d[0] = first;
    } else {
#pragma unroll
        for (int j = 1; j < V; ++j) d[j] = v[j - 1];
        const float up = __shfl_up_sync(0xffffffffu, v[V - 1], 1);
        d[0] = (threadIdx.x & 31) == 0 ? first : up;
    }
}

// What a thread reads of its nodes' plane: their own values, and what E_x,
// E_z of the +y neighbours need (y...); the -x neighbours' B (..._f) and the
// +x neighbours' J_x (..._l) where row_prev and row_next want them.
template <int V>
struct ARPlane {
    float e0[V], e1[V], e2[V], bx[V], by[V], bz[V], bz_j[V], bx_j[V], j0[V], j1[V], j1_j[V], j2_k[V];
    float ye0[V], ye2[V], ybx[V], yby[V], ybz[V], yj0[V], yj2_k[V];
    float by_f, bz_f, yby_f, j0_l, yj0_l;
};

template <int V, bool HALO>
__device__ __forceinline__ void ar_load(const StepArgs& a, int o, int xp, int yp, int zp, ARPlane<V>& v) {
    const float *Bx = a.Bn[0], *By = a.Bn[1], *Bz = a.Bn[2];
    const int nx = a.g.nx;
#ifdef PWFA_DEBUG
    o = PWFA_CHECK(a.dbg, o, 0, a.g.N, 6u);
    PWFA_CHECK(a.dbg, o + V - 1, 0, a.g.N, 6u);
    zp = PWFA_CHECK(a.dbg, o + yp + zp, 0, a.g.N, 6u) - o - yp;
    PWFA_CHECK(a.dbg, o + yp + zp + V - 1, 0, a.g.N, 6u);
    if (V == 1) PWFA_CHECK(a.dbg, o + yp + xp, 0, a.g.N, 6u);
    PWFA_CHECK(a.dbg, o - nx, -guard_elems(a.g), a.g.N, 6u);
#endif
    const bool first = V == 1 || (threadIdx.x & 31) == 0;
    row_ld(v.e0, a.E[0] + o);
    row_ld(v.e1, a.E[1] + o);
    row_ld(v.bx, Bx + o);
    row_ld(v.by, By + o);
    row_ld(v.bz, Bz + o);
    row_ld(v.bz_j, Bz + o - nx);
    row_ld(v.j0, a.J[0] + o);
    row_ld(v.j1, a.J[1] + o);
    row_ld(v.j1_j, a.J[1] + o + yp);
    v.bz_f = first ? ld_state(Bz + o - 1) : 0.0f;
    if (V == 1) v.j0_l = ld_state(a.J[0] + o + xp);
    if (HALO) {
        row_ld(v.e2, a.E[2] + o);
        row_ld(v.bx_j, Bx + o - nx);
        row_ld(v.j2_k, a.J[2] + o + zp);
        row_ld(v.ye0, a.E[0] + o + yp);
        row_ld(v.ye2, a.E[2] + o + yp);
        row_ld(v.ybx, Bx + o + yp);
        row_ld(v.yby, By + o + yp);
        row_ld(v.ybz, Bz + o + yp);
        row_ld(v.yj0, a.J[0] + o + yp);
        row_ld(v.yj2_k, a.J[2] + o + yp + zp);
        v.by_f = first ? ld_state(By + o - 1) : 0.0f;
        v.yby_f = first ? ld_state(By + o + yp - 1) : 0.0f;
        if (V == 1) v.yj0_l = ld_state(a.J[0] + o + yp + xp);
    }
}

// The fused step of the calling warp's kARLanes V nodes from node n0 of a
// plane (n = y nx + x, a multiple of V) and planes [k0, k0 + H).
template <int V, int H>
__device__ __forceinline__ void ampere_faraday_rows(const StepArgs& a, const FieldPair& out, int n0, int k0, float zc) {
    const Grid& g = a.g;
    const int nx = g.nx, ny = g.ny, nz = g.nz, nxy = nx * ny;
    const int lane = threadIdx.x & 31;
    const int n = min(n0 + lane * V, nxy - V);
    const bool own = lane < kARLanes && n0 + lane * V < nxy;
    const int y = n / nx, x = n - y * nx;
    const int xp = x < nx - 1 ? 1 : 0, yp = y < ny - 1 ? nx : 0;
    // wall masks: of the row, and of the nodes at the two x walls
    const bool yin = y >= 1 && y <= ny - 2, ylo = y <= ny - 2, y1lo = y + 1 <= ny - 2;
    const float c = a.cdt, dt = a.dt;
    float gT[V], gTy[V];
#pragma unroll
    for (int j = 0; j < V; ++j) {
        gT[j] = a.alpha != 0.0f ? driver_transverse(a, x + j, y) : 0.0f;
        gTy[j] = a.alpha != 0.0f ? driver_transverse(a, x + j, y + 1) : 0.0f;
    }
    const float glane = a.alpha != 0.0f && lane <= H ? driver_longitudinal(a, k0 + lane, zc) : 0.0f;
    const int kend = min(k0 + H, nz);
    int o = k0 * nxy + n;
    float by_k[V], bx_k[V], yby_k[V], j2[V], yj2[V], e0[V], e1[V];
#ifdef PWFA_DEBUG
    PWFA_CHECK(a.dbg, o - nxy, -guard_elems(g), g.N, 6u);
#endif
    row_ld(by_k, a.Bn[1] + o - nxy);
    row_ld(bx_k, a.Bn[0] + o - nxy);
    row_ld(yby_k, a.Bn[1] + o + yp - nxy);
    row_ld(j2, a.J[2] + o);
    row_ld(yj2, a.J[2] + o + yp);
    ARPlane<V> v;
    ar_load<V, true>(a, o, xp, yp, k0 < nz - 1 ? nxy : 0, v);
    // one plane per warp: the plane above is asked for in the same round
    ARPlane<V> w;
    if (H == 1 && k0 <= nz - 2) ar_load<V, false>(a, o + nxy, xp, yp, 0, w);
    auto inx = [&](int j) { return !(j == 0 && x == 0) && !(j == V - 1 && x == nx - V); };  // 1 <= x <= nx - 2
    auto xlo = [&](int j) { return !(j == V - 1 && x == nx - V); };                          // x <= nx - 2
    // E_x and E_y of plane k from v and B of the plane below
    auto transverse = [&](bool kin) {
        float j0_i[V], bz_i[V];
        row_next(j0_i, v.j0, v.j0_l);
        row_prev(bz_i, v.bz, v.bz_f);
#pragma unroll
        for (int j = 0; j < V; ++j) {
            e0[j] = v.e0[j];
            e1[j] = v.e1[j];
            if (yin && xlo(j) && kin)
                e0[j] = ampere_arith(c, dt, e0[j], v.bz[j] - v.bz_j[j], v.by[j] - by_k[j], 0.5f * (v.j0[j] + j0_i[j]));
            if (ylo && inx(j) && kin)
                e1[j] = ampere_arith(c, dt, e1[j], v.bx[j] - bx_k[j], v.bz[j] - bz_i[j], 0.5f * (v.j1[j] + v.j1_j[j]));
        }
    };
    transverse(k0 >= 1 && k0 <= nz - 2);
    for (int k = k0; k < kend; ++k) {
        const bool kin = k >= 1 && k <= nz - 2, klo = k <= nz - 2;
        const float gl = __shfl_sync(0xffffffffu, glane, k - k0);
        float e2[V], ex_j[V], ez_j[V], b0[V], b1[V], b2[V], e0k[V], e1k[V];
        {
            float by_i[V], yby_i[V], yj0_i[V];
            row_prev(by_i, v.by, v.by_f);
            row_prev(yby_i, v.yby, v.yby_f);
            row_next(yj0_i, v.yj0, v.yj0_l);
#pragma unroll
            for (int j = 0; j < V; ++j) {
                const float jb = a.alpha != 0.0f ? -(gT[j] * gl) : 0.0f, yjb = a.alpha != 0.0f ? -(gTy[j] * gl) : 0.0f;
                e2[j] = v.e2[j];
                ex_j[j] = v.ye0[j];
                ez_j[j] = v.ye2[j];
                if (yin && inx(j) && klo)
                    e2[j] = ampere_arith(c, dt, e2[j], v.by[j] - by_i[j], v.bx[j] - v.bx_j[j],
                                         0.5f * (j2[j] + v.j2_k[j]) + jb);
                if (y1lo && xlo(j) && kin)
                    ex_j[j] = ampere_arith(c, dt, ex_j[j], v.ybz[j] - v.bz[j], v.yby[j] - yby_k[j],
                                           0.5f * (v.yj0[j] + yj0_i[j]));
                if (y1lo && inx(j) && klo)
                    ez_j[j] = ampere_arith(c, dt, ez_j[j], v.yby[j] - yby_i[j], v.ybx[j] - v.bx[j],
                                           0.5f * (yj2[j] + v.yj2_k[j]) + yjb);
                b0[j] = v.bx[j];
                b1[j] = v.by[j];
                b2[j] = v.bz[j];
                e0k[j] = e0[j];
                e1k[j] = e1[j];
                by_k[j] = v.by[j];
                bx_k[j] = v.bx[j];
                yby_k[j] = v.yby[j];
                j2[j] = v.j2_k[j];
                yj2[j] = v.yj2_k[j];
            }
        }
        // plane k + 1: its E_x, E_y now, the rest of it in the next pass
        const int on = o + nxy;
        if (klo) {
            if (H == 1) v = w;
            else if (k + 1 < kend) ar_load<V, true>(a, on, xp, yp, k + 1 < nz - 1 ? nxy : 0, v);
            else ar_load<V, false>(a, on, xp, yp, 0, v);
            transverse(k + 1 <= nz - 2);
        } else {
#pragma unroll
            for (int j = 0; j < V; ++j) e0[j] = e1[j] = 0.0f;
        }
        float ez_i[V], ey_i[V];
        row_next(ez_i, e2);
        row_next(ey_i, e1k);
        if (own) {
#ifdef PWFA_DEBUG
            o = PWFA_CHECK(a.dbg, o, 0, g.N, 6u);
            PWFA_CHECK(a.dbg, o + V - 1, 0, g.N, 6u);
#endif
#pragma unroll
            for (int j = 0; j < V; ++j) {
                const float b[3] = {b0[j], b1[j], b2[j]};
                float bn[3];
                faraday_arith(c, b, e0k[j], e1k[j], e2[j], ez_j[j], e1[j], e0[j], ez_i[j], ey_i[j], ex_j[j],
                              ylo && inx(j) && klo, yin && xlo(j) && klo, ylo && xlo(j) && kin, bn);
                b0[j] = bn[0];
                b1[j] = bn[1];
                b2[j] = bn[2];
            }
            row_st(out.E[0] + o, e0k);
            row_st(out.E[1] + o, e1k);
            row_st(out.E[2] + o, e2);
            row_st(out.B[0] + o, b0);
            row_st(out.B[1] + o, b1);
            row_st(out.B[2] + o, b2);
        }
        o = on;
    }
}

}  // namespace pwfa
