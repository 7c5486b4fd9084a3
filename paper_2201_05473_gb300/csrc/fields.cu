// Yee FDTD field kernels of one step (bodies in fields_node.cuh): Faraday,
// Ampere (with the PIC deposit box), Ampere fused with the next step's
// Faraday, the moving window's field move and the wall-zeroing helper used
// after a state import.
#include "lbm_kernels.h"
#include "fields_fused.cuh"
#include "fields_rows.cuh"
#include "launch.cuh"

namespace pwfa {

namespace {

// Block shape of the field kernels: 64 x 2 (128 threads) measured 2.5 %
// faster than 32 x 8 for Faraday and Ampere on the 512x256x256 grid
// (0.207 / 0.291 against 0.213 / 0.298 ms).
#ifndef PWFA_FIELD_BX
#define PWFA_FIELD_BX 64
#endif
#ifndef PWFA_FIELD_BY
#define PWFA_FIELD_BY 2
#endif
constexpr int kBX = PWFA_FIELD_BX;
constexpr int kBY = PWFA_FIELD_BY;

// The separate Faraday launch (periodic grids below 4 Mi nodes, the PIC driver,
// FUSION_OFF, the step before a window move). It waits for its predecessor but
// does not announce the fluid kernel behind it: with the announcement every
// step of separate field kernels was slower, with Ampere's (whose successor
// needs a third of the fluid's registers) none. Whole steps on GB300, us,
// announced / not / all launches plain: 512x256x256 BGK FP32 3746 / 3683 /
// 3685, regularized FP16 2363 / 2300 / 2308; 256x128x128 476 / 468 / 476;
// 131x97x203 periodic 320 / 308 / 316; 64x32x32 10.3 / 9.9 / 16.4, FP16
// 11.6 / 9.4 / 16.4.
template <bool PER>
__global__ void __launch_bounds__(kBX * kBY) faraday_kernel(const StepArgs a) {
    chain_wait();
    const int i = blockIdx.x * kBX + threadIdx.x;
    const int j = blockIdx.y * kBY + threadIdx.y;
    if (i >= a.g.nx || j >= a.g.ny) return;
    faraday_node<PER>(a, i, j, blockIdx.z);
}

// Faraday with the field energy of its nodes: (|E|^2 + |Bc|^2)/2 at each
// node's index (the six staggered components stored there), summed in FP32
// over each warp (32 nodes) into energy[warp].
template <bool PER>
__global__ void __launch_bounds__(kBX * kBY) faraday_energy_kernel(const StepArgs a, float* energy) {
    const int i = blockIdx.x * kBX + threadIdx.x;
    const int j = blockIdx.y * kBY + threadIdx.y;
    float e2 = 0.0f;
    if (i < a.g.nx && j < a.g.ny) {
        faraday_node<PER>(a, i, j, blockIdx.z);
        const int64_t o = ((int64_t)blockIdx.z * a.g.ny + j) * a.g.nx + i;
        for (int c = 0; c < 3; ++c) {
            const float ev = ld_state(a.E[c] + o), bv = ld_state(a.Bc[c] + o);
            e2 += ev * ev + bv * bv;
        }
        e2 *= 0.5f;
    }
    for (int off = 16; off > 0; off >>= 1) e2 += __shfl_down_sync(0xffffffffu, e2, off);
    const int tid = threadIdx.y * kBX + threadIdx.x;
    if ((tid & 31) == 0) {
        const int64_t b = ((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
        energy[b * (kBX * kBY / 32) + (tid >> 5)] = e2;
    }
}

template <bool PER>
__global__ void __launch_bounds__(kBX * kBY) ampere_kernel(const StepArgs a) {
    chain_begin();
    const int i = blockIdx.x * kBX + threadIdx.x;
    const int j = blockIdx.y * kBY + threadIdx.y;
    if (a.jbox_next && i == 0 && j == 0 && blockIdx.z == 0) {
        // the next step's deposit box starts empty
        a.jbox_next[0] = a.jbox_next[1] = a.jbox_next[2] = 0x7fffffff;
        a.jbox_next[3] = a.jbox_next[4] = a.jbox_next[5] = -1;
    }
    if (i >= a.g.nx || j >= a.g.ny) return;
    ampere_node<PER>(a, i, j, blockIdx.z, a.zc);
}

template <bool PER>
__global__ void __launch_bounds__(kAFX * kAFY, PWFA_AF_MIN_BLOCKS)
    ampere_faraday_kernel(const StepArgs a, const FieldPair out) {
    chain_begin();
    ampere_faraday_tile<PER>(a, out, blockIdx.x, blockIdx.y, blockIdx.z, a.zc);
}

constexpr int64_t kPairNodes = (int64_t)256 << 10, kTileNodes = (int64_t)8 << 20;

// Blocks of four warps, each with its own nodes; as many blocks per SM as
// need no spills (V = 1: 64 registers, V = 2: 80).
template <int V> constexpr int kARBlocks = V == 1 ? 8 : 6;

// Blocks over a plane.
unsigned rows_blocks(const Grid& g, int V) {
    const int per = kARThreads / 32 * kARLanes * V;
    return (unsigned)((g.nx * g.ny + per - 1) / per);
}

template <int V, int H>
__global__ void __launch_bounds__(kARThreads, kARBlocks<V>) ampere_faraday_rows_kernel(const StepArgs a,
                                                                                       const FieldPair out) {
    chain_begin();
    const int n0 = (int)(blockIdx.x * (kARThreads / 32) + (threadIdx.x >> 5)) * kARLanes * V;
    if (n0 >= a.g.nx * a.g.ny) return;
    ampere_faraday_rows<V, H>(a, out, n0, blockIdx.y * H, a.zc);
}

template <int V, int H>
cudaError_t launch_rows_h(const StepArgs& a, const FieldPair& out, cudaStream_t s) {
    const dim3 grid(rows_blocks(a.g, V), (unsigned)((a.g.nz + H - 1) / H), 1);
    return launch_chained(ampere_faraday_rows_kernel<V, H>, grid, kARThreads, s, a, out);
}

// Which fused kernel an open grid takes, and how many planes a warp marches:
// more reuse more (B of the plane below, E of the plane above), fewer give
// more warps. Field update per step on GB300, events included.
//
// Pairs of nodes (an even nx; every array starts on 256 bytes) from 256 Ki
// nodes on: half the loads and address arithmetic per node, as many bytes in
// flight with fewer warps. Against single nodes, and from 8 Mi nodes against
// the tiles (15 loads a node, a barrier per plane), us: 512x256x256 398 -> 369
// (tiles; 436 with single nodes), 256x128x128 64 -> 57, 192x96x96 33 -> 29,
// 128x64x64 14.3 -> 12.6, 128x56x56 12.5 -> 11; 96x48x48 9.4 -> 10.2. Four
// consecutive nodes per thread were slower (63 us at 256x128x128: 157
// registers), and so were blocks of 256 or 384 threads and seven or eight
// blocks per SM (spills). Planes: the fewest whose blocks the GPU holds at
// once, two (one never fits from 256 Ki nodes on) to four (128x64x64: 14.6, 13.1, 14.2 us with 2, 3, 4; 256x128x128
// 87, 61.5, 59, 57 with 1 to 4, 61 with 8); eight from 8 Mi nodes on
// (512x256x256: 377 with 4, 371).
//
// Single nodes otherwise: one plane up to 96 Ki nodes (64x32x32: 6.5 us, 8
// with 2), two up to 640 Ki (96x48x48 8.7, 10.3 with 4), four above
// (203x97x131: 46, 43). From 8 Mi nodes on the tiles take an odd nx
// (512x256x255: 394 against 430).
cudaError_t launch_rows(const StepArgs& a, const FieldPair& out, cudaStream_t s) {
    if ((a.g.nx & 1) != 0 || a.g.N < kPairNodes) {
        if (a.g.N < ((int64_t)96 << 10)) return launch_rows_h<1, 1>(a, out, s);
        return a.g.N < ((int64_t)640 << 10) ? launch_rows_h<1, 2>(a, out, s) : launch_rows_h<1, 4>(a, out, s);
    }
    if (a.g.N >= kTileNodes) return launch_rows_h<2, 8>(a, out, s);
    int sms = 0;
    cudaError_t e = sm_count(&sms);
    if (e != cudaSuccess) return e;
    auto fits = [&](int h) {
        return rows_blocks(a.g, 2) * (int64_t)((a.g.nz + h - 1) / h) <= (int64_t)sms * kARBlocks<2>;
    };
    if (fits(2)) return launch_rows_h<2, 2>(a, out, s);
    if (fits(3)) return launch_rows_h<2, 3>(a, out, s);
    return launch_rows_h<2, 4>(a, out, s);
}

__global__ void __launch_bounds__(kBX * kBY) zero_walls_kernel(const StepArgs a) {
    const Grid& g = a.g;
    const int i = blockIdx.x * kBX + threadIdx.x;
    const int j = blockIdx.y * kBY + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= g.nx || j >= g.ny) return;
    const int64_t o = ((int64_t)k * g.ny + j) * g.nx + i;
    const int nx = g.nx, ny = g.ny, nz = g.nz;
    if (!(i <= nx - 2 && j >= 1 && j <= ny - 2 && k >= 1 && k <= nz - 2)) a.Eout[0][o] = 0.0f;
    if (!(i >= 1 && i <= nx - 2 && j <= ny - 2 && k >= 1 && k <= nz - 2)) a.Eout[1][o] = 0.0f;
    if (!(i >= 1 && i <= nx - 2 && j >= 1 && j <= ny - 2 && k <= nz - 2)) a.Eout[2][o] = 0.0f;
    float* Bc0 = const_cast<float*>(a.Bc[0]);
    float* Bc1 = const_cast<float*>(a.Bc[1]);
    float* Bc2 = const_cast<float*>(a.Bc[2]);
    if (!(i >= 1 && i <= nx - 2 && j <= ny - 2 && k <= nz - 2)) Bc0[o] = 0.0f;
    if (!(i <= nx - 2 && j >= 1 && j <= ny - 2 && k <= nz - 2)) Bc1[o] = 0.0f;
    if (!(i <= nx - 2 && j <= ny - 2 && k >= 1 && k <= nz - 2)) Bc2[o] = 0.0f;
}

// The moving window's field move: each thread moves kMovePlanes planes of its
// (x, y) column, with all 6 kMovePlanes loads issued before any store (one
// plane per thread left it latency-bound at 0.57 of the copy bandwidth).
// Every output element is written (moved value, or zero outside the
// conducting box).
constexpr int kMovePlanes = 4;

__global__ void __launch_bounds__(kBX * kBY) window_move_kernel(const WindowMove w) {
    const Grid& g = w.g;
    const int i = blockIdx.x * kBX + threadIdx.x;
    const int j = blockIdx.y * kBY + threadIdx.y;
    if (i >= g.nx || j >= g.ny) return;
    const int nx = g.nx, ny = g.ny, nz = g.nz;
    const bool ix = i >= 1 && i <= nx - 2, jy = j >= 1 && j <= ny - 2;
    const bool xi = i <= nx - 2, yj = j <= ny - 2;
    float v[kMovePlanes][6];
#pragma unroll
    for (int p = 0; p < kMovePlanes; ++p) {
        const int k = blockIdx.z * kMovePlanes + p;
        const int64_t up = ((int64_t)(k + 1) * ny + j) * nx + i;
        const bool in = k + 1 < nz;
        const bool kz = k >= 1 && k <= nz - 2, zk = k <= nz - 2;
        const bool m[6] = {in && xi && jy && kz, in && ix && yj && kz, in && ix && jy && zk,
                           in && ix && yj && zk, in && xi && jy && zk, in && xi && yj && kz};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            v[p][c] = m[c] ? w.E[c][up] : 0.0f;
            v[p][3 + c] = m[3 + c] ? w.B[c][up] : 0.0f;
        }
    }
#pragma unroll
    for (int p = 0; p < kMovePlanes; ++p) {
        const int k = blockIdx.z * kMovePlanes + p;
        if (k >= nz) break;
        const int64_t o = ((int64_t)k * ny + j) * nx + i;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            w.Eo[c][o] = v[p][c];
            w.Bo[c][o] = v[p][3 + c];
        }
    }
}

}  // namespace

cudaError_t launch_window_move(const WindowMove& w, cudaStream_t s) {
    dim3 block(kBX, kBY, 1);
    dim3 grid((w.g.nx + kBX - 1) / kBX, (w.g.ny + kBY - 1) / kBY, (w.g.nz + kMovePlanes - 1) / kMovePlanes);
    window_move_kernel<<<grid, block, 0, s>>>(w);
    return cudaGetLastError();
}

cudaError_t launch_zero_walls(const StepArgs& a, cudaStream_t s) {
    dim3 block(kBX, kBY, 1);
    dim3 grid((a.g.nx + kBX - 1) / kBX, (a.g.ny + kBY - 1) / kBY, a.g.nz);
    zero_walls_kernel<<<grid, block, 0, s>>>(a);
    return cudaGetLastError();
}

int64_t faraday_energy_records(const Grid& g) {
    return (int64_t)((g.nx + kBX - 1) / kBX) * ((g.ny + kBY - 1) / kBY) * g.nz * (kBX * kBY / 32);
}

cudaError_t launch_faraday(const StepArgs& a, cudaStream_t s, float* energy) {
    dim3 block(kBX, kBY, 1);
    dim3 grid((a.g.nx + kBX - 1) / kBX, (a.g.ny + kBY - 1) / kBY, a.g.nz);
    if (energy) {
        if (a.g.periodic) faraday_energy_kernel<true><<<grid, block, 0, s>>>(a, energy);
        else faraday_energy_kernel<false><<<grid, block, 0, s>>>(a, energy);
        return cudaGetLastError();
    }
    return launch_chained(a.g.periodic ? faraday_kernel<true> : faraday_kernel<false>, grid, block, s, a);
}

void fused_field_tiles(const Grid& g, int* tx, int* ty, int* tz) {
    *tx = (g.nx + kAFX - 2) / (kAFX - 1);
    *ty = (g.ny + kAFY - 2) / (kAFY - 1);
    *tz = (g.nz + kAFZ - 1) / kAFZ;
}

cudaError_t launch_ampere_faraday(const StepArgs& a, const FieldPair& out, cudaStream_t s) {
    if (a.Jb[0]) return cudaErrorInvalidValue;  // the PIC deposit is cleared by the plain Ampere kernel
    if (!a.g.periodic && (a.g.N < kTileNodes || (a.g.nx & 1) == 0)) return launch_rows(a, out, s);
    const dim3 block(kAFX, kAFY, 1);
    const dim3 grid((a.g.nx + kAFX - 2) / (kAFX - 1), (a.g.ny + kAFY - 2) / (kAFY - 1), (a.g.nz + kAFZ - 1) / kAFZ);
    return launch_chained(a.g.periodic ? ampere_faraday_kernel<true> : ampere_faraday_kernel<false>, grid, block, s, a,
                          out);
}

cudaError_t launch_ampere(const StepArgs& a, cudaStream_t s) {
    dim3 block(kBX, kBY, 1);
    dim3 grid((a.g.nx + kBX - 1) / kBX, (a.g.ny + kBY - 1) / kBY, a.g.nz);
    return launch_chained(a.g.periodic ? ampere_kernel<true> : ampere_kernel<false>, grid, block, s, a);
}

}  // namespace pwfa
