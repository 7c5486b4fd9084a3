// Set-up, state exchange and diagnostics kernels (not on the per-step path).
#include "lbm_kernels.h"
#include "lbm_node.cuh"
#include "launch.cuh"

namespace pwfa {

namespace {

// blocks of the field export
constexpr int kBX = 32;
constexpr int kBY = 4;

__device__ __forceinline__ void node_xyz(const Grid& g, int64_t node, int& x, int& y, int& z) {
    const int64_t sxy = (int64_t)g.nx * g.ny;
    z = (int)(node / sxy);
    const int64_t r = node - (int64_t)z * sxy;
    y = (int)(r / g.nx);
    x = (int)(r - (int64_t)y * g.nx);
}

// Radial multiplier: linear between r_j = j rmax/(np-1), last value beyond.
__device__ double profile_at(const double* prof, int np, double rmax, double r) {
    if (np <= 0) return 1.0;
    if (np == 1 || r >= rmax) return prof[np - 1];
    const double h = rmax / (np - 1);
    const double t = r / h;
    int j = (int)floor(t);
    if (j >= np - 1) return prof[np - 1];
    const double fr = t - j;
    return (1.0 - fr) * prof[j] + fr * prof[j + 1];
}

// Stored array S with S_i(y) = f^0_i(y + xi_i): pulling it yields the plasma
// at rest f^0 = w_i n0 prof(r) (lattice 0) and 0 (momentum lattices). Open
// grids clamp y + xi_i to the interior (such entries are only pulled by
// interior nodes, for which the clamp is the identity). Every population
// node up to Np is written: the plane above the box (present with a moving
// window) keeps this fresh plasma for good.
template <int ST>
__global__ void init_kernel(Grid g, typename Codec<ST>::T* f, float n0, const double* prof, int np,
                            double rmax, double dx) {
    const int64_t node = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (node >= g.Np) return;
    int x, y, z;
    node_xyz(g, node, x, y, z);
    const double xc = 0.5 * (g.nx - 1) * dx, yc = 0.5 * (g.ny - 1) * dx;
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
        float n = n0;
        if (np > 0) {  // FP64 only where a profile is given
            int sx = x + xi_x(q), sy = y + xi_y(q);
            if (g.periodic) { sx = wrapi(sx, g.nx); sy = wrapi(sy, g.ny); }
            else { sx = min(max(sx, 1), g.nx - 2); sy = min(max(sy, 1), g.ny - 2); }
            const double rx = sx * dx - xc, ry = sy * dx - yc;
            n = (float)((double)n0 * profile_at(prof, np, rmax, sqrt(rx * rx + ry * ry)));
        }
        const uint32_t off = pop_off(q, (uint32_t)node);
        const int64_t LS = lattice_stride(g);
        Codec<ST>::store(f + pop_elem<ST>(0, off, LS), wq(q) * n, 0, q, n0);
#pragma unroll
        for (int l = 1; l < kL; ++l) Codec<ST>::store(f + pop_elem<ST>(l, off, LS), 0.0f, l, q, n0);
    }
}

// f^n at every node (boundary nodes: f^eq of the clamped interior node).
template <int ST, bool PER>
__global__ void __launch_bounds__(kLinearThreads) export_f_kernel(const StepArgs a, const LinearMap m, float* out) {
    using T = typename Codec<ST>::T;
    const Grid& g = a.g;
    int x, y, z;
    if (!m.node(g, x, y, z)) return;
    const int64_t node = ((int64_t)z * g.ny + y) * g.nx + x;
    float f[kL][kQ];
    bool bnd;
    gather<ST, PER>(g, static_cast<const T*>(a.fin), a.n0, x, y, z, f, bnd, 0u, a.dbg);
    if (!PER && bnd) {
        float A[kL], inn, beta[3], phi[kQ];
        node_moments(f, a.n_floor, A, inn, beta);
        const float u[3] = {beta[0] * a.lat, beta[1] * a.lat, beta[2] * a.lat};
        eq_factors(u, phi);
        for (int l = 0; l < kL; ++l)
            for (int q = 0; q < kQ; ++q) f[l][q] = A[l] * phi[q];
    }
#pragma unroll
    for (int l = 0; l < kL; ++l)
#pragma unroll
        for (int q = 0; q < kQ; ++q) out[(int64_t)(l * kQ + q) * g.N + node] = f[l][q];
}

// Inverse of the pull: S_i(y) = f^n_i(y + xi_i). A block takes 128 consecutive
// nodes and one pair of lattices (blockIdx.y), and a thread issues its 38
// loads before any store: DRAM-bound (608 B/node FP32). One population after
// another had left a single round of four loads in flight per thread:
// 256x128x128 FP32 set_state 773 -> 464 us.
template <int ST, bool PER>
__global__ void __launch_bounds__(kLinearThreads) import_f_kernel(Grid g, const LinearMap m,
                                                                  const float* __restrict__ in,
                                                                  typename Codec<ST>::T* f, float n0) {
    int x, y, z;
    if (!m.node(g, x, y, z)) return;
    const int64_t node = ((int64_t)z * g.ny + y) * g.nx + x;
    // offsets to the neighbours, wrapped or clamped into the grid
    const int64_t sx = g.nx, sxy = sx * g.ny;
    const int64_t ox[3] = {x > 0 ? -1 : (PER ? g.nx - 1 : 0), 0, x < g.nx - 1 ? 1 : (PER ? 1 - g.nx : 0)};
    const int64_t oy[3] = {y > 0 ? -sx : (PER ? (g.ny - 1) * sx : 0), 0, y < g.ny - 1 ? sx : (PER ? (1 - g.ny) * sx : 0)};
    const int64_t oz[3] = {z > 0 ? -sxy : (PER ? (g.nz - 1) * sxy : 0), 0,
                           z < g.nz - 1 ? sxy : (PER ? (1 - g.nz) * sxy : 0)};
    const int l0 = 2 * (int)blockIdx.y;
    const float* p0 = in + (int64_t)l0 * kQ * g.N + node;
    const float* p1 = p0 + (int64_t)kQ * g.N;
    float v0[kQ], v1[kQ];
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
        const int64_t o = q * g.N + ox[xi_x(q) + 1] + oy[xi_y(q) + 1] + oz[xi_z(q) + 1];
        v0[q] = ld_state(p0 + o);
        v1[q] = ld_state(p1 + o);
    }
    const int64_t LS = lattice_stride(g);
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
        const uint32_t off = pop_off(q, (uint32_t)node);
        auto* d = f + pop_elem<ST>(l0, off, LS);
        if constexpr (ST == 0) {
            Codec<ST>::store(d, v0[q], l0, q, n0);
            Codec<ST>::store(d + LS, v1[q], l0 + 1, q, n0);
        } else {
            Codec<ST>::store2(d, v0[q], v1[q], l0, q, n0);
        }
    }
}

template <int ST, bool PER>
__global__ void __launch_bounds__(kBX * kBY) export_fields_kernel(const StepArgs a, unsigned mask, float* out) {
    using T = typename Codec<ST>::T;
    const Grid& g = a.g;
    const int x = blockIdx.x * kBX + threadIdx.x;
    const int y = blockIdx.y * kBY + threadIdx.y;
    const int z = blockIdx.z;
    if (x >= g.nx || y >= g.ny) return;
    const int64_t node = ((int64_t)z * g.ny + y) * g.nx + x;
    float vals[16];
    if (mask & 0xE00Fu) {
        float f[kL][kQ];
        bool bnd;
        gather<ST, PER>(g, static_cast<const T*>(a.fin), a.n0, x, y, z, f, bnd, 0u, a.dbg);
        float A[kL], inn, beta[3];
        node_moments(f, a.n_floor, A, inn, beta);
        vals[0] = A[0];
        vals[1] = beta[0]; vals[2] = beta[1]; vals[3] = beta[2];
        vals[13] = A[1]; vals[14] = A[2]; vals[15] = A[3];
    }
    const bool raw = (mask >> 31) & 1u;
    if (mask & 0x70u) {
        if (raw) { for (int c = 0; c < 3; ++c) vals[4 + c] = a.E[c][node]; }
        else { float e[3]; node_E<PER>(g, a.E, x, y, z, e, a.dbg); for (int c = 0; c < 3; ++c) vals[4 + c] = e[c]; }
    }
    if (mask & 0x380u) {
        if (raw) { for (int c = 0; c < 3; ++c) vals[7 + c] = a.Bc[c][node]; }
        else { float b[3]; node_B_sum<PER>(g, a.Bc, x, y, z, b, a.dbg); for (int c = 0; c < 3; ++c) vals[7 + c] = 0.25f * b[c]; }
    }
    if (mask & 0x1C00u) { for (int c = 0; c < 3; ++c) vals[10 + c] = a.J[c][node]; }
    int slot = 0;
    for (int bit = 0; bit < 16; ++bit)
        if (mask & (1u << bit)) out[(int64_t)(slot++) * g.N + node] = vals[bit];
}

// ---------------------------------------------------------------- line cuts
// Values along z at transverse offset r (c/omega_p) from the axis in +x,
// bilinear between the four nodes around (x_c + r, y_c): slot 0 density n,
// slot 1 node-averaged E_z (each thread one z).
template <int ST, bool PER>
__global__ void linecut_kernel(const StepArgs a, double xr, float* out) {
    using T = typename Codec<ST>::T;
    const Grid& g = a.g;
    const int z = blockIdx.x * blockDim.x + threadIdx.x;
    if (z >= g.nz) return;
    const double xs = xr / a.dx + 0.5 * (g.nx - 1), ys = 0.5 * (g.ny - 1);
    int x0 = (int)floor(xs), y0 = (int)floor(ys);
    x0 = min(max(x0, 0), g.nx - 2);
    y0 = min(max(y0, 0), g.ny - 2);
    const float fx = (float)(xs - x0), fy = (float)(ys - y0);
    float nsum = 0.0f, esum = 0.0f;
    for (int c = 0; c < 4; ++c) {
        const int x = x0 + (c & 1), y = y0 + (c >> 1);
        const float wgt = ((c & 1) ? fx : 1.0f - fx) * ((c >> 1) ? fy : 1.0f - fy);
        float f[kL][kQ];
        bool bnd;
        gather<ST, PER>(g, static_cast<const T*>(a.fin), a.n0, x, y, z, f, bnd, 0u, a.dbg);
        float A[kL], inn, beta[3];
        node_moments(f, a.n_floor, A, inn, beta);
        float e[3];
        node_E<PER>(g, a.E, x, y, z, e, a.dbg);
        nsum += wgt * A[0];
        esum += wgt * e[2];
    }
    out[z] = nsum;
    out[g.nz + z] = esum;
}

// ---------------------------------------------------------------- diagnostics
// FP64 arithmetic is scarce on this part (two lanes an SM and clock, and
// every conversion takes one): what bounds these kernels. So only the sums
// are formed in FP64; minimum and count stay in FP32 and integers, which
// hold them exactly, the maximum of |beta|^2 is kept by its bits (those of
// non-negative doubles order as integers) and its root, which is monotonic,
// is taken once per block.
struct Diag {
    double s[5];      // sums of n, n p_x, n p_y, n p_z, field energy
    float mn;         // min n (infinity: no finite one)
    long long mb;     // bits of max |beta|^2 (or of max |beta|)
    int bad;          // non-finite nodes
};
__device__ __forceinline__ Diag diag_none() { return Diag{{0, 0, 0, 0, 0}, __int_as_float(0x7f800000), 0, 0}; }

// Block reduction to one record of 8 doubles: sums over a warp by recursive
// halving (as diag8_warp of the fluid kernel: 9 adds a lane instead of 40),
// then 8 threads over the warps. ROOT: mb holds squares.
template <bool ROOT>
__device__ void diag_block_reduce(const Diag& d, double* dst) {
    constexpr int W = kDiagThreads / 32;
    __shared__ double shs[W][8];
    __shared__ float shm[W];
    __shared__ long long shb[W];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
    const double v[8] = {d.s[0], d.s[1], d.s[2], d.s[3], d.s[4], (double)d.bad, 0.0, 0.0};
    double w[4], u[2];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const double keep = b4 ? v[k + 4] : v[k], send = b4 ? v[k] : v[k + 4];
        w[k] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const double keep = b3 ? w[k + 2] : w[k], send = b3 ? w[k] : w[k + 2];
        u[k] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
    }
    double t = (b2 ? u[1] : u[0]) + __shfl_xor_sync(0xffffffffu, b2 ? u[0] : u[1], 4);
    t += __shfl_xor_sync(0xffffffffu, t, 2);
    t += __shfl_xor_sync(0xffffffffu, t, 1);
    float mn = d.mn;
    long long mb = d.mb;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, off));
        const long long o = __shfl_xor_sync(0xffffffffu, mb, off);
        mb = o > mb ? o : mb;
    }
    if ((lane & 3) == 0) shs[warp][lane >> 2] = t;
    if (lane == 0) {
        shm[warp] = mn;
        shb[warp] = mb;
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        double r = 0.0;
        for (int k = 0; k < W; ++k) r += shs[k][threadIdx.x];
        dst[threadIdx.x == 5 ? 7 : threadIdx.x] = r;
    } else if (threadIdx.x == 6) {
        for (int k = 0; k < W; ++k) mn = fminf(mn, shm[k]);
        dst[5] = isinf(mn) && mn > 0.0f ? 1e300 : (double)mn;
    } else if (threadIdx.x == 32) {
        for (int k = 0; k < W; ++k) mb = shb[k] > mb ? shb[k] : mb;
        dst[6] = ROOT ? sqrt(__longlong_as_double(mb)) : __longlong_as_double(mb);
    }
}

// Runs of kDiagThreads nodes, run after run; one partial record of 8 doubles
// per block. |beta|^2 is formed in FP64 only where its FP32 value is not
// below the largest one of the warp's runs so far (by more than the FP32 error,
// 1e-6 of it or 1e-37), and where it is not zero. Whole diagnostics call at
// 256x128x128 FP32 on GB300: 467 -> 241 us, some 25 of them the copy to the
// host (203 at the copy bandwidth); before, minimum, maximum and a root per
// node in FP64.
template <int ST, bool PER>
__global__ void __launch_bounds__(kDiagThreads, 2)
    diag_kernel(const StepArgs a, const FastDiv nxy, const FastDiv nx, double dxcube, double* partials) {
    chain_begin();
    using T = typename Codec<ST>::T;
    const Grid& g = a.g;
    Diag d = diag_none();
    float top = 0.0f;  // the warp's largest FP32 |beta|^2
    for (uint32_t run = blockIdx.x; (int64_t)run * kDiagThreads < g.N; run += gridDim.x) {
        const uint32_t node = run * kDiagThreads + threadIdx.x;
        float b2 = 0.0f, beta[3] = {0.0f, 0.0f, 0.0f};
        if (node < (uint32_t)g.N) {
            const uint32_t k = nxy.div(node), r = node - k * nxy.d, j = nx.div(r);
            float f[kL][kQ];
            bool bnd;
            gather<ST, PER>(g, static_cast<const T*>(a.fin), a.n0, (int)(r - j * nx.d), (int)j, (int)k, f, bnd, 0u,
                            a.dbg);
            float e[6];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                e[c] = ld_state(a.E[c] + node);
                e[3 + c] = ld_state(a.Bc[c] + node);
            }
            float A[kL], inn;
            node_moments(f, a.n_floor, A, inn, beta);
            const bool fin = isfinite(A[0]) && isfinite(A[1]) && isfinite(A[2]) && isfinite(A[3]);
            d.bad += fin ? 0 : 1;
#pragma unroll
            for (int l = 0; l < kL; ++l) d.s[l] += A[l];
            d.mn = fminf(d.mn, A[0]);
            b2 = beta[0] * beta[0] + beta[1] * beta[1] + beta[2] * beta[2];
#pragma unroll
            for (int c = 0; c < 6; ++c) d.s[4] += (double)e[c] * e[c];
        }
        if ((beta[0] != 0.0f || beta[1] != 0.0f || beta[2] != 0.0f) && b2 >= top * 0.999999f - 1e-37f) {
            const double v = (double)beta[0] * beta[0] + (double)beta[1] * beta[1] + (double)beta[2] * beta[2];
            d.mb = max(d.mb, __double_as_longlong(v));
        }
        top = __uint_as_float(
            __reduce_max_sync(0xffffffffu, __float_as_uint(b2 > top ? b2 : top)));
    }
    d.s[4] *= 0.5 * dxcube;
    diag_block_reduce<true>(d, partials + 8 * (int64_t)blockIdx.x);
}

__global__ void __launch_bounds__(kDiagThreads) diag_finish_kernel(const double* partials, int64_t nparts, double* out) {
    chain_begin();
    Diag d = diag_none();
    for (int64_t b = threadIdx.x; b < nparts; b += blockDim.x) {
        const double* p = partials + 8 * b;
        for (int k = 0; k < 5; ++k) d.s[k] += p[k];
        d.mn = fminf(d.mn, (float)p[5]);  // a float, or 1e300: infinity
        d.mb = max(d.mb, __double_as_longlong(p[6]));
        d.bad += (int)p[7];
    }
    diag_block_reduce<false>(d, out);
}

// Block b combines FP32 fluid records [b per, (b + 1) per) and energy
// records [b per_e, (b + 1) per_e) in FP64 into scratch[b]. A fluid record's
// slot 6 holds min(-|beta|^2) (3e38 when the warp had no node).
__global__ void __launch_bounds__(kDiagThreads) diag_chunk_kernel(const float* rec, int64_t nrec, int64_t per,
                                                                  const float* en, int64_t nen, int64_t per_e,
                                                                  double dxcube, double* scratch) {
    chain_begin();
    Diag d = diag_none();
    float b2 = 0.0f;
    const int64_t b0 = (int64_t)blockIdx.x * per;
    const int64_t b1 = b0 + per < nrec ? b0 + per : nrec;
    for (int64_t b = b0 + threadIdx.x; b < b1; b += blockDim.x) {
        const float4 p = reinterpret_cast<const float4*>(rec)[2 * b];
        const float4 q = reinterpret_cast<const float4*>(rec)[2 * b + 1];
        d.s[0] += p.x;
        d.s[1] += p.y;
        d.s[2] += p.z;
        d.s[3] += p.w;
        d.s[4] += q.x;
        if (q.y < 3.0e38f) d.mn = fminf(d.mn, q.y);
        b2 = fmaxf(b2, -q.z);
        d.bad += (int)q.w;
    }
    d.mb = __double_as_longlong((double)b2);
    const int64_t e0 = (int64_t)blockIdx.x * per_e;
    const int64_t e1 = e0 + per_e < nen ? e0 + per_e : nen;
    for (int64_t b = e0 + threadIdx.x; b < e1; b += blockDim.x) d.s[4] += en[b];
    d.s[4] *= dxcube;
    diag_block_reduce<true>(d, scratch + 8 * (int64_t)blockIdx.x);
}

// Witness slab: the x range [rows[2 j], rows[2 j + 1]) of each row j in plane
// k. One block sums E_z over it in FP64 (the slab holds at most a few
// thousand edges).
constexpr int kWitnessThreads = 256;
__global__ void __launch_bounds__(kWitnessThreads) witness_sum_kernel(Grid g, const float* Ez, int k,
                                                                      const int* rows, double* out) {
    double s = 0.0;
    const int64_t plane = (int64_t)k * g.nx * g.ny;
    for (int j = 0; j < g.ny; ++j) {
        const int lo = rows[2 * j], hi = rows[2 * j + 1];
        for (int i = lo + (int)threadIdx.x; i < hi; i += kWitnessThreads) s += Ez[plane + (int64_t)j * g.nx + i];
    }
    for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
    __shared__ double sh[kWitnessThreads / 32];
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kWitnessThreads / 32; ++w) t += sh[w];
        *out = t;
    }
}

// Ez_bar := value on the witness slab (the rest of the array is untouched).
__global__ void witness_seed_kernel(Grid g, float* Ezbar, int k, const int* rows, float value) {
    const int j = blockIdx.x;
    const int lo = rows[2 * j], hi = rows[2 * j + 1];
    const int64_t row = ((int64_t)k * g.ny + j) * g.nx;
    for (int i = lo + (int)threadIdx.x; i < hi; i += blockDim.x) Ezbar[row + i] = value;
}

}  // namespace

cudaError_t launch_witness_sum(const Grid& g, const float* Ez, int k, const int* rows, double* out, cudaStream_t s) {
    witness_sum_kernel<<<1, kWitnessThreads, 0, s>>>(g, Ez, k, rows, out);
    return cudaGetLastError();
}

cudaError_t launch_witness_seed(const Grid& g, float* Ezbar, int k, const int* rows, float value, cudaStream_t s) {
    witness_seed_kernel<<<g.ny, 128, 0, s>>>(g, Ezbar, k, rows, value);
    return cudaGetLastError();
}

cudaError_t launch_diag_finish_step(const DiagOut& d, int64_t nrec, cudaStream_t s) {
    int64_t chunks = (nrec + 1023) / 1024;
    if (chunks < 1) chunks = 1;
    if (chunks > kDiagBlocks) chunks = kDiagBlocks;
    const int64_t per = (nrec + chunks - 1) / chunks;
    const int64_t per_e = (d.nenergy + chunks - 1) / chunks;
    cudaError_t e = launch_chained(diag_chunk_kernel, (unsigned)chunks, kDiagThreads, s, (const float*)d.records, nrec, per,
                                   (const float*)d.energy, d.nenergy, per_e, d.dxcube, d.scratch);
    if (e != cudaSuccess) return e;
    return launch_chained(diag_finish_kernel, 1, kDiagThreads, s, (const double*)d.scratch, chunks, d.out);
}

cudaError_t launch_init(const Grid& g, void* f, int storage, float n0, const double* d_profile, int n_profile,
                        double profile_rmax, double dx, cudaStream_t s) {
    const int threads = 256;
    const unsigned blocks = (unsigned)((g.Np + threads - 1) / threads);
    switch (storage) {
        case 0: init_kernel<0><<<blocks, threads, 0, s>>>(g, (float*)f, n0, d_profile, n_profile, profile_rmax, dx); break;
        case 1: init_kernel<1><<<blocks, threads, 0, s>>>(g, (__nv_bfloat16*)f, n0, d_profile, n_profile, profile_rmax, dx); break;
        case 2: init_kernel<2><<<blocks, threads, 0, s>>>(g, (__half*)f, n0, d_profile, n_profile, profile_rmax, dx); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <int ST>
static cudaError_t export_f(const StepArgs& a, float* out, cudaStream_t s) {
    const LinearMap m(a.g);
    if (a.g.periodic) export_f_kernel<ST, true><<<linear_blocks(a.g), kLinearThreads, 0, s>>>(a, m, out);
    else export_f_kernel<ST, false><<<linear_blocks(a.g), kLinearThreads, 0, s>>>(a, m, out);
    return cudaGetLastError();
}

cudaError_t launch_export_f(const StepArgs& a, int storage, float* out, cudaStream_t s) {
    switch (storage) {
        case 0: return export_f<0>(a, out, s);
        case 1: return export_f<1>(a, out, s);
        case 2: return export_f<2>(a, out, s);
    }
    return cudaErrorInvalidValue;
}

template <int ST>
static cudaError_t import_f(const Grid& g, const float* in, void* f, float n0, cudaStream_t s) {
    using T = typename Codec<ST>::T;
    const dim3 grid(linear_blocks(g), kL / 2, 1);
    if (g.periodic) import_f_kernel<ST, true><<<grid, kLinearThreads, 0, s>>>(g, LinearMap(g), in, static_cast<T*>(f), n0);
    else import_f_kernel<ST, false><<<grid, kLinearThreads, 0, s>>>(g, LinearMap(g), in, static_cast<T*>(f), n0);
    return cudaGetLastError();
}

cudaError_t launch_import_f(const Grid& g, const float* in, void* f, int storage, float n0, cudaStream_t s) {
    switch (storage) {
        case 0: return import_f<0>(g, in, f, n0, s);
        case 1: return import_f<1>(g, in, f, n0, s);
        case 2: return import_f<2>(g, in, f, n0, s);
    }
    return cudaErrorInvalidValue;
}

template <int ST>
static cudaError_t export_fields(const StepArgs& a, unsigned mask, float* out, cudaStream_t s) {
    const dim3 grid((a.g.nx + kBX - 1) / kBX, (a.g.ny + kBY - 1) / kBY, a.g.nz), block(kBX, kBY, 1);
    if (a.g.periodic) export_fields_kernel<ST, true><<<grid, block, 0, s>>>(a, mask, out);
    else export_fields_kernel<ST, false><<<grid, block, 0, s>>>(a, mask, out);
    return cudaGetLastError();
}

cudaError_t launch_export_fields(const StepArgs& a, int storage, unsigned mask, float* out, cudaStream_t s) {
    switch (storage) {
        case 0: return export_fields<0>(a, mask, out, s);
        case 1: return export_fields<1>(a, mask, out, s);
        case 2: return export_fields<2>(a, mask, out, s);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_linecut(const StepArgs& a, int storage, double r, float* out, cudaStream_t s) {
    const int threads = 128;
    const unsigned blocks = (unsigned)((a.g.nz + threads - 1) / threads);
    const bool per = a.g.periodic;
    switch (storage) {
        case 0: if (per) linecut_kernel<0, true><<<blocks, threads, 0, s>>>(a, r, out); else linecut_kernel<0, false><<<blocks, threads, 0, s>>>(a, r, out); break;
        case 1: if (per) linecut_kernel<1, true><<<blocks, threads, 0, s>>>(a, r, out); else linecut_kernel<1, false><<<blocks, threads, 0, s>>>(a, r, out); break;
        case 2: if (per) linecut_kernel<2, true><<<blocks, threads, 0, s>>>(a, r, out); else linecut_kernel<2, false><<<blocks, threads, 0, s>>>(a, r, out); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <int ST>
static cudaError_t diag_t(const StepArgs& a, int blocks, double dxcube, double* partials, cudaStream_t s) {
    const LinearMap m(a.g);
    return launch_chained(a.g.periodic ? diag_kernel<ST, true> : diag_kernel<ST, false>, blocks, kDiagThreads, s, a,
                          m.nxy, m.nx, dxcube, partials);
}

cudaError_t launch_diag(const StepArgs& a, int storage, double dxcube, double* partials, double* out, cudaStream_t s) {
    const int64_t need = (a.g.N + kDiagThreads - 1) / kDiagThreads;
    int sms = 0;
    cudaError_t e = sm_count(&sms);
    if (e != cudaSuccess) return e;
    // two blocks per SM, a partial record each
    const int64_t resident = 2 * sms < kDiagBlocks ? 2 * sms : kDiagBlocks;
    const int blocks = (int)(need < resident ? need : resident);
    e = cudaErrorInvalidValue;
    switch (storage) {
        case 0: e = diag_t<0>(a, blocks, dxcube, partials, s); break;
        case 1: e = diag_t<1>(a, blocks, dxcube, partials, s); break;
        case 2: e = diag_t<2>(a, blocks, dxcube, partials, s); break;
    }
    if (e != cudaSuccess) return e;
    return launch_chained(diag_finish_kernel, 1, kDiagThreads, s, (const double*)partials, (int64_t)blocks, out);
}

}  // namespace pwfa
