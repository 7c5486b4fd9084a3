// Kernels of the 2D-axisymmetric (z, r) form: the fused step (Faraday's law,
// pull, node moments, the cylindrical terms of Eq. 13, collision), Ampere
// with the driver, and the node moments for exports.
#include "axi.h"
#include "launch.cuh"

namespace pwfa {
namespace axi {

namespace {

constexpr int kBR = 32;  // threads along r
constexpr int kBZ = 4;   // threads along z

// D2Q9 in (z, r) components: rest, +z, -z, +r, -r, (+z,+r), (-z,-r), (+z,-r), (-z,+r)
__host__ __device__ constexpr int xz(int q) {
    return (q == 1 || q == 5 || q == 7) ? 1 : ((q == 2 || q == 6 || q == 8) ? -1 : 0);
}
__host__ __device__ constexpr int xr(int q) {
    return (q == 3 || q == 5 || q == 8) ? 1 : ((q == 4 || q == 6 || q == 7) ? -1 : 0);
}
__host__ __device__ constexpr float w9(int q) { return q == 0 ? 4.0f / 9.0f : (q <= 4 ? 1.0f / 9.0f : 1.0f / 36.0f); }
// the direction with the r component reversed
__host__ __device__ constexpr int rrefl(int q) {
    return q == 3 ? 4 : (q == 4 ? 3 : (q == 5 ? 7 : (q == 7 ? 5 : (q == 6 ? 8 : (q == 8 ? 6 : q)))));
}

// offset of (l = 0, q = 0) of a node; l, q add (9 l + q) 32
constexpr int kPopStride = 32;
__device__ __forceinline__ int64_t chunk(int64_t node) { return (node >> 5) * (kL * kQ * kPopStride) + (node & 31); }

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

// f^eq of Eq. 9 in lattice units (c_s^2 = 1/3)
__device__ __forceinline__ float feq(int q, float A, float uz, float ur) {
    const float xu = (float)xz(q) * uz + (float)xr(q) * ur;
    return w9(q) * A * (1.0f + 3.0f * xu + 4.5f * xu * xu - 1.5f * (uz * uz + ur * ur));
}

// The fields around node (k, j): E_r of three z levels and two radii, E_z of
// two z levels and three radii, B_theta of the four faces, every load issued
// at once with the indices clamped into the grid (what a clamped value would
// feed is masked where it is used).
struct NodeFields {
    float er[3][2];  // (k - 1, k, k + 1) x (j - 1, j)
    float ez[2][3];  // (k - 1, k) x (j - 1, j, j + 1)
    float bt[2][2];  // (k - 1, k) x (j - 1, j)
};

__device__ __forceinline__ void load_fields(const Args& a, int k, int j, NodeFields& v) {
    const int nr = a.nr;
    const int64_t o = (int64_t)k * nr + j;
    const int64_t km = k > 0 ? -nr : 0, kp = k < a.nz - 1 ? nr : 0;
    const int jm = j > 0 ? -1 : 0, jp = j < nr - 1 ? 1 : 0;
    v.er[0][0] = ld_state(a.Er + o + km + jm);
    v.er[0][1] = ld_state(a.Er + o + km);
    v.er[1][0] = ld_state(a.Er + o + jm);
    v.er[1][1] = ld_state(a.Er + o);
    v.er[2][0] = ld_state(a.Er + o + kp + jm);
    v.er[2][1] = ld_state(a.Er + o + kp);
    v.ez[0][0] = ld_state(a.Ez + o + km + jm);
    v.ez[0][1] = ld_state(a.Ez + o + km);
    v.ez[0][2] = ld_state(a.Ez + o + km + jp);
    v.ez[1][0] = ld_state(a.Ez + o + jm);
    v.ez[1][1] = ld_state(a.Ez + o);
    v.ez[1][2] = ld_state(a.Ez + o + jp);
    v.bt[0][0] = ld_state(a.Bt + o + km + jm);
    v.bt[0][1] = ld_state(a.Bt + o + km);
    v.bt[1][0] = ld_state(a.Bt + o + jm);
    v.bt[1][1] = ld_state(a.Bt + o);
}

// Faraday on the face (k - 1 + K, j - 1 + J): B_theta(t_{n+1}) = B_theta(t_n) +
// dt (dE_z/dr - dE_r/dz) on the active faces, zero elsewhere (axis, outer
// wall, outside the grid).
template <int K, int J>
__device__ __forceinline__ float faraday_bt(const Args& a, const NodeFields& v, int k, int j) {
    const int kf = k - 1 + K, jf = j - 1 + J;
    if (kf < 0 || kf > a.nz - 2 || jf < 1 || jf > a.nr - 2) return 0.0f;
    return v.bt[K][J] - a.cdt * ((v.er[K + 1][J] - v.er[K][J]) - (v.ez[K][J + 1] - v.ez[K][J]));
}

// The 27 values an interior node c pulls, f_i(c) = S_i(c - xi_i).
__device__ __forceinline__ void pull(const Args& a, int64_t c, float (&f)[kL][kQ]) {
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
        const float* p = a.fin + chunk(c - xz(q) * a.nr - xr(q));
#pragma unroll
        for (int l = 0; l < kL; ++l) f[l][q] = ld_state(p + (l * kQ + q) * kPopStride);
    }
}

// Pre-collision moments of every node: interior nodes sum their pulled
// populations; the z walls and the outer row take their clamped interior
// node's moments (their state is its equilibrium, Eq. 14); the axis row
// mirrors row 1 (n p_r changes sign).
__global__ void __launch_bounds__(kBR * kBZ) moments_kernel(const Args a) {
    const int j = blockIdx.x * kBR + threadIdx.x;
    const int k = blockIdx.y * kBZ + threadIdx.y;
    if (j >= a.nr || k >= a.nz) return;
    const int kc = clampi(k, 1, a.nz - 2);
    const int jc = clampi(j, 1, a.nr - 2);
    const int64_t base = (int64_t)kc * a.nr + jc;
    float f[kL][kQ], A[kL];
    pull(a, base, f);
#pragma unroll
    for (int l = 0; l < kL; ++l) {
        float s = 0.0f;
#pragma unroll
        for (int q = 0; q < kQ; ++q) s += f[l][q];
        A[l] = s;
    }
    if (j == 0) A[2] = -A[2];
    const int64_t o = (int64_t)k * a.nr + j;
#pragma unroll
    for (int l = 0; l < kL; ++l) a.Am[(int64_t)l * a.N + o] = A[l];
}

// One fused step of every node of rows 1..nr-1. A block takes a run of kRun
// consecutive nodes (whole chunks: its stores are aligned) and, in two lanes
// of one more warp, the node before and the one after the run; every thread
// gathers the pulled populations of its clamped node (its own node when
// interior; the clamped interior node for the z walls, the outer row and the
// mirror row, which negates n p_r), and the radial neighbours' moments of
// dA/dr meet in shared memory without a separate moments pass. Faraday's law
// runs here too: each node evaluates B_theta at t_{n+1} on the four faces
// around it and stores the one it owns (rows 1..nr-1; the axis row's B_theta
// stays zero). Then: the equilibrium of the clamped node on boundary nodes
// (Eq. 14), Lorentz source with the node fields, the cylindrical terms
// D (1/r) dA/dr - A u_r / r of Eq. 13 on interior nodes, BGK collision
// (Eq. 7) with S_i = w_i S dt, store; row 1 also writes the axis row as its
// mirror image. Node current J = -n* beta(p*) of the post-collision moments.
//
// Bound by memory latency and instruction issue about equally (ncu: issue
// 66 %, DRAM 47 % before). Step on 2400 x 402 (GB300): 60.1 us with the field
// values loaded face by face behind bounds checks, in warps of 30 nodes
// between two halo lanes; 53.9 with all 43 values of a node in one round;
// 50.9 with runs and chunks, four blocks of 160 threads per SM (three 51.1,
// five 53.1, six 55.5; runs of 64: 51.3, of 256: 54.0).
constexpr int kRun = 128;
__global__ void __launch_bounds__(kRun + 32, 4) fluid_kernel(const Args a) {
    chain_begin();
    __shared__ float sA[kL][kRun + 2];
    const int tid = (int)threadIdx.x;
    const int64_t first = (int64_t)blockIdx.x * kRun;
    // the run's nodes; in the last warp, lanes 0 and 1: the nodes before and
    // after it, whose moments its ends need
    const bool inner = tid < kRun;
    if (tid >= kRun + 2) return;
    const int64_t want = inner ? first + tid : (tid == kRun ? first - 1 : first + kRun);
    const int64_t node = want < 0 ? 0 : (want < a.N ? want : a.N - 1);
    const int k = (int)a.dnr.div((uint32_t)node);
    const int j = (int)(node - (int64_t)k * a.nr);
    const int kc = clampi(k, 1, a.nz - 2);
    const int jc = clampi(j, 1, a.nr - 2);
    const bool bnd = k == 0 || k == a.nz - 1 || j == a.nr - 1;
    // the node's fields and its 27 pulled values in one round of loads
    NodeFields fields;
    if (a.couple) load_fields(a, k, j, fields);
    float f[kL][kQ];
    float A[kL];
    pull(a, (int64_t)kc * a.nr + jc, f);
    const int slot = inner ? tid + 1 : (tid == kRun ? 0 : kRun + 1);
#pragma unroll
    for (int l = 0; l < kL; ++l) {
        float s = 0.0f;
#pragma unroll
        for (int q = 0; q < kQ; ++q) s += f[l][q];
        A[l] = l == 2 && j == 0 ? -s : s;
        sA[l][slot] = A[l];
    }
    __syncthreads();
    if (!inner || want >= a.N || j == 0) return;
    // radial neighbours' moments (pre-collision, every node's own rule)
    float Am1[kL], Ap1[kL];
#pragma unroll
    for (int l = 0; l < kL; ++l) {
        Am1[l] = sA[l][slot - 1];
        Ap1[l] = sA[l][slot + 1];
    }
    const int64_t o = node;
    // one division and one reciprocal square root (p = A_k / n, beta = p / gamma)
    const float inn = 1.0f / (A[0] > a.n_floor ? A[0] : a.n_floor);
    const float pz = A[1] * inn, pr = A[2] * inn;
    const float ig = rsqrtf(1.0f + pz * pz + pr * pr);
    const float bz = pz * ig, br = pr * ig;
    const float uz = bz * a.lat, ur = br * a.lat;
    // equilibrium factors shared by the three lattices: f^eq_l,i = A_l phi_i
    float phi[kQ];
#pragma unroll
    for (int q = 0; q < kQ; ++q) phi[q] = feq(q, 1.0f, uz, ur);
    if (bnd) {
        // Eq. 14: the equilibrium of the clamped node
#pragma unroll
        for (int l = 0; l < kL; ++l)
#pragma unroll
            for (int q = 0; q < kQ; ++q) f[l][q] = A[l] * phi[q];
#pragma unroll
        for (int l = 0; l < kL; ++l) {
            float s = 0.0f;
#pragma unroll
            for (int q = 0; q < kQ; ++q) s += f[l][q];
            A[l] = s;
        }
    }
    float S[kL] = {0.0f, 0.0f, 0.0f};
    // B_theta(t_{n+1}) of the node's own face
    const float btn = a.couple ? faraday_bt<1, 1>(a, fields, k, j) : 0.0f;
    float nst = A[0], pzs = A[1], prs = A[2];  // post-collision moments
    if (a.collision != 2) {
        if (a.couple) {
            // node fields: E_z of its two z edges, E_r of its two r edges,
            // B_theta over the four surrounding faces of both time levels
            const NodeFields& v = fields;
            const bool below = k > 0;  // (j > 0 here)
            const float ez = 0.5f * ((below ? v.ez[0][1] : 0.0f) + v.ez[1][1]);
            const float er = 0.5f * (v.er[1][0] + v.er[1][1]);
            float bs = 0.0f;
            bs += (below ? v.bt[0][0] : 0.0f) + faraday_bt<0, 0>(a, v, k, j);
            bs += (below ? v.bt[0][1] : 0.0f) + faraday_bt<0, 1>(a, v, k, j);
            bs += v.bt[1][0] + faraday_bt<1, 0>(a, v, k, j);
            bs += v.bt[1][1] + btn;
            const float bt = bs * 0.125f;
            // F_z = -n (E_z + beta_r B_theta), F_r = -n (E_r - beta_z B_theta)
            S[1] = -A[0] * (ez + br * bt);
            S[2] = -A[0] * (er - bz * bt);
        }
        if (!bnd) {
            // D (1/r) dA/dr - A u_r / r, dA/dr = (A(r + dx) - A(r - dx)) / 2 dx
            const float inv_r = 1.0f / (((float)j - 0.5f) * a.dx);
            const float c = 0.5f * a.D / a.dx;
#pragma unroll
            for (int l = 0; l < kL; ++l) S[l] += (c * (Ap1[l] - Am1[l]) - A[l] * br) * inv_r;
        }
        nst = A[0] + S[0] * a.dt;
        pzs = A[1] + S[1] * a.dt;
        prs = A[2] + S[2] * a.dt;
    }
    // collide and store (row 1 also writes its mirror image into the axis row)
    const int64_t om = (int64_t)k * a.nr;  // axis row node of this column
    const float omc = 1.0f - a.omega;
#pragma unroll
    for (int l = 0; l < kL; ++l) {
        float* fo = a.fout + chunk(o) + l * kQ * kPopStride;
        float* fm = a.fout + chunk(om) + l * kQ * kPopStride;
        const float sg = l == 2 ? -1.0f : 1.0f;
        // f* = (1 - omega) f + omega A phi_i + w_i S dt, the weights applied
        // once per lattice
        const float oA = a.omega * A[l], sdt = S[l] * a.dt;
        const float sw[3] = {sdt * w9(0), sdt * w9(1), sdt * w9(5)};
#pragma unroll
        for (int q = 0; q < kQ; ++q) {
            float fs = f[l][q];
            if (a.collision != 2) fs = fmaf(fs, omc, fmaf(oA, phi[q], sw[q == 0 ? 0 : (q <= 4 ? 1 : 2)]));
            fo[q * kPopStride] = fs;
            if (j == 1) fm[rrefl(q) * kPopStride] = sg * fs;
        }
    }
    const float insn = 1.0f / (nst > a.n_floor ? nst : a.n_floor);
    const float qz = pzs * insn, qr = prs * insn;
    const float ngs = -nst * rsqrtf(1.0f + qz * qz + qr * qr);
    const float jz = ngs * qz, jr = ngs * qr;
    if (a.couple) a.Btn[o] = btn;
    a.Jz[o] = jz;
    a.Jr[o] = jr;
    if (j == 1) {
        a.Jz[om] = jz;
        a.Jr[om] = -jr;
    }
}

// Ampere: dE_r/dt = -dB_theta/dz - J_r, dE_z/dt = (1/r) d(r B_theta)/dr - J_z - J_b.
// A thread takes kAmpRows z levels of one radius, with every load issued
// before the first use and the neighbours clamped into the grid (the walls
// discard what a clamped one feeds): the kernel is a few waves of latency.
// Step on 2400 x 402: 50.9 us with loads inside the wall branches and 2D
// blocks, 50.6, 48.8, 49.3, 51.4 with 1, 2, 4, 8 levels.
constexpr int kAmpRows = 2, kAmpThreads = 128;
__global__ void __launch_bounds__(kAmpThreads) ampere_kernel(const Args a) {
    chain_begin();
    const uint32_t t = blockIdx.x * kAmpThreads + threadIdx.x;
    const int k0 = (int)a.dnr.div(t) * kAmpRows, j = (int)(t - a.dnr.div(t) * (uint32_t)a.nr);
    if (k0 >= a.nz || j < 1 || j > a.nr - 2) return;  // (the walls keep their zeros)
    const int64_t o = (int64_t)k0 * a.nr + j;
    float bt[kAmpRows + 1], bt_j[kAmpRows], jr[kAmpRows], jr_j[kAmpRows], jz[kAmpRows + 1], er[kAmpRows], ez[kAmpRows];
    bt[0] = ld_state(a.Btn + o - (k0 > 0 ? a.nr : 0));
    jz[kAmpRows] = ld_state(a.Jz + (int64_t)min(k0 + kAmpRows, a.nz - 1) * a.nr + j);
#pragma unroll
    for (int i = 0; i < kAmpRows; ++i) {
        const int64_t p = (int64_t)min(k0 + i, a.nz - 1) * a.nr + j;
        bt[i + 1] = ld_state(a.Btn + p);
        bt_j[i] = ld_state(a.Btn + p - 1);
        jr[i] = ld_state(a.Jr + p);
        jr_j[i] = ld_state(a.Jr + p + 1);
        jz[i] = ld_state(a.Jz + p);
        er[i] = a.ErO[p];
        ez[i] = a.EzO[p];
    }
    const float r = ((float)j - 0.5f) * a.dx;
#pragma unroll
    for (int i = 0; i < kAmpRows; ++i) {
        const int k = k0 + i;
        const int64_t p = (int64_t)k * a.nr + j;
        if (k >= 1 && k <= a.nz - 2) {
            const float je = 0.5f * (jr[i] + jr_j[i]);
            a.ErO[p] = er[i] - a.cdt * (bt[i + 1] - bt[i]) - a.dt * je;
        }
        if (k <= a.nz - 2) {
            const float curl = ((float)j * bt[i + 1] - (float)(j - 1) * bt_j[i]) / ((float)j - 0.5f);
            const float je = 0.5f * (jz[i] + jz[i + 1]);
            float jb = 0.0f;
            if (a.alpha != 0.0f) {
                const float zeta = ((float)k + 0.5f) * a.dx - a.zc;
                jb = -a.alpha * expf(-r * r * a.inv2sr2 - zeta * zeta * a.inv2sz2);
            }
            a.EzO[p] = ez[i] + a.cdt * curl - a.dt * (je + jb);
        }
    }
}

__global__ void init_kernel(const Args a, float* f) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)kL * kQ * a.Np) return;
    const int lq = (int)(i / kPopStride % (kL * kQ));
    f[i] = lq < kQ ? w9(lq) * a.n0 : 0.0f;
}

// Chunks to planes [3][9][N] and back, one thread per node.
template <bool PACK>
__global__ void pack_kernel(const Args a, const float* in, float* out) {
    const int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= a.N) return;
    const int64_t c = chunk(o);
#pragma unroll
    for (int lq = 0; lq < kL * kQ; ++lq) {
        const int64_t chunked = c + lq * kPopStride, plane = lq * a.N + o;
        out[PACK ? chunked : plane] = in[PACK ? plane : chunked];
    }
}

__global__ void export_kernel(const Args a, float* out) {
    const int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= a.N) return;
    const float n = a.Am[o], A1 = a.Am[a.N + o], A2 = a.Am[2 * a.N + o];
    const float nn = n > a.n_floor ? n : a.n_floor;
    const float pz = A1 / nn, pr = A2 / nn;
    const float g = sqrtf(1.0f + pz * pz + pr * pr);
    out[o] = n;
    out[a.N + o] = pz / g;
    out[2 * a.N + o] = pr / g;
}

dim3 grid_of(const Args& a) { return dim3((a.nr + kBR - 1) / kBR, (a.nz + kBZ - 1) / kBZ, 1); }

}  // namespace

cudaError_t launch_moments(const Args& a, cudaStream_t s) {
    moments_kernel<<<grid_of(a), dim3(kBR, kBZ), 0, s>>>(a);
    return cudaGetLastError();
}
cudaError_t launch_fluid(const Args& a, cudaStream_t s) {
    return launch_chained(fluid_kernel, (unsigned)((a.N + kRun - 1) / kRun), kRun + 32, s, a);
}
cudaError_t launch_ampere(const Args& a, cudaStream_t s) {
    const int64_t threads = (int64_t)a.nr * ((a.nz + kAmpRows - 1) / kAmpRows);
    return launch_chained(ampere_kernel, (unsigned)((threads + kAmpThreads - 1) / kAmpThreads), kAmpThreads, s, a);
}
cudaError_t launch_pack(const Args& a, const float* planes, float* f, cudaStream_t s) {
    pack_kernel<true><<<(unsigned)((a.N + 255) / 256), 256, 0, s>>>(a, planes, f);
    return cudaGetLastError();
}
cudaError_t launch_unpack(const Args& a, const float* f, float* planes, cudaStream_t s) {
    pack_kernel<false><<<(unsigned)((a.N + 255) / 256), 256, 0, s>>>(a, f, planes);
    return cudaGetLastError();
}
cudaError_t launch_init(const Args& a, float* f, cudaStream_t s) {
    const int64_t n = (int64_t)kL * kQ * a.Np;
    init_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(a, f);
    return cudaGetLastError();
}
cudaError_t launch_export_moments(const Args& a, float* out, cudaStream_t s) {
    export_kernel<<<(unsigned)((a.N + 255) / 256), 256, 0, s>>>(a, out);
    return cudaGetLastError();
}

}  // namespace axi
}  // namespace pwfa
