// The fluid step of the adjoint's recompute: the fused fluid kernel of
// fluid.cu that also stores each node's lattice sums A_l for the reverse
// step (a translation unit of its own, so that the production kernels'
// build is unchanged).
#include "lbm_kernels.h"
#include "fluid_node.cuh"
#include "launch.cuh"

namespace pwfa {

namespace {

template <int ST, int COLL, bool PER>
__global__ void __launch_bounds__(kLinearThreads, FluidOcc<ST, COLL>::blocks)
    fluid_mom_kernel(const StepArgs a, const LinearMap m) {
    chain_begin();
    int x, y, z;
    if (m.node(a.g, x, y, z)) fluid_node<ST, COLL, PER, false, true>(a, x, y, z);
}

template <int ST, int COLL>
cudaError_t launch_t(const StepArgs& a, cudaStream_t s) {
    if (!a.mom) return cudaErrorInvalidConfiguration;
    return launch_chained(a.g.periodic ? fluid_mom_kernel<ST, COLL, true> : fluid_mom_kernel<ST, COLL, false>,
                          linear_blocks(a.g), kLinearThreads, s, a, LinearMap(a.g));
}

template <int ST>
cudaError_t launch_s(const StepArgs& a, int collision, cudaStream_t s) {
    switch (collision) {
        case 0: return launch_t<ST, 0>(a, s);
        case 1: return launch_t<ST, 1>(a, s);
        case 2: return launch_t<ST, 2>(a, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_fluid_mom(const StepArgs& a, int storage, int collision, cudaStream_t s) {
    switch (storage) {
        case 0: return launch_s<0>(a, collision, s);
        case 1: return launch_s<1>(a, collision, s);
        case 2: return launch_s<2>(a, collision, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace pwfa
